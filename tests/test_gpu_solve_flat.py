"""The global solve for flat kernels, whose factor has badly conditioned diagonal blocks: the
residual and the error between the nodes against substitution's.

rbfsl_global_solve under stream capture has no scratch and substitutes through 64-row blocks
in FP64; otherwise it multiplies by the blocks' inverses with one correction each. Both are
backward stable, with the same constants in front of eps |L| |U| |c|, so that their residuals
for the same factor differ by rounding alone: a factor of two of the largest of some ten
thousand residuals, where a product with the inverses alone is off by ten to fifty.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV, dtype)


def _phi(kind, eps, P, X):
    d2 = torch.zeros((P.shape[0], X.shape[0]), dtype=torch.float64, device=DEV)
    for i in range(3):
        d2 += (P[:, None, i] - X[None, :, i]) ** 2
    return torch.exp(-eps * eps * d2) if kind == rbfsl.GAUSS else torch.rsqrt(1.0 + eps * eps * d2)


# the shape parameter of inputs.config_global_rotation and the same eps h on a coarser set; a flat IMQ
@pytest.mark.parametrize("N,kind,eps", [(10242, rbfsl.GAUSS, 6.0), (2562, rbfsl.GAUSS, 3.0), (4001, rbfsl.GAUSS, 3.73),
                                        (2562, rbfsl.IMQ, 1.0), (5003, rbfsl.IMQ, 2.0)])
def test_residual_is_substitutions(N, kind, eps):
    w = inputs.config_global_rotation(N=N, T=8)
    X = w.X
    rng = np.random.default_rng(N)
    P = X[::5] + 0.3 / np.sqrt(N) * rng.standard_normal((len(X[::5]), 3))
    P /= np.linalg.norm(P, axis=1, keepdims=True)
    x, q = _t(X), _t(w.tracers(X))
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_global_factor(x, kind, eps, LU, perm)
    c, plain = torch.empty_like(q), torch.empty_like(q)
    rbfsl.rbfsl_global_solve(LU, perm, q, c)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rbfsl.rbfsl_global_solve(LU, perm, q, plain)
    g.replay()
    torch.cuda.synchronize()
    A = _phi(kind, eps, x, x)
    res = [(A @ v - q).abs().max().item() for v in (c, plain)]
    del A
    E, exact = _phi(kind, eps, _t(P), x), _t(w.tracers(P))
    err = [(E @ v - exact).abs().max().item() for v in (c, plain)]
    print(f"N={N} eps={eps}: residual {res[0]:.2e} / {res[1]:.2e}, error {err[0]:.2e} / {err[1]:.2e}")
    assert res[0] <= 2.0 * res[1]
    assert err[0] <= 2.0 * err[1]
