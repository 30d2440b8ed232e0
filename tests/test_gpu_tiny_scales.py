"""Products and solves of the global method scale with their input down to the subnormal numbers:
2^k q gives 2^k times the result for q. Scaling by a power of two changes no rounding but those
below 2^-1074, which lie 2^(-1074 - k) below the data: at k = -1000 2^-74, times the number of
terms (and, in a solve, the condition of the matrix, below 1e7 here)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV, dtype)


# few and many columns; a matrix of tiny rows beside ordinary ones
@pytest.mark.parametrize("k", [-700, -960, -1000])
@pytest.mark.parametrize("T", [5, 40])
def test_apply(k, T):
    rng = np.random.default_rng(T)
    E, q = rng.standard_normal((70, 300)), rng.standard_normal((300, T))
    q[:, 2] = 0.0
    ref, out = torch.empty((70, T), dtype=torch.float64, device=DEV), torch.empty((70, T), dtype=torch.float64, device=DEV)
    rbfsl.rbfsl_cardinal_apply(_t(E), _t(q), ref)
    bound = 1e-15 * (np.abs(E) @ np.abs(q)) + 0.0
    rbfsl.rbfsl_cardinal_apply(_t(E), _t(np.ldexp(q, k)), out)
    assert np.all(np.abs(np.ldexp(out.cpu().numpy(), -k) - ref.cpu().numpy()) <= bound)
    rows = np.where(np.arange(70) % 3 == 0, k, 0)[:, None]
    rbfsl.rbfsl_cardinal_apply(_t(np.ldexp(E, rows)), _t(q), out)
    assert np.all(np.abs(np.ldexp(out.cpu().numpy(), -rows) - ref.cpu().numpy()) <= bound)


@pytest.mark.parametrize("k", [-700, -960, -1000])
@pytest.mark.parametrize("N,T", [(642, 5), (642, 40)])
def test_solve_and_evaluation(k, N, T):
    X = inputs.nodes(N, 3)
    x = _t(X)
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_global_factor(x, rbfsl.GAUSS, 4.0, LU, perm)
    q = np.random.default_rng(N + T).standard_normal((N, T))
    res = []
    for s in (0, k):
        c, o = (torch.empty((N, T), dtype=torch.float64, device=DEV) for _ in range(2))
        rbfsl.rbfsl_global_solve(LU, perm, _t(np.ldexp(q, s)), c)
        rbfsl.rbfsl_global_eval(x, x, rbfsl.GAUSS, 4.0, _t(np.ldexp(q, s)), o)
        res.append([np.ldexp(v.cpu().numpy(), -s) for v in (c, o)])
    for a, b in zip(*res):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()
