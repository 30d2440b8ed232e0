"""Stateless global calls that are too small for their scratch to pay take the form without it,
which under capture runs for any size: the same bits there. Larger calls agree to the bounds of the
other tests, at the edges of the solve's 64- and 128-row blocks and column tiles."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

from test_gpu_global import lu_residual_bound  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV, dtype)


def _captured(call):
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    g.replay()
    torch.cuda.synchronize()


def _factor(N, eps):
    x = _t(inputs.nodes(N, 3))
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_global_factor(x, rbfsl.IMQ, eps, LU, perm)
    return x, LU, perm


@pytest.mark.parametrize("N,T", [(65, 1), (128, 64), (257, 9), (383, 33)])
def test_small_calls_do_not_change_under_capture(N, T):
    eps = 0.1 * np.sqrt(N)
    x, LU, perm = _factor(N, eps)
    q = _t(np.random.default_rng(N).standard_normal((N, T)))
    c, c2, o, o2 = (torch.empty_like(q) for _ in range(4))
    rbfsl.rbfsl_global_solve(LU, perm, q, c)
    _captured(lambda: rbfsl.rbfsl_global_solve(LU, perm, q, c2))
    assert torch.equal(c, c2)
    rbfsl.rbfsl_global_eval(x, x, rbfsl.IMQ, eps, c, o)
    _captured(lambda: rbfsl.rbfsl_global_eval(x, x, rbfsl.IMQ, eps, c, o2))
    assert torch.equal(o, o2)


# one row, half a block, a block and one row beyond three blocks of 128; few nodes with many tracers
@pytest.mark.parametrize("N,T", [(384, 1), (385, 8), (447, 9), (448, 32), (449, 33), (511, 64), (512, 65), (513, 130),
                                 (192, 512), (65, 1600)])
@pytest.mark.parametrize("chol", [False, True])
def test_solve_edges_with_scratch(orc, N, T, chol):
    X = inputs.nodes(N, 3)
    q = np.random.default_rng(N + T).standard_normal((N, T))
    eps = 0.16 * np.sqrt(N)
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    (rbfsl.rbfsl_global_factor_chol if chol else rbfsl.rbfsl_global_factor)(_t(X), rbfsl.GAUSS, eps, LU, perm)
    c = torch.empty((N, T), dtype=torch.float64, device=DEV)
    rbfsl.rbfsl_global_solve(LU, perm, _t(q), c)
    C = c.cpu().numpy()
    A = orc.global_matrix(X, orc.GAUSS, eps)
    assert np.abs(A @ C - q).max() <= lu_residual_bound(N, np.abs(A).sum(1).max(), C)


# products on the tensor cores by the number of nodes and by the number of points, against FP64
@pytest.mark.parametrize("Nq,N,T", [(1, 384, 4), (33, 400, 65), (12000, 128, 5), (8000, 64, 130)])
def test_evaluation_with_scratch(Nq, N, T):
    x = _t(inputs.nodes(N, 3))
    p = _t(inputs.nodes(max(Nq, 12), 4)[:Nq])
    c = _t(np.random.default_rng(T).standard_normal((N, T)))
    o = torch.empty((Nq, T), dtype=torch.float64, device=DEV)
    rbfsl.rbfsl_global_eval(p, x, rbfsl.IMQ, 2.0, c, o)
    E = torch.rsqrt(1.0 + 4.0 * ((p[:, None] - x[None]) ** 2).sum(-1))
    assert torch.all((o - E @ c).abs() <= 1e-13 * (E @ c.abs()))
