"""The global method's products and solves on the tensor cores (digit-split FP64) at the edges of
their tiles, over wide scales and with values that are not finite.

Tolerances: a digit product cuts a chunk's entries off at 2^-61 of the row's and the column's largest
and drops digit products below 2^-65 of them, so 128 terms lie within 128 (2 * 2^-61 + 2^-62) < 2^-52
of largest times largest, and the chunk sums are added in FP64: for rows and columns whose entries
are of one size that is below 1e-13 of sum |E| |q|, the bound of the FP64 product's tests. Solves: the
backward-error bound of the solve's other tests.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

from test_gpu_global import lu_residual_bound  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV, dtype)


# one block, one and two halves of a diagonal block, ragged ends, one to three column tiles
@pytest.mark.parametrize("N,T", [(64, 3), (65, 1), (128, 8), (129, 9), (192, 32), (200, 33), (257, 64), (400, 65),
                                 (640, 130)])
@pytest.mark.parametrize("chol", [False, True])
def test_solve_edges(orc, N, T, chol):
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
    c2 = torch.empty_like(c)
    rbfsl.rbfsl_global_solve(LU, perm, _t(q), c2)
    assert torch.equal(c, c2)


@pytest.mark.parametrize("Nq,N,T", [(1, 1, 1), (16, 16, 8), (31, 127, 7), (32, 128, 32), (33, 129, 33), (64, 256, 64),
                                    (65, 257, 72), (700, 1500, 3)])
def test_apply_edges_and_scales(Nq, N, T):
    rng = np.random.default_rng(Nq + 7 * N + T)
    E = rng.uniform(0.5, 1.0, (Nq, N)) * rng.choice([-1.0, 1.0], (Nq, N)) * 10.0 ** rng.uniform(-140, 140, (Nq, 1))
    q = rng.uniform(0.5, 1.0, (N, T)) * rng.choice([-1.0, 1.0], (N, T)) * 10.0 ** rng.uniform(-140, 140, (1, T))
    out = torch.empty((Nq, T), dtype=torch.float64, device=DEV)
    rbfsl.rbfsl_cardinal_apply(_t(E), _t(q), out)
    assert np.all(np.abs(out.cpu().numpy() - E @ q) <= 1e-13 * (np.abs(E) @ np.abs(q)))


@pytest.mark.parametrize("T", [5, 40])
def test_apply_not_finite(T):
    """A NaN or an infinity reaches the rows and columns that it reaches in FP64, and no others. A sum
    of finite products beyond the doubles' range is not finite: an infinity or, where partial sums of
    both signs overflow (as the order of the sum has it in any FP64 form), a NaN."""
    Nq, N = 70, 300
    rng = np.random.default_rng(5)
    E, q = rng.standard_normal((Nq, N)), rng.standard_normal((N, T))
    q[200, 1] = np.nan
    q[10, 2] = np.inf
    E[3, 7] = -np.inf
    E[40, 290] = np.nan
    E[50] *= 1e200
    q[:, 4] *= 1e200
    with np.errstate(all="ignore"):
        ext = np.array([[np.sum(E[i].astype(np.longdouble) * q[:, t]) for t in range(T)] for i in range(Nq)])
        ref = ext.astype(float)
    out = torch.empty((Nq, T), dtype=torch.float64, device=DEV)
    rbfsl.rbfsl_cardinal_apply(_t(E), _t(q), out)
    got = out.cpu().numpy()
    assert (np.isfinite(got) == np.isfinite(ref)).all()
    inside = ~(np.isfinite(ext) & ~np.isfinite(ref))
    assert (np.isnan(got) == np.isnan(ref))[inside].all()
    fin = np.isfinite(ref)
    with np.errstate(all="ignore"):
        scale = np.abs(np.where(np.isfinite(E), E, 0)) @ np.abs(np.where(np.isfinite(q), q, 0))
        assert np.all((np.abs(got - ref) <= 1e-13 * scale)[fin])


def test_solve_under_capture():
    """A captured solve takes the form without scratch and replays to the same values."""
    N, T = 300, 4
    X = inputs.nodes(N, 4)
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_global_factor(_t(X), rbfsl.IMQ, 2.0, LU, perm)
    q = _t(np.random.default_rng(1).standard_normal((N, T)))
    ref, c = torch.empty_like(q), torch.zeros_like(q)
    rbfsl.rbfsl_global_solve(LU, perm, q, ref)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        rbfsl.rbfsl_global_solve(LU, perm, q, c)
    g.replay()
    torch.cuda.synchronize()
    assert (c - ref).abs().max().item() <= 1e-9 * ref.abs().max().item()


# the update's three arrangements (warps along the inner dimension 4, 2 and 1, by blocks of 16 rows) and their
# edges: 16, 17, 32, 33 and 64 columns over 128 + 1 to 5,002 rows, against the solve column by column
@pytest.mark.parametrize("N,T", [(129, 16), (1300, 17), (2700, 33), (2700, 64), (5002, 34), (5002, 64)])
def test_solve_update_arrangements(N, T):
    X = inputs.nodes(N, 6)
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_global_factor_chol(_t(X), rbfsl.IMQ, 0.1 * np.sqrt(N), LU, perm)
    q = _t(np.random.default_rng(N + T).standard_normal((N, T)))
    c, one = torch.empty_like(q), torch.empty((N, 1), dtype=torch.float64, device=DEV)
    rbfsl.rbfsl_global_solve(LU, perm, q, c)
    L = torch.tril(LU, -1) + torch.eye(N, dtype=torch.float64, device=DEV)
    r = L @ (torch.triu(LU) @ c) - q[perm.long()]
    for t in (0, T - 1):
        rbfsl.rbfsl_global_solve(LU, perm, q[:, t:t + 1].contiguous(), one)
        assert (c[:, t:t + 1] - one).abs().max() <= 1e-10 * one.abs().max()
    A_inf = (L.abs() @ torch.triu(LU).abs()).sum(1).max().item()
    assert r.abs().max().item() <= lu_residual_bound(N, A_inf, c.cpu().numpy())
