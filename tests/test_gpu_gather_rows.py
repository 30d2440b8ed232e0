"""Gather-dot at the edges of its row shapes: odd and even tracer counts up to and above a warp's lanes, row
lengths with and without 16-byte loads, few and many rows, a failed stencil. Sums of n products in FP64 or
FP32 with a unit bound on each: n eps against the plain product."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,eps", [(torch.float64, 2.0 ** -52), (torch.float32, 2.0 ** -23)])
@pytest.mark.parametrize("T", [1, 2, 3, 5, 6, 8, 11, 12, 31, 32, 33, 48, 64, 65, 130])
@pytest.mark.parametrize("n,Nq", [(31, 77), (40, 77), (84, 3001), (1, 5), (7, 1)])
def test_gather_rows(dtype, eps, T, n, Nq):
    rng = np.random.default_rng([T, n])
    N = 300
    I, w, q = rng.integers(0, N, (Nq, n)), rng.uniform(-1, 1, (Nq, n)), rng.uniform(-1, 1, (N, T))
    w, q = (np.asarray(torch.tensor(a, dtype=dtype), dtype=float) for a in (w, q))
    if Nq > 5:
        I[4, n // 2] = -1
    dev = lambda a, d: torch.tensor(a, dtype=d, device="cuda")
    out = torch.empty((Nq, T), dtype=dtype, device="cuda")
    rbfsl.rbfsl_gather_dot(dev(I, torch.int32), dev(w, dtype), dev(q, dtype), out)
    got = out.cpu().numpy().astype(float)
    ref = np.einsum("ij,ijt->it", w, q[I])
    if dtype == torch.float32:  # the difference form q_c + sum w (q - q_c), as for weights that sum to one
        c = q[I[:, 0]]
        ref = c + np.einsum("ij,ijt->it", w, q[I] - c[:, None])
    ok = np.arange(Nq) != 4 if Nq > 5 else np.ones(Nq, bool)
    assert np.abs(got - ref)[ok].max() <= 2 * (n + 2) * n * eps
    assert np.isnan(got[~ok]).all()
