"""Stencil weights of systems without the reduced form (exponents above the harmonics' order) at the
edges of their launch shapes: one warp per point up to 12 KB, four warps in 72 registers up to 37 KB,
four warps above; the batch, with shapes of its own, gives the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

import test_gpu_local as loc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,ell,p", [(38, 2, 7), (39, 2, 7), (72, 3, 9), (73, 3, 9), (84, 4, 11)])
def test_weights_and_batch(orc, n, ell, p):
    N = 1201
    X = inputs.nodes(N, 5)
    P = loc._departures(X, 6)[:301]
    I = orc.knn(X, P, n)
    w = torch.empty((len(P), n), dtype=torch.float64, device="cuda")
    st = torch.empty(len(P), dtype=torch.int32, device="cuda")
    rbfsl.rbfsl_stencil_weights(loc._t(X), loc._t(I, torch.int32), n, ell, rbfsl.PHS, p, loc._t(P), w, st)
    assert (st.cpu().numpy() == 0).all()
    W = w.cpu().numpy()
    q = inputs.config_local_deformation(N=N, n_random=4).tracers(X)
    loc.assert_within_noise_floor(orc, X, I, P, q, np.einsum("ij,ijt->it", W, q[I]), ell, p)

    vp = inputs.deformation_params(2.0, 1.0)
    b = rbfsl.Batch(0, stream=torch.cuda.Stream())
    i = b.add(X, q, n, ell, p, rbfsl.VEL_DEFORM_Y2, vp, 1.0 / 60, mode=rbfsl.DIRECT, precision=rbfsl.FP64)
    b.step(2)
    got = b.get_q(i)
    b.close()
    c = rbfsl.Context(0)
    c.set_nodes(X)
    c.set_velocity(rbfsl.VEL_DEFORM_Y2, vp)
    c.set_method(rbfsl.LOCAL, rbfsl.DIRECT)
    c.set_stencil_size(n)
    c.set_sh_degree(ell)
    c.set_kernel(rbfsl.PHS, p)
    c.set_dt(1.0 / 60)
    c.set_tracers(q)
    c.step(2)
    np.testing.assert_array_equal(got, c.get_q())
    c.close()
