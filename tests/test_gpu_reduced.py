"""Stencil weights in the reduced (null-space) form at the edges of its launch shapes and panels,
and the systems that take the pivoted factorisation instead."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

import _parity  # noqa: E402
import test_gpu_local as loc  # noqa: E402

pytestmark = pytest.mark.gpu


# K = n - M of 1, 7, 8, 9, 16 (panels of 8); n + 1 of 32 and 33 (a warp of points); one harmonic
# (K up to 158), 64 harmonics, the largest systems; one and four warps per point; and exponents
# above the harmonics' order (p = 9, ell = 2) and n < M, which keep the indefinite factorisation
@pytest.mark.parametrize("n,ell,p", [(10, 2, 5), (16, 2, 5), (17, 2, 3), (18, 2, 5), (32, 3, 7), (31, 2, 5), (32, 2, 5),
                                     (9, 0, 1), (159, 0, 1), (135, 4, 9), (96, 7, 15), (84, 4, 9), (55, 3, 7),
                                     (84, 4, 3), (31, 2, 9)])
def test_reduced_weights_interpolate(orc, n, ell, p):
    N = 1200
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


def test_rank_deficient_harmonics_are_singular():
    """Nodes on the equator: the harmonic proportional to z vanishes at all of them, P has a zero
    column and the system is exactly singular, as by the indefinite factorisation."""
    n = 12
    a = 2.0 * math.pi * np.arange(40) / 40
    X = np.stack([np.cos(a), np.sin(a), np.zeros_like(a)], axis=1)
    b = a[:7] + 0.03
    P = np.stack([np.cos(b), np.sin(b), np.zeros_like(b)], axis=1)
    I = np.argsort(((P[:, None] - X[None]) ** 2).sum(-1), axis=1)[:, :n]
    w = torch.empty((len(P), n), dtype=torch.float64, device="cuda")
    st = torch.empty(len(P), dtype=torch.int32, device="cuda")
    rbfsl.rbfsl_stencil_weights(loc._t(X), loc._t(I, torch.int32), n, 1, rbfsl.PHS, 3, loc._t(P), w, st)
    assert (st.cpu().numpy() == rbfsl.ESINGULAR).all()
    assert np.isnan(w.cpu().numpy()).all()


# centre stencils: half a warp per point (K <= 32, M <= 16) with a ragged last block, a full warp,
# products on both pipes, one node besides the pivots, and exponents that keep the LU factors
@pytest.mark.parametrize("n,ell,p", [(31, 2, 5), (41, 2, 5), (42, 2, 5), (49, 3, 7), (84, 4, 9), (10, 2, 5), (17, 1, 3),
                                     (31, 2, 9)])
@pytest.mark.parametrize("prec", [rbfsl.FP64, rbfsl.MIXED])
def test_centre_stencils_match_oracle(orc, n, ell, p, prec):
    N, dt, steps = 901, 1.0 / 60, 3
    X = inputs.nodes(N, 11)
    vp = inputs.deformation_params(2.0, 1.0)
    fields = inputs.TracerSet([lambda P: inputs.gaussian_hills(P, [[0.6, 0.0, 0.8], [0.0, 1.0, 0.0]]),
                               lambda P: inputs.cosine_bell(P, [1.0, 0.0, 0.0], 0.9)])
    q = fields(X)
    c = rbfsl.Context(0)
    c.set_nodes(X)
    c.set_velocity(rbfsl.VEL_DEFORM_Y2, vp)
    c.set_method(rbfsl.LOCAL, rbfsl.CENTER)
    c.set_stencil_size(n)
    c.set_sh_degree(ell)
    c.set_kernel(rbfsl.PHS, p)
    c.set_precision(prec)
    c.set_dt(dt)
    c.set_tracers(q)
    c.step(steps)
    got, st = c.get_q(), c.get_stats()
    c.close()
    assert st.singular_points == 0 and st.knn_failures == 0
    ref = orc.local_run(X, q, n, ell, p, rbfsl.VEL_DEFORM_Y2, vp, dt, steps, mode=orc.CENTER)
    exact = _parity.exact_field(fields, X, rbfsl.VEL_DEFORM_Y2, vp, steps * dt)
    _parity.check_run(f"centre n={n} ell={ell} r^{p} prec={prec}", got, ref, exact, strict=False)


# coarse node sets, where the reduced matrix is worst conditioned: one step at the oracle's noise floor
# (its change when every coordinate moves by one ulp; five times it, plus 1e-12 of max|q|)
@pytest.mark.parametrize("N,n,ell,p", [(642, 84, 4, 9), (900, 84, 4, 9), (642, 55, 3, 7), (642, 31, 2, 5)])
def test_centre_stencils_on_coarse_nodes(orc, N, n, ell, p):
    X = inputs.nodes(N, 11)
    vp = inputs.nl_deformation_params(5.0)
    rng = np.random.default_rng(N)
    q = np.stack([inputs.plane_wave_field(rng, 6.0)(X) for _ in range(3)], axis=1)

    def reference(Y):
        return orc.local_run(Y, q, n, ell, p, rbfsl.VEL_NL, vp, 0.1, 1, mode=orc.CENTER)

    ref = reference(X)
    floor = np.abs(reference(np.nextafter(X, X + rng.choice([-1.0, 1.0], size=X.shape))) - ref).max()
    c = rbfsl.Context(0)
    c.set_nodes(X)
    c.set_velocity(rbfsl.VEL_NL, vp)
    c.set_method(rbfsl.LOCAL, rbfsl.CENTER)
    c.set_stencil_size(n)
    c.set_sh_degree(ell)
    c.set_kernel(rbfsl.PHS, p)
    c.set_dt(0.1)
    c.set_tracers(q)
    c.step(1)
    err = np.abs(c.get_q() - ref).max()
    c.close()
    assert err <= 5 * floor + 1e-12 * np.abs(q).max()


# two warps per point (up to 28 KB a point): in the batch two points share a block, the last block of an odd
# node count holds one; the context's kernel has a block per point
@pytest.mark.parametrize("n,ell,N", [(33, 3, 901), (55, 3, 643), (60, 3, 1200)])
def test_two_warps_per_point_in_a_batch(n, ell, N):
    X = inputs.nodes(N, 3)
    q = np.stack([inputs.gaussian_hills(X, [[0.6, 0.0, 0.8]]), inputs.cosine_bell(X, [1.0, 0.0, 0.0], 0.9)], axis=1)
    vp = inputs.deformation_params(2.0, 1.0)
    b = rbfsl.Batch(0, stream=torch.cuda.Stream())
    i = b.add(X, q, n, ell, 2 * ell + 1, rbfsl.VEL_DEFORM_Y2, vp, 1.0 / 60, mode=rbfsl.DIRECT, precision=rbfsl.FP64)
    b.step(2)
    got = b.get_q(i)
    b.close()
    c = rbfsl.Context(0)
    c.set_nodes(X)
    c.set_velocity(rbfsl.VEL_DEFORM_Y2, vp)
    c.set_method(rbfsl.LOCAL, rbfsl.DIRECT)
    c.set_stencil_size(n)
    c.set_sh_degree(ell)
    c.set_kernel(rbfsl.PHS, 2 * ell + 1)
    c.set_dt(1.0 / 60)
    c.set_tracers(q)
    c.step(2)
    np.testing.assert_array_equal(got, c.get_q())
    c.close()
