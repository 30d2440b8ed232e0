"""RBF-PU coefficients from the reduced factors and the blend at the edges of their tiles: patch sizes
around the 16-row tiles, one to 49 harmonics, tracer counts around the 8-column tiles, the 16-tracer
blocks and the lanes of a warp; systems that keep LU factors; fields with a NaN tracer.

Tolerance as in test_gpu_pu.py: 5 times the oracle's change when every coordinate moves by one ulp,
plus 1e-12 of max|q| (FP64) or the pair sums' rounding: 2^-45 (factor, coefficient, dropped product and
sum, 2^-48 each, and a factor of two) of the largest sum of |terms|, taken from the oracle's coefficients."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

import _parity  # noqa: E402
import test_gpu_pu as pu  # noqa: E402

pytestmark = pytest.mark.gpu


def _fields(X, T, rng):
    q = np.stack([inputs.plane_wave_field(rng, 6.0)(X) for _ in range(T)], axis=1)
    return q * 10.0 ** rng.integers(-6, 7, size=T)  # tracers of very different sizes


# (n, ell, p): K a little below and above 16 and 32 rows, M = 1, 4, 9, 16, 25, 49; p above the
# harmonics' order and patches of fewer nodes than harmonics keep the LU factors
@pytest.mark.parametrize("n,ell,p", [(14, 0, 1), (20, 1, 3), (31, 2, 5), (50, 3, 7), (100, 3, 7), (84, 4, 9), (90, 6, 11),
                                     (40, 1, 7), (20, 3, 7)])
@pytest.mark.parametrize("T", [1, 2, 9])
def test_systems(orc, n, ell, p, T):
    _check(orc, n, ell, p, T, 701)


@pytest.mark.parametrize("T", [3, 7, 8, 15, 16, 17, 24, 33, 66])
def test_tracer_counts(orc, T):
    _check(orc, 40, 2, 5, T, 1203)


def _sum_of_terms(orc, ref, X, P, q, ell, p):
    """The largest sum of |terms| of a patch's interpolant over the patches and points."""
    coef, off, T = ref.coefficients(q)
    Y, worst = np.abs(orc.sh_eval(ell, P)), 0.0
    for l, om in enumerate(ref.Om):
        own = np.linalg.norm(P - om, axis=1) < ref.R
        I = ref.members[ref.mstart[l]:ref.mstart[l + 1]]
        c = np.abs(coef[off[l]:off[l] + (len(I) + (ell + 1) ** 2) * T]).reshape(-1, T)
        terms = np.concatenate([np.linalg.norm(P[own][:, None] - X[I], axis=2) ** p, Y[own]], axis=1) @ c
        worst = max(worst, terms.max(initial=0.0))
    return worst


def _check(orc, n, ell, p, T, Nq):
    N = 1203
    X, Om, R = pu._setup(N, n)
    rng = np.random.default_rng([n, T])
    P = inputs.random_unit_vectors(Nq, rng)  # Nq = N: points in the node grid's order
    q = _fields(X, T, rng)
    size = np.abs(q).max(axis=0)
    ref = orc.PUInterpolator(X, Om, n, ell, p, R=R).apply(P, q).reshape(Nq, T) / size
    s = np.random.default_rng(0).choice([-1.0, 1.0], size=X.shape)
    alt = orc.PUInterpolator(np.nextafter(X, X + s), Om, n, ell, p, R=R).apply(P, q).reshape(Nq, T) / size
    floor = np.abs(alt - ref).max()
    pairs_tol = 2.0 ** -45 * _sum_of_terms(orc, orc.PUInterpolator(X, Om, n, ell, p, R=R), X, P, q / size, ell, p)
    for pairs, tol in ((False, 1e-12), (True, 1e-12 + pairs_tol)):
        got, st = pu._gpu_apply(X, Om, R, q, P, ell=ell, power=p, pairs=pairs)
        assert (st == 0).all()
        err = np.abs(got / size - ref).max()
        _parity.record(test=f"PU n={n} ell={ell} r^{p} T={T} pairs={pairs}", oracle_floor=float(floor), gpu_diff=float(err))
        assert err <= 5 * floor + tol


def test_nan_and_zero_tracers_keep_to_themselves():
    N, n, T = 1203, 40, 5
    X, Om, R = pu._setup(N, n)
    rng = np.random.default_rng(3)
    P = inputs.random_unit_vectors(400, rng)
    q = _fields(X, T, rng)
    q[:, 2] = 0.0
    ref, _ = pu._gpu_apply(X, Om, R, q, P, ell=2, power=5)
    bad = q.copy()
    bad[7, 1] = np.nan
    bad[9, 3] = np.inf
    got, st = pu._gpu_apply(X, Om, R, bad, P, ell=2, power=5)
    assert (st == 0).all()
    for c in (0, 2, 4):
        assert (got[:, c] == ref[:, c]).all()
    assert (got[:, 2] == 0.0).all()
    near = np.linalg.norm(P[:, None] - X[None, [7, 9]], axis=2) < 0.2 * R
    assert np.isnan(got[near[:, 0], 1]).all() and not np.isfinite(got[near[:, 1], 3]).any()
    far = np.linalg.norm(P[:, None] - X[None, [7, 9]], axis=2) > 2.0 * R
    assert (got[far[:, 0], 1] == ref[far[:, 0], 1]).all() and (got[far[:, 1], 3] == ref[far[:, 1], 3]).all()


def test_more_points_than_one_launch_takes():
    """Values do not depend on how the points fall into launches of at most 16,384 (small node sets)."""
    N, n, T = 1203, 40, 3
    X, Om, R = pu._setup(N, n)
    rng = np.random.default_rng(5)
    P = inputs.random_unit_vectors(2 * 16384 + 5, rng)
    q = _fields(X, T, rng)
    got, st = pu._gpu_apply(X, Om, R, q, P, ell=2, power=5)
    assert (st == 0).all()
    for a, b in ((0, 9001), (9001, 25000), (25000, len(P))):
        part, _ = pu._gpu_apply(X, Om, R, q, P[a:b], ell=2, power=5)
        assert (part == got[a:b]).all()
