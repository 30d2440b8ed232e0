"""FP64 results stored as FP32 pairs: hi = fl32(v), lo = fl32(v - hi), as numpy's conversions give
them, also at ties, at the end of FP32's range and for values that are not finite."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV, dtype)


def _split(v):
    with np.errstate(all="ignore"):
        hi = v.astype(np.float32)
        return np.stack([hi, (v - hi.astype(np.float64)).astype(np.float32)], axis=-1)


def test_pair_split_is_the_conversions():
    """1 x value through the pair product, whose sum of one term is exact."""
    rng = np.random.default_rng(1)
    m, u = np.float32(1.0), 2.0 ** -24
    special = [(1.0, u), (1.0 + 2 * u, u), (1.0 + 4 * u, u), (1.0, u * (1 + 2.0 ** -20)), (-1.0, -u), (1.0, 0.0),
               (0.0, 0.0), (np.finfo(np.float32).max, 2.0 ** 103), (-np.finfo(np.float32).max, -(2.0 ** 103)),
               (np.finfo(np.float32).max, 2.0 ** 102), (np.inf, 0.0), (-np.inf, 0.0), (np.nan, np.nan), (np.nan, 0.0)]
    hi = (rng.standard_normal(500) * 10.0 ** rng.uniform(-20, 20, 500)).astype(np.float32)
    lo = (hi * rng.uniform(-0.5, 0.5, 500).astype(np.float32) * m * np.float32(2.0 ** -23)).astype(np.float32)
    q = np.concatenate([np.array(special, dtype=np.float32), np.stack([hi, lo], axis=1)])
    E = np.zeros((1, 1, 2), dtype=np.float32)
    E[..., 0] = 1.0
    out = torch.empty((1, len(q), 2), dtype=torch.float32, device=DEV)
    rbfsl.rbfsl_cardinal_apply(_t(E, torch.float32), _t(q[None], torch.float32), out)
    with np.errstate(all="ignore"):
        v = q[:, 0].astype(np.float64) + q[:, 1].astype(np.float64)
    np.testing.assert_array_equal(out.cpu().numpy()[0], _split(v))


def test_failed_weights_are_nan_in_both_parts():
    """RBFSL_F32X2 weights: the split of the FP64 weights; a failed row is NaN, high and low part."""
    n, ell, p = 31, 2, 5
    X = inputs.nodes(642, 3)
    I = np.stack([np.arange(n), np.arange(50, 50 + n), np.arange(100, 100 + n)]).astype(np.int32)
    I[1, 4] = -1
    P = X[[1, 52, 103]] + 1e-3
    P /= np.linalg.norm(P, axis=1, keepdims=True)
    w = torch.empty((3, n), dtype=torch.float64, device=DEV)
    w2 = torch.empty((3, n, 2), dtype=torch.float32, device=DEV)
    for o in (w, w2):
        st = torch.zeros(3, dtype=torch.int32, device=DEV)
        rbfsl.rbfsl_stencil_weights(_t(X), _t(I, torch.int32), n, ell, rbfsl.PHS, p, _t(P), o, status=st)
        assert st.tolist() == [rbfsl.OK, rbfsl.EKNN, rbfsl.OK]
    np.testing.assert_array_equal(w2.cpu().numpy(), _split(w.cpu().numpy()))
    assert np.isnan(w2[1].cpu().numpy()).all()


def test_nan_through_the_pair_evaluation():
    X = inputs.nodes(200, 4)
    c = np.ones((200, 3))
    c[7, 1] = np.nan
    out = torch.empty((200, 3, 2), dtype=torch.float32, device=DEV)
    rbfsl.rbfsl_global_eval_pairs(_t(X), _t(X), rbfsl.IMQ, 2.0, _t(c), out)
    o = out.cpu().numpy()
    assert np.isnan(o[:, 1]).all() and np.isfinite(o[:, [0, 2]]).all()
