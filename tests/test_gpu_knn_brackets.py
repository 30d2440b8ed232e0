"""Neighbour searches where the node density varies too much for one rescaled radius: clusters, a cap,
a lattice with many equal distances, nodes off the unit sphere and queries far from them. Every
query has an answer, the brute-force one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _unit(v):
    return v / np.linalg.norm(v, axis=1, keepdims=True)


def _nodes(kind, rng):
    if kind == "cluster":
        return _unit(np.array([0.3, 0.2, 0.9]) + 1e-4 * rng.standard_normal((2000, 3)))
    if kind == "cluster in a sphere":
        return np.concatenate([inputs.nodes(642, 1), _unit(np.array([0.3, 0.2, 0.9]) + 1e-5 * rng.standard_normal((1000, 3)))])
    if kind == "cap":
        return _unit(np.array([0.0, 0.0, 1.0]) + 0.2 * rng.standard_normal((4000, 3)))
    if kind == "radius 2.5":
        return 2.5 * inputs.nodes(2000, 2)
    return np.stack(np.meshgrid(*[np.linspace(-1.0, 1.0, 13)] * 3), -1).reshape(-1, 3)


@pytest.mark.parametrize("kind", ["cluster", "cluster in a sphere", "cap", "radius 2.5", "lattice"])
@pytest.mark.parametrize("k", [1, 2, 7, 15, 31, 84])
def test_every_query_is_answered(orc, kind, k):
    rng = np.random.default_rng(k)
    X = np.ascontiguousarray(_nodes(kind, rng))
    Q = np.concatenate([X[:200] + 1e-3 * rng.standard_normal((200, 3)), inputs.random_unit_vectors(150, rng),
                        3.0 * inputs.random_unit_vectors(50, rng)])
    ix = rbfsl.rbfsl_knn_index_create(torch.as_tensor(X).to(DEV), 30)
    idx = torch.empty((len(Q), k), dtype=torch.int32, device=DEV)
    st = torch.empty(len(Q), dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_knn_query(ix, torch.as_tensor(Q).to(DEV), k, idx, st)
    ix.close()
    assert (st.cpu().numpy() == rbfsl.OK).all()
    np.testing.assert_array_equal(idx.cpu().numpy(), orc.knn(X, Q, k))
