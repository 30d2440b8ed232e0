"""Stateless global calls on one stream leave a capture of another stream alone, whichever thread and
mode it runs in."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _t(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a)).to(DEV, dtype)


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
@pytest.mark.parametrize("own_thread", [False, True])
def test_calls_beside_a_capture(mode, own_thread):
    N, eps = 1000, 4.0
    x = _t(inputs.nodes(N, 3))
    LU = torch.empty((N, N), dtype=torch.float64, device=DEV)
    perm = torch.empty(N, dtype=torch.int32, device=DEV)
    rbfsl.rbfsl_global_factor(x, rbfsl.IMQ, eps, LU, perm)
    q = _t(np.random.default_rng(1).standard_normal((N, 3)))
    res = [[torch.zeros_like(q) for _ in range(2)] for _ in range(2)]
    other = torch.cuda.Stream()

    def calls(c, o, stream):
        rbfsl.rbfsl_global_solve(LU, perm, q, c, stream=stream)
        rbfsl.rbfsl_global_eval(x, x, rbfsl.IMQ, eps, c, o, stream=stream)

    calls(*res[0], None)
    a, b = torch.ones(100, device=DEV), torch.zeros(100, device=DEV)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode=mode):
        torch.add(a, a, out=b)
        if own_thread:
            t = threading.Thread(target=calls, args=(*res[1], other))
            t.start()
            t.join()
        else:
            calls(*res[1], other)
    g.replay()
    torch.cuda.synchronize()
    assert b.sum().item() == 200.0
    for u, v in zip(*res):
        assert torch.equal(u, v)
