"""What the server charges a partition-of-unity request covers what the same problem holds on the
device in a context of its own."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1804_01609_gb300 import inputs, rbfsl  # noqa: E402

pytestmark = pytest.mark.gpu


# many small patches (their factors are padded to 16 x 16 tiles), the usual ones, exponents without the reduced form
@pytest.mark.parametrize("N,n,ell,p,T", [(163842, 31, 2, 5, 1), (163842, 25, 1, 3, 4), (40962, 100, 3, 7, 16), (10242, 60, 2, 9, 3)])
def test_charge_covers_the_request(N, n, ell, p, T):
    X = inputs.nodes(N, 3)
    q, C = np.zeros((N, T)), inputs.fibonacci_nodes(math.ceil(2.5 * N / n))
    vp = inputs.rigid_rotation_params([0.0, 0.0, 1.0], 1.0)
    c = rbfsl.Context(0)
    c.set_nodes(X)
    c.set_velocity(rbfsl.VEL_RIGID, vp)
    c.set_method(rbfsl.PU)
    c.set_stencil_size(n)
    c.set_sh_degree(ell)
    c.set_kernel(rbfsl.PHS, p)
    c.set_pu(C)
    c.set_dt(0.01)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    c.set_tracers(q)
    c.step(1)
    held = max(c.get_stats().device_bytes, free - torch.cuda.mem_get_info()[0])
    c.close()
    s = rbfsl.Server(0, budget_bytes=4 * 10 ** 9, max_slots=2)
    t = s.submit(X, q, n, ell, p, rbfsl.VEL_RIGID, vp, 0.01, 1, method=rbfsl.PU, centers=C)
    s.wait_idle(100)
    st = s.result(t)[1]
    s.close()
    assert st.status == rbfsl.OK and st.device_bytes >= held
