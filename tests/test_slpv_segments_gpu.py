"""The adjoint in segments of the time axis where a segment's map overflows: a
state that nothing excites and nothing reads, and that would grow by `a` a
sample.  The state and its adjoint stay zero, and the gradient is that of the
same model with a stable one (a = 0.5).  FP32 sums in other parts: 1e-3 of the
largest entry, as in test_slpv_gpu.py.
"""
import numpy as np
import pytest

from tests.gpu_util import need_gpu
from tests.test_slpv_gpu import _data, _theta

pytestmark = pytest.mark.gpu
SC = np.array([20.0, 20.0, 2.0, 0.1, 0.1, 0.05], dtype=np.float32)


# segments of 80 and 1,875 samples, and two windows of 4 segments
@pytest.mark.parametrize("nx,n,T,a", [(4, 2, 2200, 4.0), (6, 1, 60000, 1.1), (8, 2, 2200, 4.0), (4, 300, 2500, 1.3)])
def test_a_map_that_overflows(nx, n, T, a):
    torch = need_gpu()
    from paper_2604_12505_gb300.slpv import VelocityModel, layout
    _, th = _theta(nx, 5)
    L, h = layout(nx), nx - 1
    u, y = _data(min(n, 4), T, 9, SC)
    reps = -(-n // u.shape[0])
    u, y = (torch.tensor(q, device="cuda").repeat(reps, 1, 1)[:n].contiguous() for q in (u, y))
    g = []
    for own in (0.5, a):
        for m in ("M0", "M1"):
            M = th[L[m]].reshape(nx + 3, nx + 3)
            M[h], M[:, h] = 0.0, 0.0
        th[L["W1"]].reshape(4, nx + 3)[:, h] = 0.0
        th[L["M0"]].reshape(nx + 3, nx + 3)[h, h] = own
        m = VelocityModel(nx=nx)
        m.set_params(th, SC)
        loss, grad = m.loss_grad(u, y)
        g.append(grad.cpu().numpy())
        assert np.isfinite(float(loss.item()))
        m.close()
    assert np.isfinite(g[1]).all()
    assert np.abs(g[1] - g[0]).max() <= 1e-3 * np.abs(g[0]).max()
