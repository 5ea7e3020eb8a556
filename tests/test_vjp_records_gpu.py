"""The adjoint of a window longer than its records' room (2 GB: about 90 steps
of the 15,532-particle tank), which is reversed group by group, against the
same window as two calls, the second half's adjoint handed to the first.

Both take the same arithmetic but for the re-binning of the state between the
calls, which reorders the sums of the few particles that change a cell: FP32
rounding, 1e-4 of the largest entry as in the transpose test.
"""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu, oracle_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("every", [7, 50, 200])
def test_groups_of_segments_equal_two_calls(orc, every):
    torch = need_gpu()
    from paper_2604_12505_gb300.sph import Sim
    cfg, K = dict(W.JVP, outer_every=10), 120
    xv, *_ = oracle_state(orc, cfg, 0.1, 0.2, seed=4)
    body = np.array([0.002, -0.001, 0.05, 0.01, 0.0, 0.2])
    u = W.bang_bang_slew(K, cfg["dt"], tau=400.0, t1=K * cfg["dt"] / 2)
    rng = np.random.default_rng(3)
    yb, xb, bb = rng.normal(size=(1, 12, 11)), rng.normal(size=(xv.shape[0], 4)).astype(np.float32), rng.normal(size=(1, 6))
    h = K // 2
    with Sim(cfg) as s:
        s.set_state(xv, body)
        x0, b0, u0 = s.vjp(K, u=u[None], ybar=yb, xvbar=xb, bodybar=bb, checkpoint_every=every)
        s.check()
        s.set_state(xv, body)
        s.step(h, u=u[None, :h], record=False)
        mid = s.state()
        x1, b1, u1 = s.vjp(h, u=u[None, h:], ybar=yb[:, 6:], xvbar=xb, bodybar=bb)
        s.set_state(xv, body)
        x2, b2, u2 = s.vjp(h, u=u[None, :h], ybar=yb[:, :6], xvbar=x1, bodybar=b1)
        assert torch.allclose(s.state()[0], mid[0], rtol=0, atol=1e-6)
        s.check()
    for got, want in ((x0, x2), (b0, b2), (u0, torch.cat([u2, u1], 1))):
        assert (got - want).abs().max() <= 1e-4 * want.abs().max()
