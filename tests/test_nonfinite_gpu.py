"""A particle whose position is not finite meets nothing: it is reported, and the
rest of the tank and the body go on as with the passes of one thread per
particle, which the same tank takes in a batch with one that fills the GPU.
Equal bit for bit, with four lanes per particle and in the resident kernel; the
particle's own row and the fluid's centre of mass apart.
"""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

LANES, RESIDENT = dict(W.BASE, dx=0.009, fill=0.6, outer_every=1), dict(W.PAPER_RINGS, outer_every=1)


@pytest.mark.parametrize("cfg", [LANES, RESIDENT], ids=["lanes", "resident"])
# the particles of a wall tile beside which the bad one is sorted
@pytest.mark.parametrize("height", [-0.1, 0.0, 0.05, 0.1])
@pytest.mark.parametrize("bad", [(np.nan, None), (-np.inf, None), (None, np.nan), (np.nan, np.inf)])
def test_a_particle_that_is_not_finite_leaves_the_others_alone(cfg, height, bad):
    need_gpu()
    from paper_2604_12505_gb300 import _lib
    from paper_2604_12505_gb300.sph import Sim
    large = dict(W.LARGE, outer_every=1)
    got, n = [], 5
    for tanks in ([cfg], [cfg, large]):
        with Sim(tanks) as s:
            xv, body = s.state()
            own = xv[:s.offsets[1]].cpu().numpy()
            i = int(np.argmin(np.hypot(own[:, 0] + cfg["R"], own[:, 1] - height * cfg["R"])))
            for c, v in enumerate(bad):
                if v is not None:
                    xv[i, c] = v
            body[0] = body.new_tensor([0.0, 0.0, 0.1, 0.02, -0.01, 0.1])
            s.set_state(xv, body)
            y = s.step(n)[0].cpu().numpy()
            assert s.check(raise_on_error=False) & _lib.FLAG_NAN
            xv, body = s.state()
            got.append((y[:, :9], np.delete(xv[:s.offsets[1]].cpu().numpy(), i, axis=0), body[0].cpu().numpy()))
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.isfinite(b).all()
        np.testing.assert_array_equal(a, b)
