"""Health flags of the adjoint's recorded steps.

At h = 2 dx the small tank's 4x4 tiles have more particles around them (532)
than a tile stages (432), while 8x8 tiles hold theirs (650 of 1,200).  The
adjoint always takes 4x4 tiles, so it cannot differentiate such a step, and
must say so however the forward steps ran.
"""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,every", [(0, 10), (5, 10), (5, 2)])
@pytest.mark.parametrize("tanks", [1, 3])
def test_vjp_reports_a_tile_that_it_cannot_stage(tile, every, tanks):
    need_gpu()
    from paper_2604_12505_gb300 import _lib
    from paper_2604_12505_gb300.sph import Sim
    # the last tank of the batch is the one that does not fit
    cfgs = [W.SMALL] * (tanks - 1) + [dict(W.SMALL, h_over_dx=2.0)]
    with Sim(cfgs) as s:
        s.set_tile(tile)
        state = s.state()
        if tile == 5:
            s.step(6)
            assert s.check(raise_on_error=False) == 0
        s.set_state(*state)
        s.vjp(6, ybar=np.ones((tanks, s.samples_for(6), 11)), checkpoint_every=every)
        assert s.check(raise_on_error=False) & _lib.FLAG_STAGE_FULL
        with pytest.raises(_lib.SphError):
            s.check()
    with Sim(W.SMALL) as s:
        s.set_tile(tile)
        s.vjp(6, ybar=np.ones((1, s.samples_for(6), 11)), checkpoint_every=every)
        assert s.check() == 0
