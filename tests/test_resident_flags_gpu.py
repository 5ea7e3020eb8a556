"""A tank whose 4x4 tiles have more particles around them than the step kernels
stage (432) is refused however many steps a call takes: by the step kernels
(one step), by the cluster that keeps a small tank in shared memory (three and
more), and by the passes of a batch.  Particles around the fullest tile, on
the spawn lattice: 412, 420 and 400 below the limit, 441, 532 and 576 above it.
"""
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fill,h,full", [(0.5, 1.75, False), (0.9, 1.69, False), (0.9, 1.7, False), (0.9, 1.75, True),
                                         (0.5, 2.0, True), (0.9, 2.0, True)])
@pytest.mark.parametrize("how", ["one", "three", "relax", "batch"])
def test_tiles_that_cannot_be_staged_are_reported(fill, h, full, how):
    need_gpu()
    from paper_2604_12505_gb300 import _lib
    from paper_2604_12505_gb300.sph import Sim
    cfg = dict(W.SMALL, fill=fill, h_over_dx=h)
    with Sim([cfg, W.JVP] if how == "batch" else cfg) as s:
        if how == "relax":
            s.relax(4, 0.01)
        else:
            s.step(1 if how == "one" else 3)
        flags = s.check(raise_on_error=False)
        assert bool(flags & _lib.FLAG_STAGE_FULL) == full
        if not full:
            assert flags == 0
