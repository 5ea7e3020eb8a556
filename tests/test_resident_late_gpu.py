"""The steps of a long call while the fluid falls to one side: the cluster's CTAs
share the tank anew as it moves, so that a call of many steps takes no longer a
step than calls of few (1.4 times as long at most, with 2.5 when the shares
stayed those of the call's start), and gives the same."""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def test_a_long_call_follows_the_fluid():
    torch = need_gpu()
    from paper_2604_12505_gb300.sph import Sim
    n = 1000
    with Sim(dict(W.PAPER_RINGS, fill=0.2, grav_x=3.0)) as s:
        first = s.state()
        time, end = {}, {}
        for each in (100, n, 100, n, 100, n):
            s.set_state(*first)
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            for _ in range(n // each):
                s.step(each, record=False)
            e[1].record()
            torch.cuda.synchronize()
            time[each] = min(time.get(each, np.inf), e[0].elapsed_time(e[1]))
            end[each] = s.state()
    assert time[n] <= 1.4 * time[100]
    for a, b in zip(end[n], end[100]):
        assert torch.equal(a, b)
