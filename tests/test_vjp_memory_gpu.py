"""Device memory that the adjoint's records take and keep."""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu
KEPT = 8 << 30  # records that all handles together keep between calls


def _free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _run(s, K, every=10):
    s.set_state(*s.first)
    return s.vjp(K, ybar=np.ones((1, s.samples_for(K), 11)), checkpoint_every=every)


def _sim():
    from paper_2604_12505_gb300.sph import Sim
    s = Sim(W.JVP)
    s.first = s.state()
    _run(s, 1)
    return s


def test_handles_keep_eight_gigabytes_together():
    torch = need_gpu()
    sims = [_sim() for _ in range(6)]
    free = _free(torch)
    want = None
    for s in sims * 2:
        g = _run(s, 90)  # 2 GB of records each
        want = want or g
        assert all(torch.equal(a, b) for a, b in zip(g, want))
        assert free - _free(torch) <= KEPT + (64 << 20)
    for s in sims:
        s.close()
    assert free - _free(torch) <= 64 << 20


def test_records_take_what_the_checkpoints_leave():
    """91 checkpoints are 45 MB; so much room is left that the records of half
    the steps would leave less than that."""
    torch = need_gpu()
    s = _sim()
    free = _free(torch)
    half = _run(s, 45, 1)
    records = free - _free(torch)
    s.close()
    s = _sim()
    want = _run(s, 90, 1)
    s.close()
    s = _sim()
    torch.cuda.empty_cache()
    y = torch.ones((1, s.samples_for(90), 11), dtype=torch.float64, device="cuda")
    fill = torch.empty(_free(torch) - records - (24 << 20), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        s.set_state(*s.first)
        got = s.vjp(90, ybar=y, checkpoint_every=1)
        assert all(torch.equal(a, b) for a, b in zip(got, want))
    del fill, half
    s.close()
    torch.cuda.empty_cache()
