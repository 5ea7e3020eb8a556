"""Steps with four lanes per particle (tanks whose tiles all have a place on the
GPU at once) against the passes with a thread per particle, which the same tank
takes in a batch with one that fills the GPU.  Both round and add alike, so
samples, particles and body are equal bit for bit; and, as the passes of chained
steps start early, one call of many steps equals calls of one step.
"""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

BASE, PAPER = dict(W.BASE, dx=0.009, fill=0.6), dict(W.PAPER_RINGS, R=0.2, dx=0.004, fill=0.6)

CASES = {
    "more than a tank that is kept in shared memory": (BASE, 41, {}),
    # tiles of more particles than the 128 taken at once
    "paper": (PAPER, 41, {}),
    "clamped": (dict(PAPER, ghost_pressure_clamp=1), 20, {}),
    # more ghosts around a tile than are staged
    "rings": (dict(BASE, n_rings=12), 12, {}),
    "dense": (dict(BASE, h_over_dx=1.65), 12, {}),
    "relaxed": (BASE, 35, dict(relax=True)),
    "a small tank's single steps": (W.TINY, 5, dict(each=1)),
}


@pytest.mark.parametrize("name", list(CASES))
def test_lanes_equal_one_thread(name):
    torch = need_gpu()
    from paper_2604_12505_gb300.sph import Sim
    cfg, n, how = CASES[name]
    large = dict(W.LARGE, outer_every=cfg["outer_every"])
    rng = np.random.default_rng(5)
    u = rng.normal(size=(2, n, 3)) * [300.0, 300.0, 40.0]
    body = rng.normal(size=(2, 6)) * [0.001, 0.001, 0.1, 0.02, 0.02, 0.1]
    got = []
    for tanks, each in (([cfg], how.get("each", n)), ([cfg], 1), ([cfg, large], n)):
        with Sim(tanks) as s:
            k = len(tanks)
            s.set_state(s.state()[0], body[:k])
            if how.get("relax"):
                for _ in range(0, n, each):
                    s.relax(each, 0.01)
                y = np.zeros(0)
            else:
                y = np.concatenate([s.step(each, u=u[:k, i:i + each]).cpu().numpy() for i in range(0, n, each)], axis=1)[0]
            assert s.check(raise_on_error=False) == 0
            got.append((y, s.state()[0].cpu().numpy()[:s.offsets[1]], s.state()[1].cpu().numpy()[0]))
    for other in got[1:]:
        for a, b in zip(got[0], other):
            np.testing.assert_array_equal(a, b)
