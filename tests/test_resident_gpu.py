"""Steps of tanks that one cluster of CTAs holds in its shared memory, against
the step kernels' path, which the same tanks take in a batch with one that is
too large for a cluster.  Both round and add alike, so results are equal bit for
bit: samples, particles, body, flags and the number of pairs.
"""
import numpy as np
import pytest

from paper_2604_12505_gb300 import workloads as W
from tests.gpu_util import need_gpu

pytestmark = pytest.mark.gpu

PAPER = dict(W.PAPER_RINGS, R=0.2, dx=0.006, fill=0.6)
LARGE = dict(W.BASE, dx=0.01, fill=0.3)  # 2,356 particles
BASE = dict(W.BASE, dx=0.02)

CASES = {
    # one tile's particles, on a few CTAs of the cluster; steps beyond one launch's
    "tiny": ([W.TINY], 1030, {}),
    "two steps and three": ([BASE], 5, dict(calls=(2, 3))),
    # tiles of more than 128 particles, whose threads sum two particles each
    "paper": ([PAPER], 60, {}),
    "clamped": ([dict(PAPER, ghost_pressure_clamp=1)], 60, {}),
    # nearly the most particles that fit
    "most": ([dict(PAPER, fill=0.62)], 40, {}),
    # the fluid falls to one side: more particles in a CTA than it takes at once
    "gathered": ([dict(PAPER, grav_x=3.0, grav_y=-1.2)], 400, {}),
    "relaxed": ([BASE], 41, dict(relax=True)),
    "held to an angle": ([dict(BASE, fill=0.3, outer_every=7)], 40, dict(ctrl=dict(omega=30.0, xi=0.7))),
    # eight CTAs a tank, tanks of different sizes
    "twelve": ([dict(PAPER, fill=0.05 + 0.05 * i) for i in range(8)] + [dict(BASE, outer_every=50)] * 4, 50, {}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_resident_steps_equal_step_kernels(name):
    torch = need_gpu()
    from paper_2604_12505_gb300.sph import Sim
    tanks, n, how = CASES[name]
    large = dict(LARGE, outer_every=tanks[0]["outer_every"])
    rng = np.random.default_rng(7)
    u = rng.normal(size=(len(tanks) + 1, n, 3)) * [300.0, 300.0, 40.0]
    body = rng.normal(size=(len(tanks) + 1, 6)) * [0.001, 0.001, 0.1, 0.02, 0.02, 0.1]
    got = []
    for extra in ([], [large]):
        with Sim(tanks + extra) as s:
            k = len(tanks + extra)
            xv = s.state()[0]
            s.set_state(xv, body[:k])
            if how.get("relax"):
                s.relax(n, 0.01)
                y = None
            else:
                ys, at = [], 0
                for m in how.get("calls", (n,)):
                    ref = None if "ctrl" not in how else np.tile(np.linspace(0.0, 0.4, s.samples_for(m)), (k, 1))
                    ys.append(s.step(m, u=u[:k, at:at + m], ctrl=how.get("ctrl"), theta_ref=ref).cpu().numpy())
                    at += m
                y = np.concatenate(ys, axis=1)
            pairs = s.pair_count()
            f = s.check(raise_on_error=False)
            # the state as the step kernels find it: a step of theirs, timed, and a sample after it
            s.time_kernels(2)
            xv, b = (t.cpu().numpy() for t in s.state())
            got.append((y, xv, b, f, pairs, s.offsets))
    with Sim(large) as s:
        s.set_state(s.state()[0], body[-1:])
        if how.get("relax"):
            s.relax(n, 0.01)
        else:
            for at, m in zip(np.cumsum((0,) + how.get("calls", (n,))), how.get("calls", (n,))):
                ref = None if "ctrl" not in how else np.linspace(0.0, 0.4, s.samples_for(m))[None]
                s.step(m, u=u[-1:, at:at + m], ctrl=how.get("ctrl"), theta_ref=ref)
        large_pairs = s.pair_count()
    (y0, x0, b0, f0, p0, off), (y1, x1, b1, f1, p1, _) = got
    assert f0 == f1 == 0
    assert p0 == p1 - large_pairs
    if y0 is not None:
        np.testing.assert_array_equal(y0, y1[:len(tanks)])
    np.testing.assert_array_equal(x0, x1[:off[-1]])
    np.testing.assert_array_equal(b0, b1[:len(tanks)])
