"""The first particles of an instance: the cost goes with the particles added, not
with the room the instance has, and the run does not depend on that room."""
import time

import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu


def _sim(w, cap):
    return lbm.LBM([lbm.config_from_workload(w, max_particles=cap)])


@gpu
@pytest.mark.parametrize("cap", [3, 6, 7, 600, 900, 5000, 1 << 20])
def test_the_room_does_not_matter(cap):
    w = W.many_disks(seed=2, nx=120, ny=200, count=3)
    a, b = _sim(w, 3), _sim(w, cap)
    for sim in (a, b):
        sim.add_particles(0, w.pos, w.radius, w.ratio, vel=[[1e-3, -2e-3]] * 3, omega=[1e-4] * 3)
        sim.step(25)
        sim.sync()
    for (k, x), y in zip(a.particles().items(), b.particles().values()):
        assert np.array_equal(x, y), k
    assert np.array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()


@gpu
def test_one_particle_in_a_large_instance_is_quick():
    """At most 20 times the time with room for 64 (it was some hundred times: the
    image of 2^20 slots); the quickest of four each."""
    w = W.many_disks(seed=2, nx=120, ny=200, count=1)
    took = {}
    for cap in (64, 1 << 20):
        for _ in range(4):
            sim = _sim(w, cap)
            sim.sync()
            t = time.perf_counter()
            sim.add_particles(0, w.pos, w.radius, w.ratio)
            sim.sync()
            took[cap] = min(took.get(cap, 1e9), time.perf_counter() - t)
            sim.close()
    assert took[1 << 20] < 20 * took[64]
