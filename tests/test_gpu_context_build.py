"""Building a context: particles added to any instance in any order, in one go or
in parts (the first insertion and the append take different copies), before and
after steps, give the run of a context that is built plainly; read back together
and one by one."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu


def _ws():
    return [W.many_disks(seed=s, nx=120 + 30 * s, ny=200, count=2 + s) for s in range(4)]


def _build(order, parts, extra_cap=0):
    ws = _ws()
    sim = lbm.LBM([lbm.config_from_workload(w, max_particles=w.num_particles + extra_cap) for w in ws])
    for i in order:
        w, n = ws[i], ws[i].num_particles
        cuts = [0, n] if parts == 1 else [0, 1, n]
        for a, b in zip(cuts, cuts[1:]):
            sim.add_particles(i, w.pos[a:b], w.radius[a:b], w.ratio[a:b])
    return sim


def _state(sim):
    out = []
    for i in range(4):
        out += [v for _, v in sorted(sim.particles(i).items())] + list(sim.fields(i))
    return out


@gpu
@pytest.mark.parametrize("order,parts,cap", [((0, 1, 2, 3), 1, 9), ((3, 1, 0, 2), 1, 0), ((2, 0, 3, 1), 2, 0), ((1, 3, 2, 0), 2, 70)])
def test_order_and_parts_do_not_matter(order, parts, cap):
    a, b = _build((0, 1, 2, 3), 1), _build(order, parts, cap)
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(x, y)
    for sim in (a, b):
        sim.step(37)
        sim.sync()
    for x, y in zip(_state(a), _state(b)):
        assert np.array_equal(x, y)
    a.close()
    b.close()


@gpu
def test_particles_added_after_steps_leave_the_others_running():
    ws = _ws()
    a = lbm.LBM([lbm.config_from_workload(w) for w in ws])
    for i in (0, 1, 3):
        a.add_particles(i, ws[i].pos, ws[i].radius, ws[i].ratio)
    a.step(17)
    a.add_particles(2, ws[2].pos, ws[2].radius, ws[2].ratio)
    a.step(20)
    a.sync()
    for i in (0, 1, 3):  # their run does not notice
        b = lbm.from_workloads([ws[i]])
        b.step(37)
        b.sync()
        for k, v in b.particles().items():
            assert np.array_equal(a.particles(i)[k], v), (i, k)
        b.close()
    b = lbm.from_workloads([ws[2]])  # the flow of instance 2 was still at rest
    b.step(20)
    b.sync()
    for k, v in b.particles().items():
        assert np.array_equal(a.particles(2)[k], v), k
    a.close()
    b.close()


@gpu
def test_repeated_adjoint_passes_of_other_lengths():
    """Checkpoints and slots are kept between passes, grow and are given back."""
    def grad(sim, n):
        sim.adjoint_forward(n)
        return sim.adjoint_backward([{"U": np.ones((w.num_particles, 2))} for w in ws])

    ws = _ws()
    sim = lbm.from_workloads(ws)
    blob = sim.save_state()
    for n in (5, 90, 4, 30):
        sim.load_state(blob)
        got = grad(sim, n)
        one = lbm.from_workloads(ws)
        want = grad(one, n)
        for g, t in zip(got, want):
            for k in t:
                x, y = np.asarray(g[k]), np.asarray(t[k])
                # the particle sums are FP64 atomics of FP32 warp sums: any order
                assert np.abs(x - y).max() <= 1e-9 * max(np.abs(y).max(), 1e-30), (n, k)
        one.close()
    sim.close()
