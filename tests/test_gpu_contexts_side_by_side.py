"""Contexts that are alive together run as if each were alone: the shared memory
that the staged kernel may take is a property of the kernel and not of a context, so
a context with few instances, created later, must leave the launches of one
with many (a larger table in shared memory) and its recomputation valid."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu


def _many(storage):
    ws = [W.random_small(s, n=(64 + s % 7, 80, 1), periodic=(0, 0, 1), nparticles=1, rlo=3.0, rhi=5.0) for s in range(64)]
    return lbm.from_workloads(ws, storage)  # 64 boxes of 2^12.3 nodes: the staged kernel


def _run(sim, graphs):
    sim.set_graphs(graphs)
    sim.step(35)
    sim.sync()
    return [sim.get_populations(i) for i in (0, 63)]


@gpu
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16])
@pytest.mark.parametrize("graphs", [0, 16])
def test_a_smaller_context_leaves_a_larger_one_running(graphs, storage):
    one = W.random_small(5, n=(640, 520, 1), periodic=(0, 0, 1), nparticles=2, rlo=3.0, rhi=5.0)
    alone = _many(storage)
    want = _run(alone, graphs)
    alone.close()
    many = _many(storage)
    later = lbm.from_workloads([one], storage)
    later.step(3)
    for a, b in zip(want, _run(many, graphs)):
        assert np.array_equal(a, b)
    many.adjoint_forward(6, 3)
    many.adjoint_backward([{"X": np.ones((1, 2))}] * 64)
    many.sync()
    later.close()
    many.close()
