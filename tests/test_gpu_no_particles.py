"""Contexts without particles: every kernel of a run is a fluid kernel, and the
next step's may be resident while the one before still writes the populations
that it reads.  Many steps give the bits of the register path (whose launches
do not overlap), replayed from graphs and launched one by one, in 2D below and above
2^18 nodes and in 3D."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

from harness import random_state

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16])
@pytest.mark.parametrize("D,n,periodic", [(2, (100, 70, 1), (1, 0, 1)), (2, (601, 530, 1), (0, 0, 1)),
                                          (2, (640, 513, 1), (1, 1, 1)), (3, (70, 40, 38), (0, 0, 0)),
                                          (3, (131, 67, 34), (1, 0, 1))])
def test_many_steps_without_particles(D, n, periodic, storage):
    w = W.random_small(1, D=D, n=n, periodic=periodic, nparticles=0, tau=0.9, g_drive=(1e-5, 0, 0))
    f0 = random_state(2, 9 if D == 2 else 19, n[::-1] if D == 3 else (n[1], n[0]))
    out = []
    for shape, graphs in ((None, 16), (None, 0), ((2, 4, 4), 0)):
        sim = lbm.from_workloads([w], storage)
        if shape:
            sim.set_kernel_shape(*shape)
        sim.set_graphs(graphs)
        sim.set_populations(f0)
        sim.step(209)
        sim.sync()
        out.append(sim.get_populations())
        sim.close()
    assert np.abs(out[0]).max() > 0
    assert np.array_equal(out[0], out[2])
    assert np.array_equal(out[1], out[2])
