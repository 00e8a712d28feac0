"""D2Q9 grids of up to 2^18 nodes take the kernel that loads straight into
registers, larger ones the staged kernel: the two give the same bits on every
form of a grid (segment and tile edges, walls, periodic faces, both storage
types), on both sides of the line, in batches, and in graph replay."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

from harness import random_state
from test_gpu_fluid_edges import CASES, _run

gpu = pytest.mark.gpu


@gpu
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16])
@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("n", [n for D, n in CASES if D == 2] + [(2, 2, 1), (3, 9, 1)])
def test_staged_kernel_matches_the_default(n, periodic, storage):
    w = W.random_small(n[0] + n[1], D=2, n=n, periodic=(periodic, 0, 1) if n[0] % 2 else (0, periodic, 1),
                       nparticles=2 if n[0] >= 16 else 0, rlo=2.1, rhi=3.7, tau=1.0 if n[1] % 2 else 0.8,
                       g_grav=(0, -1e-4, 0), g_drive=(0, 0, 0) if n[0] % 2 else (1e-5, 0, 0))
    f0 = random_state(n[0], 9, (n[1], n[0]))
    a = _run(w, storage, f0, None, 18)
    for shape in ((0, 8, 8), (0, 4, 4)):
        for x, y in zip(a, _run(w, storage, f0, shape, 18)):
            assert np.array_equal(x, y), shape


@gpu
@pytest.mark.parametrize("ny", [512, 513])
def test_both_sides_of_the_line(ny):
    w = W.many_disks(seed=3, nx=512, ny=ny, count=20)
    f0 = random_state(4, 9, (ny, 512))
    a = _run(w, lbm.LBM_FP32, f0, None, 20)
    for shape in ((0, 8, 8), (2, 4, 4)):
        for x, y in zip(a, _run(w, lbm.LBM_FP32, f0, shape, 20)):
            assert np.array_equal(x, y), shape


@gpu
def test_batch_of_small_grids_matches_single_contexts():
    ws = [W.random_small(s, n=(40 + 17 * s, 50, 1), periodic=(1, 0, 1), nparticles=1 + s, rlo=3.0, rhi=5.0) for s in range(4)]
    both = lbm.from_workloads(ws)
    both.step(33)
    both.sync()
    for i, w in enumerate(ws):
        one = lbm.from_workloads([w])
        one.step(33)
        one.sync()
        for x, y in zip(both.fields(i), one.fields()):
            assert np.array_equal(x, y), i
        one.close()
    both.close()
