"""What lbm_kernel_shape reports is what runs, and setting it again changes nothing:
also for the kernel that small D2Q9 grids start in, which a context can be
given back after another one, and after lbm_autotune."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu

SMALL, LARGE = (100, 120, 1), (640, 520, 1)


def _sim(n, storage=lbm.LBM_FP32):
    D = 2 if n[2] == 1 else 3
    return lbm.from_workloads([W.random_small(3, D=D, n=n, periodic=(0, 0, 1) if D == 2 else (0, 0, 0), nparticles=2, rlo=3.0,
                                              rhi=4.0)], storage)


@gpu
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16])
@pytest.mark.parametrize("n,vec", [(SMALL, -1), (LARGE, 0), ((40, 36, 34), 0)])
def test_the_reported_shape_is_taken_back(n, vec, storage):
    a, b = _sim(n, storage), _sim(n, storage)
    assert a.kernel_shape()[0] == vec
    for sim in (a, b):
        sim.set_graphs(0)
        sim.step(5)
    first = b.kernel_shape()
    b.set_kernel_shape(*first)
    assert b.kernel_shape() == first
    b.set_kernel_shape(2, 4, 4)
    b.set_kernel_shape(*first)
    assert b.kernel_shape() == first
    b.autotune(1)
    tuned = b.kernel_shape()
    b.set_kernel_shape(*tuned)
    assert b.kernel_shape() == tuned
    for sim in (a, b):
        sim.step(6)
        sim.sync()
    assert np.array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()


@gpu
def test_the_way_back_to_the_direct_kernel():
    sim = _sim(SMALL)
    for ask in ((0, 8, 8), (-1, 4, 4), (4, 4, 4), (-1, 8, 4), (0, 4, 4)):
        sim.set_kernel_shape(*ask)
        assert sim.kernel_shape() == ask
    sim.close()


@gpu
@pytest.mark.parametrize("n,shape", [(SMALL, (-1, 2, 4)), (SMALL, (-2, 4, 4)), (SMALL, (-1, 4, 9)), ((40, 36, 34), (-1, 4, 4))])
def test_refused_shapes(n, shape):
    sim = _sim(n)
    before = sim.kernel_shape()
    with pytest.raises(lbm.LBMError):
        sim.set_kernel_shape(*shape)
    assert sim.kernel_shape() == before
    sim.close()


@gpu
@pytest.mark.parametrize("rows,warps", [(4, 1), (4, 4), (8, 4), (8, 8)])
def test_the_direct_kernel_on_a_large_grid(rows, warps):
    """It may be asked for on any D2Q9 grid, with the same bits."""
    a, b = _sim(LARGE), _sim(LARGE)
    b.set_kernel_shape(-1, rows, warps)
    for sim in (a, b):
        sim.step(18)
        sim.sync()
    assert np.array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()
