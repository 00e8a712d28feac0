"""The default fluid kernels (D2Q9 staged, D3Q19 direct) at the edges of their
row segments and tiles against the register path, bit for bit: rows that end
inside, at and after a 64-node segment, tiles that hold both x faces, rows at
walls and at periodic faces, with and without a body force (the collision
without forcing terms), at tau = 1 and not.  Every operation of the step is
written out (no contraction freedom), so the two paths give the same bits."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

from harness import random_state

gpu = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu_setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    lbm.build()
    yield


def _run(w, storage, f0, shape, steps):
    sim = lbm.from_workloads([w], storage)
    if shape:
        sim.set_kernel_shape(*shape)
    sim.set_populations(f0)
    sim.step(steps)
    sim.sync()
    out = [sim.get_populations(), *sim.fields()] + [v for _, v in sorted(sim.particles().items())]
    sim.close()
    return out


CASES = [(2, (n, 23, 1)) for n in (20, 63, 64, 65, 66, 100, 127, 128, 129, 130, 193, 257)] + \
        [(2, (70, n, 1)) for n in (16, 17, 24)] + \
        [(3, (n, 17, 18)) for n in (18, 31, 63, 64, 65, 66, 129)] + [(3, (33, 16, 19))]


@gpu
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16])
@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("D,n", CASES)
def test_default_path_matches_register_path(D, n, periodic, storage):
    odd = n[0] % 2
    per = ((periodic, 0, 1) if odd else (0, periodic, 1)) if D == 2 else ((periodic, 0, 0) if odd else (0, periodic, periodic))
    w = W.random_small(n[0] + n[1], D=D, n=n, periodic=per, nparticles=2, rlo=2.1, rhi=3.7, tau=1.0 if n[1] % 2 else 0.8,
                       g_grav=(0, -1e-4, 0) if D == 2 else (0, 0, -1e-4), g_drive=(0, 0, 0) if odd else (1e-5, 0, 0))
    f0 = random_state(n[0], 9 if D == 2 else 19, n[::-1] if D == 3 else (n[1], n[0]))
    a = _run(w, storage, f0, None, 5)
    b = _run(w, storage, f0, (1 if storage == lbm.LBM_FP32 else 2, 4, 4), 5)
    for x, y in zip(a, b):
        assert np.array_equal(x, y)
