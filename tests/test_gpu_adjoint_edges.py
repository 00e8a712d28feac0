"""The adjoint fluid kernel at the edges of its 64-node segments and tiles,
against the FP64 autograd of the oracle's step (oracle/twin.py) at the bound of
the adjoint tests (1e-4 of the largest entry of each gradient): rows that end
inside, at and after a segment, walls and periodic faces, a body force (the
general collision on every node), tau = 1 and not, one tile or several per row."""
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


def _grad(w, f0, shape, seed):
    sim = lbm.from_workloads([w])
    if shape:
        sim.set_kernel_shape(*shape)
    sim.set_populations(f0)
    sim.adjoint_forward(3, 2)
    rng = np.random.default_rng(seed)
    n = w.num_particles
    gp = {"X": rng.normal(size=(n, w.D)), "U": rng.normal(size=(n, w.D)) * 10}
    gf = rng.normal(size=f0.shape).astype(np.float32)
    gf[0] = 0
    import torch
    res, field = sim.adjoint_backward([gp], seed_field=torch.from_numpy(gf).cuda(), want_field=True)
    sim.close()
    return res[0], field.cpu().numpy().reshape(f0.shape), gp, gf


CASES = [(2, (n, 11, 1)) for n in (20, 63, 64, 65, 127, 129, 130)] + [(2, (40, 17, 1)), (3, (33, 16, 18)), (3, (65, 17, 16))]


@gpu
@pytest.mark.parametrize("periodic", [0, 1])
@pytest.mark.parametrize("D,n", CASES)
def test_shapes_agree_and_match_the_derivative(D, n, periodic):
    """Staged and register tile shapes (other segment splits) give the same
    gradients to the order of the particle sums (1e-6 of the largest entry: FP32
    sums of fewer than 2^11 terms in another order), and the field gradient
    matches a central difference of the FP64 oracle along itself (a direction that
    weighs every node, so a wrong edge column or row shows)."""
    import oracle
    from harness import oracle_config
    per = (periodic, 0, 1) if D == 2 else (0, periodic, 0)
    drive = (0, 0, 0) if n[0] % 2 else (1e-5, 0, 0)
    w = W.random_small(n[0], D=D, n=n, periodic=per, nparticles=1, rlo=2.1, rhi=3.4, tau=1.0 if n[0] % 4 < 2 else 0.8,
                       g_grav=(0, -1e-4, 0) if D == 2 else (0, 0, -1e-4), g_drive=drive)
    f0 = random_state(n[0], 9 if D == 2 else 19, n[::-1] if D == 3 else (n[1], n[0]))
    ra, fa, gp, gf = _grad(w, f0, None, 3)
    rb, fb, _, _ = _grad(w, f0, (1, 4, 4), 3)
    assert np.abs(fa - fb).max() <= 1e-6 * np.abs(fa).max()
    for k in ("alpha", "ratio", "X", "U"):
        a, b = np.asarray(ra[k]), np.asarray(rb[k])
        assert np.abs(a - b).max() <= 1e-6 * max(np.abs(a).max(), 1e-30), k
    d = fa.astype(np.float64) * (1e-3 / np.abs(fa).max())
    J = []
    h = 1e-3
    for s in (1, -1):
        ref = oracle.Sim(oracle_config(w))
        ref.set_f(f0.astype(np.float64) + s * h * d)
        ref.add_particles(w.pos, w.radius, w.ratio)
        ref.step(3)
        p = ref.particles()
        J.append((gp["X"] * p["X"][:, :D]).sum() + (gp["U"] * p["U"][:, :D]).sum() + (gf.astype(np.float64)[1:] * ref.get_f()[1:]).sum())
        ref.close()
    fd = (J[0] - J[1]) / (2 * h)
    want = (fa.astype(np.float64) * d).sum()
    assert abs(want - fd) < 1e-4 * want
