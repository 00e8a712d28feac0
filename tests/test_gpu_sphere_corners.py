"""Spheres whose centre lies near the far corner of its lattice cell: every node
that Eq. 9 gives them enters the sums of Eq. 22, also those farther than
ceil(R) + 1 from floor(X) in the y-z plane (up to R + sqrt(2)).  Against the
oracle, with the one-step bounds of the parity tests (equal counts, FP32 rounding of
the node velocities, 2e-6 of the largest particle velocity), and against
the allocation-free projection of the same spheres (equal counts)."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

from harness import compare_particles, make_pair, random_state

gpu = pytest.mark.gpu

SPHERES = [(8.0, (0.0, 0.99, 0.85)), (8.0, (0.5, 0.85, 0.99)), (6.0, (0.2, 0.97, 0.95)), (10.0, (0.3, 0.9, 0.95)),
           (24.5, (0.1, 0.93, 0.97)), (8.0, (0.99, 0.5, 0.5))]


def _nodes_beyond(R, off):
    """Nodes of the sphere beyond ceil(R) + 1 of floor(X) in the y-z plane."""
    g = np.arange(-int(R) - 3, int(R) + 4)
    x, y, z = np.meshgrid(g, g, g, indexing="ij")
    inside = (x - off[0]) ** 2 + (y - off[1]) ** 2 + (z - off[2]) ** 2 <= R * R
    return int((inside & (y * y + z * z > (np.ceil(R) + 1) ** 2)).sum())


def test_the_cases_have_such_nodes():
    assert sum(_nodes_beyond(R, off) > 0 for R, off in SPHERES) >= 3


@gpu
@pytest.mark.parametrize("shape", [None, (2, 4, 4)], ids=str)
@pytest.mark.parametrize("R,off", SPHERES)
def test_sums_of_a_sphere_near_a_cell_corner(R, off, shape):
    torch = pytest.importorskip("torch")
    m = int(2 * R) + 12
    n = (m, m + 1, m + 3)
    w = W.random_small(1, D=3, n=n, periodic=(0, 0, 0), nparticles=1, rlo=3.0, rhi=3.5, tau=0.9, g_grav=(0, 0, -1e-4))
    w.pos, w.radius, w.ratio = [[m // 2 + o for o in off]], [R], [1.3]
    sim, ref = make_pair(w, f0=random_state(3, 19, n[::-1]), shape=shape)
    u = torch.zeros(3 * sim.nodes(), device="cuda")
    sim.fields_device(0, u)
    sim.sync()
    sim.step(1)
    sim.sync()
    ref.step(1)
    cp = compare_particles(sim, ref)
    assert cp["count_equal"], cp
    assert cp["dU"] < 2e-6 * cp["Uscale"] and cp["dW"] < 2e-6 * cp["Uscale"] and cp["dX"] < 1e-8, cp
    pos, rad = (torch.tensor(v, dtype=torch.float64, device="cuda") for v in (w.pos, w.radius))
    vel, om = (torch.zeros(3, dtype=torch.float64, device="cuda") for _ in range(2))
    cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    fn = lbm.lib().lbm_rigid_projection_noalloc
    fn.restype = C.c_int
    p = lambda t: C.c_void_p(t.data_ptr())
    rc = fn(3, (C.c_int * 3)(*n), (C.c_int * 3)(0, 0, 0), p(u), 1, p(pos), p(rad), C.c_double(R), p(vel), p(om), p(cnt),
            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0
    part = sim.particles()
    assert int(cnt[0]) == int(part["count"][0])
    assert np.abs(vel.cpu().numpy() - part["U"][0]).max() < 2e-6 * cp["Uscale"]
    sim.close()
