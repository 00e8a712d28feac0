"""Collision forces far along a long axis (Eqs. 19-21): contacts at the edge of their
range, where the FP32 coordinates round a pair, or a particle and the far wall,
apart by more than a hundredth.  The same particles at the same distance from the far wall
of a short box give the same A after one step, up to the rounding of the predicted
positions: 2^-33 at 2^20, against a depth of the contact of 0.016, so 1e-7 of the force
(bound: 1e-6)."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu

R = 8.04
# offsets from n: the first touches the far wall, the other two each other
OFFSETS = [round(v * 2 ** 20) / 2 ** 20 for v in (-9.0315, -39.968, -57.0315)]


def test_the_contacts_are_in_range_and_fp32_rounds_them_apart():
    for n in (128, 1 << 20):
        x = [n + o for o in OFFSETS]
        assert 0 < R + 0.5 - (n - 0.5 - x[0]) < 0.01
        assert 0 < 2 * R + 1 - (x[1] - x[2]) < 0.02
    f = [np.float32((1 << 20) + o) for o in OFFSETS]
    assert np.float32(1 << 20) - np.float32(0.5) - f[0] > R + 0.5 + 0.01
    assert f[1] - f[2] > 2 * R + 1 + 0.01


@gpu
@pytest.mark.parametrize("K", [1, 2])
def test_a_far_contact_acts_like_a_near_one(K):
    A = []
    for n in (128, 1 << 20):
        w = W.random_small(1, D=2, n=(n, 40, 1), periodic=(0, 0, 1), nparticles=1, rlo=3.0, rhi=3.5, tau=0.9, g_grav=(0, -1e-4, 0))
        w.pos, w.radius, w.ratio, w.K = [[n + o, 19.5] for o in OFFSETS], [R] * 3, [1.5, 1.3, 1.4], K
        sim = lbm.from_workloads([w])
        sim.step(1)
        sim.sync()
        A.append(sim.particles()["A"][:, 0])
        sim.close()
    near, far = A
    assert np.all(near != 0)
    assert np.abs(far - near).max() <= 1e-6 * np.abs(near).min()


@gpu
def test_gradient_of_a_far_wall_contact():
    """The adjoint's own pre-test: dJ / dX of J = X after one step."""
    g = []
    for n in (128, 1 << 20):
        w = W.random_small(1, D=2, n=(n, 40, 1), periodic=(0, 0, 1), nparticles=1, rlo=3.0, rhi=3.5, tau=0.9, g_grav=(0, -1e-4, 0))
        w.pos, w.radius, w.ratio = [[n + OFFSETS[0], 19.5]], [R], [1.5]
        sim = lbm.from_workloads([w])
        sim.adjoint_forward(1)
        r = sim.adjoint_backward([{"A": [[1.0, 0.0]]}])[0]
        g.append(r["ratio"][0])
        sim.close()
    assert g[0] != 0 and abs(g[1] - g[0]) <= 1e-6 * abs(g[0])
