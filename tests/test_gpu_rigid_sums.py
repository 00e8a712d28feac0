"""The sums of Eq. 22 that the fluid kernels add up and the particle kernel
that finishes them: radii on both sides of the narrow sums (R < 30), particles
that share rows, overlap, wrap around a periodic axis or touch, several
sub-steps, one or many particles per instance and several instances.  Against
the FP64 oracle with the one-step bounds of the parity tests (FP32 rounding of
the node velocities, 2e-6 of the largest particle velocity), and bit for bit
between contexts of one and several instances (integer sums have no order)."""
import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

from harness import compare_fields, compare_particles, make_pair, random_state

gpu = pytest.mark.gpu


def test_split_of_a_velocity_is_its_fixed_point_integer():
    """hi 2^20 + lo of the device's split (adding 1.5 2^23 in FP32 rounds to the
    nearest integer) equals round-half-even(u 2^40), ties and limits included."""
    rng = np.random.default_rng(0)
    f = np.float32
    u = np.concatenate([rng.uniform(-0.5, 0.5, 400000), rng.uniform(-1, 1, 400000) * 2.0 ** rng.integers(-45, -1, 400000),
                        (np.arange(-4096, 4096) + 0.5) * 2.0 ** -40, (np.arange(-4096, 4096) + 0.5) * 2.0 ** -20,
                        [0.0, -0.0, 0.49999997, -0.49999997, 2.0 ** -41, -2.0 ** -41]]).astype(f)
    u = np.clip(u, f(-0.49999997), f(0.49999997))
    magic = f(12582912.0)
    v = u * f(1048576.0)
    r = v + magic
    rem = v - (r - magic)
    low = rem * f(1048576.0) + magic  # the product is exact
    hi = r.view(np.int32).astype(np.int64) - 0x4B400000
    lo = low.view(np.int32).astype(np.int64) - 0x4B400000
    assert np.abs(hi).max() <= 1 << 19 and np.abs(lo).max() <= 1 << 19
    assert np.array_equal(hi * (1 << 20) + lo, np.rint(u.astype(np.float64) * 2.0 ** 40).astype(np.int64))


def _workload(D, n, per, pos, radius, K=1):
    w = W.random_small(1, D=D, n=n, periodic=per, nparticles=1, rlo=3.0, rhi=3.5, tau=0.9,
                       g_grav=(0, -1e-4, 0) if D == 2 else (0, 0, -1e-4))
    w.pos, w.radius, w.ratio = [list(p) for p in pos], list(radius), [1.2 + 0.1 * k for k in range(len(radius))]
    w.K = K
    return w


CASES = {
    "radius 28.9": (2, (90, 80, 1), (0, 0, 1), [(40.3, 38.7)], [28.9]),
    "radius 29.9 and 30.1": (2, (140, 75, 1), (0, 0, 1), [(33.2, 36.1), (101.6, 37.9)], [29.9, 30.1]),
    "radius 62": (2, (150, 140, 1), (0, 0, 1), [(71.9, 68.4)], [62.0]),
    "one row": (2, (200, 40, 1), (0, 0, 1), [(12.0 + 17.3 * k, 19.5 + 0.3 * k) for k in range(10)], [8.2] * 10),
    "overlap": (2, (66, 48, 1), (0, 0, 1), [(30.1, 22.2), (33.7, 24.9), (30.4, 27.3)], [7.0, 6.0, 8.5]),
    "wrapped": (2, (65, 67, 1), (1, 1, 1), [(0.3, 66.8), (64.6, 30.2)], [9.0, 6.5]),
    "touching, K = 3": (2, (80, 60, 1), (0, 0, 1), [(30.0, 30.0), (46.6, 30.4), (38.2, 44.9)], [8.0, 8.0, 8.2], 3),
    "spheres": (3, (40, 36, 38), (0, 1, 0), [(14.2, 35.7, 15.1), (26.9, 14.4, 22.3)], [7.0, 6.2]),
    "a large sphere": (3, (66, 66, 64), (0, 0, 0), [(32.3, 31.9, 30.2)], [24.5]),
}


@gpu
@pytest.mark.parametrize("shape", [None, (1, 4, 4), (4, 4, 2), (0, 8, 4)], ids=str)
@pytest.mark.parametrize("case", CASES)
def test_particle_sums_match_oracle(case, shape):
    D, n, per, pos, radius, *K = CASES[case]
    w = _workload(D, n, per, pos, radius, *K)
    f0 = random_state(5, 9 if D == 2 else 19, n[::-1] if D == 3 else (n[1], n[0]))
    sim, ref = make_pair(w, f0=f0, shape=shape)
    for steps in (1, 7):
        sim.step(steps)
        sim.sync()
        ref.step(steps)
        if steps > 1:
            continue  # the rounding of several steps: only the solid domains are compared below
        cp = compare_particles(sim, ref)
        assert cp["count_equal"], cp
        assert cp["dU"] < 2e-6 * cp["Uscale"], cp
        assert cp["dW"] < 2e-6 * cp["Uscale"], cp
        assert cp["dX"] < 1e-8, cp
    assert compare_fields(sim, ref)["owner_equal"]
    sim.close()


@gpu
def test_instances_of_a_batch_match_single_contexts():
    ws = [_workload(*CASES[k][:5]) for k in ("radius 28.9", "one row", "radius 62", "overlap", "wrapped")]
    both = lbm.from_workloads(ws)
    both.step(40)
    both.sync()
    for i, w in enumerate(ws):
        one = lbm.from_workloads([w])
        one.step(40)
        one.sync()
        a, b = both.particles(i), one.particles()
        for k in a:
            assert np.array_equal(a[k], b[k]), (i, k)
        one.close()
    both.close()


@gpu
def test_backward_pass_leaves_the_trajectory():
    """The adjoint's recomputation keeps totals and step inputs of its own: the
    context continues as if only the forward pass had run."""
    w = _workload(*CASES["one row"][:5])
    a, b = lbm.from_workloads([w]), lbm.from_workloads([w])
    a.adjoint_forward(21, 4)
    a.adjoint_backward([{"X": np.ones((10, 2))}])
    b.step(21)
    for sim in (a, b):
        sim.step(19)
        sim.sync()
    pa, pb = a.particles(), b.particles()
    for k in pa:
        assert np.array_equal(pa[k], pb[k]), k
    assert np.array_equal(a.get_populations(), b.get_populations())
    a.close()
    b.close()
