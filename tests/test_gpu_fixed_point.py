"""The device's fixed-point image of a node velocity (split_fx, to_fx32: round-half-even
of u 2^40, |u| < 1/2) and the exact sums of Eq. 22 over it, from velocities that are
known to the bit: ties, limits and 24-bit values.  A velocity reaches a fluid kernel
exactly through a state whose only nonzero populations move along the axes, one per
axis, with the particle accelerations zero (no gravity, A = 0): u_d(x) = f_d(x - c_d).
U = (sum of integers) 2^-40 / n; one unit in one node's integer would show as 2^-40 / n,
and the bound is a thousandth of that, plus the roundings of the division (below 1e-15
of U)."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu

F = np.float32


def _values(rng, shape):
    """FP32 velocity components, |u| < 0.28: random, ties of the low and of the high half, tiny."""
    n = int(np.prod(shape))
    v = np.concatenate([rng.uniform(-0.28, 0.28, n), rng.uniform(-1, 1, n) * 2.0 ** rng.integers(-42, -3, n),
                        (rng.integers(-4096, 4096, n) + 0.5) * 2.0 ** -40, (rng.integers(-65536, 65536, n) + 0.5) * 2.0 ** -20,
                        rng.integers(-1 << 18, 1 << 18, n) * 2.0 ** -20 + 2.0 ** -41]).astype(F)
    return rng.choice(v, n).reshape(shape)


def _integer(u):
    return np.rint(u.astype(np.float64) * 2.0 ** 40).astype(np.int64)


def _sums(w, u):
    """(count, U by exact integers) of the first particle; u [D, ...] indexed [.., z, y, x]."""
    g = np.meshgrid(*[np.arange(k) for k in (w.n if w.D == 3 else w.n[:2])][::-1], indexing="ij")
    d2 = sum((c - p) ** 2 for c, p in zip(g[::-1], w.pos[0]))
    inside = d2 <= w.radius[0] ** 2
    cnt = int(inside.sum())
    return cnt, np.array([int(_integer(u[d])[inside].sum()) for d in range(w.D)], dtype=object), inside


def _case(D, n, pos, R):
    w = W.random_small(1, D=D, n=n, periodic=(1, 1, 1), nparticles=1, rlo=3.0, rhi=3.5, tau=0.9, g_grav=(0, 0, 0),
                       g_drive=(0, 0, 0))
    w.pos, w.radius, w.ratio = [list(pos)], [R], [1.5]
    return w


CASES = [(2, (70, 66, 1), (30.3, 31.8), 12.4), (2, (171, 166, 1), (84.9, 83.2), 40.3), (3, (41, 40, 43), (19.4, 20.1, 21.9), 9.7)]


@gpu
@pytest.mark.parametrize("shape", [None, (0, 8, 8), (0, 4, 4), (1, 4, 4), (4, 4, 2)], ids=str)
@pytest.mark.parametrize("D,n,pos,R", CASES)
def test_sums_of_known_velocities(D, n, pos, R, shape):
    w = _case(D, n, pos, R)
    dims = n[::-1] if D == 3 else (n[1], n[0])
    rng = np.random.default_rng(D * 100 + n[0])
    u = np.stack([_values(rng, dims) for _ in range(D)])
    f = np.zeros((9 if D == 2 else 19,) + tuple(dims), F)
    heads = (1, 2) if D == 2 else (1, 3, 5)  # the velocities +x, +y(, +z)
    for d, q in enumerate(heads):
        f[q] = np.roll(u[d], -1, axis=D - 1 - d)  # population q moves one node along axis d
    sim = lbm.from_workloads([w])
    if shape:
        sim.set_kernel_shape(*shape)
    sim.set_graphs(0)
    sim.set_populations(f)
    field, _, _ = sim.fields()
    assert np.array_equal(np.moveaxis(field, -1, 0), u)  # the velocities are what they are meant to be
    sim.step(1)
    part = sim.particles()
    cnt, S, _ = _sums(w, u)
    assert int(part["count"][0]) == cnt
    for d in range(D):
        assert abs(part["U"][0, d] - float(S[d]) * 2.0 ** -40 / cnt) <= 1e-3 * 2.0 ** -40 / cnt + 1e-15 * abs(part["U"][0, d])
    sim.close()


@gpu
@pytest.mark.parametrize("D,n,pos,R", CASES)
def test_projection_of_known_velocities(D, n, pos, R):
    torch = pytest.importorskip("torch")
    w = _case(D, n, pos, R)
    dims = n[::-1] if D == 3 else (n[1], n[0])
    u = np.stack([_values(np.random.default_rng(D), dims) for _ in range(D)])
    cnt, S, _ = _sums(w, u)
    dev = lambda a, t: torch.tensor(np.asarray(a), dtype=t, device="cuda")
    ut, p, r = dev(u, torch.float32), dev(w.pos, torch.float64), dev(w.radius, torch.float64)
    vel, om, c = dev(np.zeros(3), torch.float64), dev(np.zeros(3), torch.float64), dev([0], torch.int32)
    torch.cuda.synchronize()
    fn = lbm.lib().lbm_rigid_projection_noalloc
    fn.restype = C.c_int
    q = lambda t: C.c_void_p(t.data_ptr())
    rc = fn(D, (C.c_int * 3)(*n), (C.c_int * 3)(1, 1, 1), q(ut), 1, q(p), q(r), C.c_double(R), q(vel), q(om), q(c),
            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lbm.STATUS.get(rc, rc)
    assert int(c[0]) == cnt
    for d in range(D):
        U = float(vel[d])
        assert abs(U - float(S[d]) * 2.0 ** -40 / cnt) <= 1e-3 * 2.0 ** -40 / cnt + 1e-15 * abs(U)
