"""The fields kernel and the allocation-free projection at the edges of their
work splits: rows that end inside, at and after a 32-node chunk and a warp's
segment, chunks that touch an x face, and projections whose boxes fit one
block's slice, just exceed it, or mix both.

Tolerances: u sums Q - 1 populations of at most 1e-3 in FP32 and u itself is
of that size, so (Q - 1)^2 2^-24 < 2e-5 / 4 bounds the relative error of the
largest entry (5e-6); the projection's exact sums round each u to 2^-41
(1e-9 relative with the FP64 second pass)."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

import oracle
from harness import compare_fields, make_pair, oracle_config, random_state

gpu = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu_setup():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    lbm.build()
    yield


@gpu
@pytest.mark.parametrize("storage", [lbm.LBM_FP32, lbm.LBM_FP16])
@pytest.mark.parametrize("D,n,periodic", [
    (2, (31, 20, 1), (0, 0, 1)), (2, (32, 21, 1), (1, 0, 1)), (2, (33, 20, 1), (0, 1, 1)), (2, (65, 24, 1), (1, 1, 1)),
    (2, (128, 20, 1), (0, 0, 1)), (2, (129, 20, 1), (1, 0, 1)), (2, (257, 19, 1), (0, 0, 1)),
    (3, (31, 18, 17), (0, 0, 0)), (3, (33, 17, 18), (1, 0, 1)), (3, (65, 18, 19), (0, 1, 0)), (3, (97, 17, 17), (1, 1, 1))])
def test_fields_at_chunk_edges(D, n, periodic, storage):
    w = W.random_small(n[0], D=D, n=n, periodic=periodic, nparticles=2, rlo=2.2, rhi=3.9,
                       g_grav=(0, -1e-4, 0) if D == 2 else (0, 0, -1e-4), g_drive=(1e-5, 0, 0))
    f0 = random_state(n[0], 9 if D == 2 else 19, n[::-1] if D == 3 else (n[1], n[0]))
    if storage == lbm.LBM_FP16:  # values the storage holds exactly
        f0 = (f0 * 16384.0).astype(np.float16).astype(np.float32) / 16384.0
    sim, ref = make_pair(w, storage=storage, f0=f0)
    c = compare_fields(sim, ref)
    sim.close()
    assert c["owner_equal"], c
    assert c["du"] <= 5e-6 and c["dp"] <= 5e-6, c


@gpu
@pytest.mark.parametrize("D,radii", [(2, [4.0, 29.9]), (2, [30.6, 3.0]), (2, [61.0]), (3, [6.0, 2.5]), (3, [6.2, 3.0]),
                                     (3, [15.3])])
@pytest.mark.parametrize("periodic", [0, 1])
def test_projection_at_slice_edges(D, radii, periodic):
    import torch

    from test_zz_no_alloc import _entry

    n = (161, 147, 1) if D == 2 else (53, 47, 61)
    rng = np.random.default_rng(len(radii) + D)
    pos = np.array([[rng.uniform(0.45, 0.55) * n[d] for d in range(D)] for _ in radii])  # they overlap
    if periodic:
        pos[0, 0] = 1.3  # across the x face
    w = W.Workload("slices", D, n, (periodic, 0, 1 if D == 2 else 0), 1.0, 1.0, pos=pos.tolist(), radius=radii,
                   ratio=[1.5] * len(radii))
    u = rng.uniform(-0.1, 0.1, (D,) + n[::-1]).astype(np.float32)
    ref = oracle.Sim(oracle_config(w))
    ref.add_particles(w.pos, w.radius, w.ratio)
    U, Wr, cnt = ref.rigid_projection(np.moveaxis(u.astype(np.float64), 0, -1).reshape(ref.shape + (D,)))
    ref.close()
    k, dev = len(radii), "cuda"
    f64 = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)
    ud, X, R = torch.tensor(u, device=dev), f64(pos), f64(radii)
    vel, om = f64(np.full((k, D), np.nan)), f64(np.full((k, 1 if D == 2 else 3), np.nan))
    c = torch.full((k,), -1, dtype=torch.int32, device=dev)
    torch.cuda.synchronize()
    p = lambda t: C.c_void_p(t.data_ptr())
    rc = _entry()(D, (C.c_int * 3)(*n), (C.c_int * 3)(*w.periodic), p(ud), k, p(X), p(R), max(radii), p(vel), p(om), p(c),
                  None)
    own = np.asarray(cnt) > 0  # a particle covered by one of lower index owns nothing: reported
    assert rc == (0 if own.all() else -8), lbm.STATUS.get(rc, rc)
    assert np.array_equal(c.cpu().numpy(), cnt)
    Wref = Wr[:, 2:3] if D == 2 else Wr
    vel, om = vel.cpu().numpy(), om.cpu().numpy()
    assert np.all(vel[~own] == 0.0) and np.all(om[~own] == 0.0)
    vel, om, U, Wref = vel[own], om[own], U[own, :D], Wref[own]  # (the oracle has no value for the others)
    assert np.abs(vel - U).max() <= 1e-9 * np.abs(U).max() + 1e-12
    assert np.abs(om - Wref).max() <= 1e-9 * np.abs(Wref).max() + 1e-12
