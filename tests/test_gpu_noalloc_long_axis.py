"""The allocation-free projection on wall axes so long that FP32 no longer
resolves a lattice unit: of two overlapping particles the lower index owns the
shared nodes there too.  The counts are those of Eq. 9 by integers and FP64 on the
host; the field is constant, so U is that constant (within the rounding of the
fixed-point sums, 2^-41 per component)."""
import ctypes as C

import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm

gpu = pytest.mark.gpu


def _owned(n, pos, radius):
    """Nodes owned by each disk (lowest index first)."""
    taken, counts = set(), []
    for (px, py), r in zip(pos, radius):
        mine = {(x, y) for x in range(max(int(px - r) - 1, 0), min(int(px + r) + 2, n[0]))
                for y in range(n[1]) if (x - px) ** 2 + (y - py) ** 2 <= r * r} - taken
        taken |= mine
        counts.append(len(mine))
    return counts


@gpu
@pytest.mark.parametrize("x0", [1000.0, 1048560.0, 9.0e6, 20000001.0, 40000001.99], ids=str)
def test_overlap_far_along_a_wall_axis(x0):
    torch = pytest.importorskip("torch")
    R = 4.25
    pos = [(x0, 1.2), (x0 + 8.11, 1.1), (x0 + 40.0, 0.6)]  # the first two share a column of nodes
    n = (int(x0) + 60, 3)
    want = _owned(n, pos, [R] * 3)
    u = torch.empty((2, n[1], n[0]), dtype=torch.float32, device="cuda")
    u[0], u[1] = 0.01, -0.02
    dev = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")
    p, r = dev(pos), dev([R] * 3)
    vel, om = torch.zeros((3, 2), dtype=torch.float64, device="cuda"), dev([0.0] * 3)
    cnt = torch.zeros(3, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    fn = lbm.lib().lbm_rigid_projection_noalloc
    fn.restype = C.c_int
    q = lambda t: C.c_void_p(t.data_ptr())
    rc = fn(2, (C.c_int * 3)(*n, 1), (C.c_int * 3)(0, 0, 1), q(u), 3, q(p), q(r), C.c_double(R), q(vel), q(om), q(cnt),
            C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, lbm.STATUS.get(rc, rc)
    assert cnt.tolist() == want
    exact = np.float32([0.01, -0.02]).astype(np.float64)
    assert np.abs(vel.cpu().numpy() - exact).max() <= 2.0 ** -40


def test_the_disks_share_a_node():
    pos = [(40000001.99, 1.2), (40000010.1, 1.1)]
    assert _owned((40000061, 3), pos, [4.25] * 2)[1] < _owned((40000061, 3), pos[1:], [4.25])[0]
