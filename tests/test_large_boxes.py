"""D3Q19 boxes whose population buffer holds more than 2^31 elements: lbm_create
bounds the nodes (n0 n1 n2 19 <= 2e9), but rows are padded to 32 nodes, so the
buffer's 18 populations can exceed 32-bit offsets.

On the CPU the kernels' own address arithmetic (pull_source, pop) is compiled
for the host and compared with Python integers at the corners of such boxes.  On
the GPU a box that is periodic along z with period 8 has to give the bits of
the 8-layer box it repeats: stepped, read as fields and differentiated."""
import ctypes as C
import itertools
import os
import subprocess

import numpy as np
import pytest

from paper_2511_01629_gb300 import lbm
from paper_2511_01629_gb300 import workloads as W

gpu = pytest.mark.gpu

# just below the line, where the whole buffer has 32-bit offsets
NARROW = [(64, 1300, 1260), (100, 965, 965), (33, 1366, 1364), (2, 1931, 1930)]
BOXES = [(100, 1000, 1000), (65, 1200, 1300), (129, 900, 900), (33, 1785, 1785), (2, 7200, 7200), (5, 200, 100000)]

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "lbm_common.cuh"
using namespace lbmpen;
template <int q> void offsets(const InstDesc& in, int x, int y, int z) {
    if constexpr (q < 19) {
        const PullSrc s = pull_source<19, q>(in, x, y, z);
        const char* f = reinterpret_cast<const char*>(uintptr_t{1} << 40);  // never dereferenced
        const int src = s.axis >= 0 ? Lat<19>::opp(q) : q;
        const char* from = pop(f, src, in.qstride) + s.off;
        if (elem(f, src, in.qstride, s.off) != from) exit(1);
        if (!wide_offsets(19, in.qstride) && elem(f, src, (int)in.qstride, s.off) != from) exit(2);
        printf("%lld %d %d\n", (long long)(from - f), s.axis, s.face);
        offsets<q + 1>(in, x, y, z);
    }
}
int main(int argc, char** argv) {
    InstDesc in{};
    for (int d = 0; d < 3; ++d) {
        in.n[d] = atoi(argv[1 + d]);
        in.periodic[d] = atoi(argv[4 + d]);
    }
    in.pitch = (in.n[0] + 31) & ~31;
    in.qstride = (long long)in.pitch * in.n[1] * in.n[2];
    int x, y, z;
    while (scanf("%d %d %d", &x, &y, &z) == 3) offsets<1>(in, x, y, z);
}
"""

C19 = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
       (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("offsets")
    src, exe = d / "offsets.cu", d / "offsets"
    src.write_text(PROGRAM)
    csrc = os.path.join(os.path.dirname(lbm.__file__), "csrc")
    subprocess.check_call([lbm._nvcc(), "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a", "-I", csrc,
                           str(src), "-o", str(exe)])
    return str(exe)


@pytest.mark.parametrize("periodic", [(0, 0, 0), (1, 1, 1), (0, 1, 0)])
@pytest.mark.parametrize("n", BOXES + NARROW)
def test_offsets_of_large_boxes(program, n, periodic):
    assert n[0] * n[1] * n[2] * 19 <= 2e9  # accepted by lbm_create
    pitch = (n[0] + 31) // 32 * 32
    qs = pitch * n[1] * n[2]
    assert qs < 2 ** 31  # one population has 32-bit offsets,
    assert (18 * qs + 64 < 2 ** 31) == (n in NARROW)  # the buffer only in these
    nodes = list(itertools.product(*[sorted({0, 1, m // 2, m - 2, m - 1}) for m in n]))
    out = subprocess.run([program, *map(str, n), *map(str, periodic)], input="\n".join("%d %d %d" % v for v in nodes),
                         capture_output=True, text=True, check=True).stdout.split()
    got = iter(np.array(out, np.int64).reshape(-1, 3).tolist())
    top = 0
    for node in nodes:
        for q, c in enumerate(C19):
            src = [a - b for a, b in zip(node, c)]
            axis, face = -1, 0
            for d in range(3):
                if not 0 <= src[d] < n[d]:
                    if periodic[d]:
                        src[d] %= n[d]
                    elif axis < 0:
                        axis, face = d, int(src[d] > 0)
            if axis >= 0:
                src, q = node, q ^ 1  # the opposite population (pairs are adjacent)
            want = q * qs + (src[2] * n[1] + src[1]) * pitch + src[0]
            assert next(got) == [want, axis, face], (node, c)
            assert 0 <= want < 18 * qs
            top = max(top, want)
    assert top >= (2 ** 31 if n in BOXES else 2 ** 30)  # the box reaches the range


def test_planar_boxes_have_32_bit_offsets():
    """The largest D2Q9 buffers that lbm_create accepts (nodes 19 <= 2e9, axes up to 2^20)."""
    for n0 in list(range(2, 4200)) + [2 ** 20]:
        n1 = min(2 ** 20, int(2e9 / 19 / n0))
        assert 8 * ((n0 + 31) // 32 * 32) * n1 + 64 < 2 ** 31


def _context(n, storage, f):
    sim = lbm.LBM([lbm.make_config(lbm.LBM_D3Q19, n, bc=(lbm.LBM_WALL, lbm.LBM_WALL, lbm.LBM_PERIODIC), storage=storage,
                                   tau=0.8, max_particles=0)])
    sim._check(lbm.lib().lbm_set_populations(sim._h, 0, C.c_void_p(f.data_ptr()), 1))
    return sim


@gpu
@pytest.mark.parametrize("n,storage,gradient", [((129, 900, 900), lbm.LBM_FP32, False), ((129, 900, 900), lbm.LBM_FP16, True),
                                                ((5, 1500, 3600), lbm.LBM_FP16, True)])
def test_large_box_repeats_its_period(n, storage, gradient):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    if torch.cuda.get_device_properties(0).total_memory < 150e9:
        pytest.skip("needs 150 GB")
    lbm.build()
    period = 8
    reps = -(-n[2] // period)
    n = (n[0], n[1], reps * period)
    shape = (19, period, n[1], n[0])
    g = torch.Generator(device="cuda").manual_seed(7)
    f = (torch.rand(shape, device="cuda", generator=g) - 0.5) * 2e-3
    f[0] = 0
    seed = torch.rand(shape, device="cuda", generator=g) - 0.5

    def run(nz):
        def whole(t):
            return t if nz == period else t.repeat(1, reps, 1, 1)

        sim = _context((n[0], n[1], nz), storage, whole(f))
        out = {}
        if gradient:
            sim.adjoint_forward(2)
            s = whole(seed).reshape(-1)
            out["gradient"] = sim.adjoint_backward(seed_field=s, want_field=True)[1].reshape(19, nz, n[1], n[0])
            del s
            sim.adjoint_release()
        else:
            sim.step(2)
        N = sim.nodes()
        u, p = torch.empty(3 * N, device="cuda"), torch.empty(N, device="cuda")
        sim.fields_device(0, u, p)
        state = torch.empty(19 * N, device="cuda")
        sim._check(lbm.lib().lbm_get_populations(sim._h, 0, C.c_void_p(state.data_ptr()), 1))
        sim.sync()
        out.update(u=u.reshape(3, nz, n[1], n[0]), p=p.reshape(1, nz, n[1], n[0]), state=state.reshape(19, nz, n[1], n[0]))
        sim.close()
        return out

    small, large = run(period), run(n[2])
    for k in small:
        assert bool(small[k].abs().max() > 0), k
        for r in range(reps):
            assert torch.equal(large[k][:, r * period:(r + 1) * period], small[k]), (k, r)
    del small, large
    torch.cuda.empty_cache()
