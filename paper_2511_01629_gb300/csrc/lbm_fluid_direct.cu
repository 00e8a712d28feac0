// Fused stream-collide-penalize kernel that loads straight into registers, one
// warp per 64-node row of a tile: D3Q19, and D2Q9 on small grids.
//
// Pull streaming reads every population value once, so staging a D3Q19 tile
// through shared memory saves no traffic, and its tensor copies are small (18
// boxes of a few 64-node rows): the copy engine, not HBM, set the time of the
// staged kernel (FP32 and FP16 storage took the same time per node).  Here a
// lane takes two adjacent nodes: populations with c_x = 0 arrive by one
// 8-byte (FP16: 4-byte) load, the others by two scalar loads of the shifted
// pair; all 18 are in flight before the first is used, and enough warps are
// resident to cover the latency: 80 registers, 24 warps per SM (some 200 bytes of
// spills, in the solid path) beat 128 registers and 16 warps (256 x 256 x 512, 8
// spheres, per step: FP32 934 -> 812 us, 5.95 TB/s; FP16 151 x 133 x 203
// 157 -> 135 us; 72 registers: 879 and 136).  Rows at a y or z face take
// pull_pre_all; the x faces only change the address of an edge node's load.
// On a small D2Q9 grid the kernel is bound by its chain of latencies, which is
// shorter here than the staged kernel's (default_shape has the figures).
#include "lbm_common.cuh"

namespace lbmpen {

namespace {

constexpr int TW = 64;

struct DescEnv {
    const InstDesc& in;
    long long* sums;
    __device__ __forceinline__ int n(int d) const { return in.n[d]; }
    __device__ __forceinline__ int per(int d) const { return in.periodic[d]; }
    __device__ __forceinline__ const PRec* prec() const { return in.prec; }
    __device__ __forceinline__ float gdrive(int d) const { return in.gdrive[d]; }
    __device__ __forceinline__ long long* tot() const { return sums; }
};

}  // namespace

template <int Q, class S, class I>
__global__ void __launch_bounds__(256, Q == 9 ? 4 : 3) k_fluid_direct(const InstDesc* __restrict__ insts,
                                                         const uint16_t* __restrict__ tile_inst, int ninst, int par, Shape sh,
                                                         int commit) {
    using L = Lat<Q>;
    constexpr int D = L::D;
    constexpr int QS = Q - 1;
    __shared__ Cand cand[LIST_CAP];
    const int t = blockIdx.x;
    const InstDesc& in = insts[ninst > 1 ? (int)tile_inst[t] : 0];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const int local = t - in.tile0;
    const int ntx = in.ntile[0], nty = in.ntile[1];
    const int rest = local / ntx;
    const int x0 = (local - rest * ntx) * TW, y0 = (rest % nty) * sh.ty, z0 = (rest / nty) * sh.tz;
    const int nx = in.n[0], ny = in.n[1], nz = in.n[2];
    const int rows = sh.ty * sh.tz, lty = __ffs(sh.ty) - 1;  // tile rows along y: a power of two
    const int x = x0 + 2 * lane;
    const bool edge = x0 == 0 || x0 + TW >= nx;
    const float sload = in.s_load;
    const S* fin = static_cast<const S*>(in.f[par]);
    const I qs = (I)in.qstride;
    float2 f[QS];
    dep_wait();  // the populations and lists of the previous step
    dep_launch();
    auto pull_row = [&](int r) {  // false: the row lies beyond the box
        const int y = y0 + (r & (sh.ty - 1)), z = z0 + (r >> lty);
        if (r >= rows || y >= ny || z >= nz) return false;
        if (y >= 1 && y + 1 < ny && (D == 2 || (z >= 1 && z + 1 < nz))) {
            if (edge) pull_pair<Q, S, true>(in, fin, qs, x, y, z, f);
            else pull_pair<Q, S, false>(in, fin, qs, x, y, z, f);
        } else {
            float g[QS];
            pull_pre_all<Q, S>(in, fin, min(x, nx - 1), y, z, qs, g);
#pragma unroll
            for (int q = 0; q < QS; ++q) f[q].x = g[q];
            pull_pre_all<Q, S>(in, fin, min(x + 1, nx - 1), y, z, qs, g);
#pragma unroll
            for (int q = 0; q < QS; ++q) f[q].y = g[q];
        }
        return true;
    };
    // the first row's populations are in flight while the candidates arrive
    int r = warp;
    bool have = pull_row(r);
    int ncand = 0;
    if (in.np > 0) {
        ncand = min(in.list_cnt[par][local], LIST_CAP);
        const uint4* src = reinterpret_cast<const uint4*>(static_cast<const Cand*>(in.list_rec[par]) +
                                                          (long long)local * LIST_CAP);
        for (int i = threadIdx.x; i < ncand * (CAND_BYTES / 16); i += blockDim.x) reinterpret_cast<uint4*>(cand)[i] = src[i];
        if (commit && threadIdx.x == 0) in.list_cnt[par ^ 1][local] = 0;  // the next step's list starts empty
        __syncthreads();
    }
    const CollK ck = make_collk<Q>(make_collp(in));
    const bool free = in.gdrive[0] == 0.f && in.gdrive[1] == 0.f && in.gdrive[2] == 0.f;
    const DescEnv env{in, commit ? in.tot[par] : in.tot_scratch};
    S* __restrict__ fout = static_cast<S*>(in.f[par ^ 1]);
    bool bad = false;
    for (;;) {
        if (have) {
            const int y = y0 + (r & (sh.ty - 1)), z = z0 + (r >> lty);
            bad |= finish_pair<Q, S, false>(env, f, ck, sload, in.s_store, free, cand, ncand, x0, x, y, z, lane,
                                            fout + ((z * ny + y) * in.pitch + x), (int)in.qstride);
        }
        r += nwarps;
        if (r >= rows) break;
        have = pull_row(r);
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(in.status, ST_DIVERGED);
}

int direct_tile_width() { return TW; }

// The kernel of a lattice, storage type and width of offsets (wide_offsets).  64-bit
// addresses on every box cost 151 x 133 x 203 FP16 1.5 % (160 steps 21.55 ms against
// 21.25) and 256 x 256 x 512 FP32 0.2 %.
template <class F>
static auto direct_kernel(int Q, int fp16, bool wide, F&& go) {
    if (Q == 9) return fp16 ? go(k_fluid_direct<9, __half, int>) : go(k_fluid_direct<9, float, int>);
    if (!wide) return fp16 ? go(k_fluid_direct<19, __half, int>) : go(k_fluid_direct<19, float, int>);
    return fp16 ? go(k_fluid_direct<19, __half, long long>) : go(k_fluid_direct<19, float, long long>);
}

int fluid_direct_blocks_per_sm(int Q, int fp16, bool wide, const Shape& sh) {
    return direct_kernel(Q, fp16, wide, [&](auto kern) {
        int nb = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 32 * sh.warps, 0);
        return nb;
    });
}

cudaError_t launch_fluid_direct(int Q, int fp16, bool wide, const InstDesc* insts, const uint16_t* tile_inst, int ninst,
                                int ntiles, int par, const Shape& sh, int commit, cudaStream_t st) {
    return direct_kernel(Q, fp16, wide, [&](auto kern) {
        return launch_dep(kern, dim3((unsigned)ntiles), 32 * sh.warps, 0, st, insts, tile_inst, ninst, par, sh, commit);
    });
}

}  // namespace lbmpen
