// Rigid-body projection (Eq. 22) of a velocity field onto a set of particles,
// in a variant that allocates no memory: its scratch is a fixed array in the
// library's device image instead of memory from cudaMalloc or an allocator.
//
// It exists for callers that cannot allocate device memory at the point where
// they need the projection: a plugin whose host owns all device memory and
// forbids allocation, a frame loop that must not stall on the implicit device
// synchronisation of cudaMalloc/cudaFree, or code holding a stream it may only
// enqueue work on.  The context-based path (lbm_create ... lbm_step) computes
// the same sums inside the fused fluid kernel, with scratch from the caller's
// allocator.
//
// Limits: at most LBM_NOALLOC_MAX_PARTICLES particles, radii <= 120 lattice
// units in 2D and <= 40 in 3D (the bounds under which the exact integer sums
// fit in 64 bits).  Every call uses the same array: calls that overlap on the GPU (on
// different streams, or from several host threads) race and give wrong sums.
// The array stays allocated on every GPU that loads the library until the
// process exits.
#include <mutex>

#include "../../include/lbmpen.h"
#include "lbm_common.cuh"

namespace lbmpen {
namespace {

constexpr int NA_MAXP = LBM_NOALLOC_MAX_PARTICLES;
constexpr int NA_ERR = NA_MAXP * NPV;  // index of the error word after the sums
constexpr int NA_BLOCK = 256;
constexpr int NA_SLICE = 4096;         // nodes of a particle's box per block

// Scratch: int64 sums of Eq. 22 per particle (fixed point, as in the fused
// kernel) followed by one error word.
__device__ __align__(256) long long g_noalloc_scratch[NA_MAXP * NPV + 32];

__global__ void k_na_clear(long long* scratch, int np) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < np * NPV) scratch[i] = 0;
    if (i == 0) scratch[NA_ERR] = 0;
}

struct NaGrid {
    int n[3];
    int per[3];
    int D;
};

// Eq. 22 of particle p from its exact sums v: U = sum u / n and the angular
// velocity from the moments about floor(X), as in the context path's
// finalisation.  One warp; an FP64 instruction costs the same for one lane as
// for 32, so lane d < D divides for U_d and lane 8 + c for omega_c at once.
template <int D>
__device__ void na_finalize(int p, const double* Xp, const long long* v, double* U, double* W, int* count,
                            unsigned long long* err, int lane) {
    const double scale = 1.0 / (double)(1LL << FXBITS);
    const double cnt = (double)v[0];
    if (lane == 0) count[p] = (int)v[0];
    double phi[3] = {0, 0, 0}, Sd[3], Su[3], Sl[3];
    for (int d = 0; d < 3; ++d) {
        if (d < D) phi[d] = Xp[d] - floor(Xp[d]);
        Sd[d] = (double)v[1 + d];
        Su[d] = (double)v[10 + d] * scale;
        Sl[d] = (double)v[13 + d] * scale;
    }
    const double Lv[3] = {Sl[0] - (phi[1] * Su[2] - phi[2] * Su[1]), Sl[1] - (phi[2] * Su[0] - phi[0] * Su[2]),
                          Sl[2] - (phi[0] * Su[1] - phi[1] * Su[0])};
    const int ii[6] = {0, 1, 2, 0, 0, 1}, jj[6] = {0, 1, 2, 1, 2, 2};
    double rr[3][3];
    for (int k = 0; k < 6; ++k) {
        const int i = ii[k], j = jj[k];
        const double val = (double)v[4 + k] - phi[i] * Sd[j] - phi[j] * Sd[i] + cnt * phi[i] * phi[j];
        rr[i][j] = val;
        rr[j][i] = val;
    }
    double den, num = 0.0;  // omega_c = num / den on lane 8 + c
    const int c = lane - 8;
    if (D == 2) {
        den = rr[0][0] + rr[1][1];
        num = Lv[2];
    } else {
        const double tr = rr[0][0] + rr[1][1] + rr[2][2];
        double I[3][3];
        for (int i = 0; i < 3; ++i)
            for (int j = 0; j < 3; ++j) I[i][j] = (i == j ? tr : 0.0) - rr[i][j];
        den = I[0][0] * (I[1][1] * I[2][2] - I[1][2] * I[2][1]) - I[0][1] * (I[1][0] * I[2][2] - I[1][2] * I[2][0]) +
              I[0][2] * (I[1][0] * I[2][1] - I[1][1] * I[2][0]);
        double M[3][3];  // Cramer's rule: column c of I replaced by L
        for (int r = 0; r < 3; ++r)
            for (int q = 0; q < 3; ++q) M[r][q] = (q == c) ? Lv[r] : I[r][q];
        num = M[0][0] * (M[1][1] * M[2][2] - M[1][2] * M[2][1]) - M[0][1] * (M[1][0] * M[2][2] - M[1][2] * M[2][0]) +
              M[0][2] * (M[1][0] * M[2][1] - M[1][1] * M[2][0]);
    }
    // no node, or a node set without rotational inertia (I is positive
    // semi-definite; singular for collinear node sets)
    const bool degenerate = v[0] == 0 || !(den > 0.0);
    if (degenerate && lane == 0) atomicOr(err, 8ull);
    if (lane < D) num = lane == 0 ? Su[0] : (lane == 1 ? Su[1] : Su[2]);
    const double q = num / (lane < D ? cnt : den);
    const double out = degenerate ? 0.0 : q;
    constexpr int NW = D == 2 ? 1 : 3;
    if (lane < D) U[p * D + lane] = out;
    else if (c >= 0 && c < NW) W[p * NW + c] = out;
}

// One block per (particle p, slice of up to NA_SLICE nodes of p's bounding
// box).  A node is counted for p when it lies inside p (Eq. 9) and inside no
// particle of lower index, the owner rule of the fused kernel.  Bound by
// latency: the bytes are the particles' own nodes, a few per thread.  So the
// indicator goes through the fused kernel's FP32 band and only nodes in the
// band take the exact FP64 test (an FP64 instruction holds its pipe for ~64
// cycles; testing every node of the box in FP64 was most of the time), the
// sums are exact integer warp reductions, and with ONE (every box fits one
// slice) the block goes on to the second pass itself: one launch, no scratch
// sums.  500 disks R ~ U(6,12) in a 1024 x 4096 field, the whole call with its
// host wait: 69 us before (every node of the largest box in FP64, 64-bit
// shuffles and atomics, three launches), 36 us now.  NA_SLICE nodes take 16
// rounds of a block; larger boxes spread over blocks instead.
template <int D, bool ONE>
__global__ void __launch_bounds__(NA_BLOCK) k_na_accumulate(NaGrid g, const float* __restrict__ u, int np,
                                                            const double* __restrict__ X,
                                                            const double* __restrict__ R, double max_radius,
                                                            long long* scratch, double* U, double* W, int* count) {
    __shared__ int lower[64];  // lower-index particles that overlap p
    __shared__ int nlower;
    __shared__ long long red[NA_BLOCK / 32][NPV];
    __shared__ long long tot[NPV];
    unsigned long long* err = reinterpret_cast<unsigned long long*>(scratch + NA_ERR);
    const int p = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    double Xp[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < D; ++d) Xp[d] = X[p * D + d];
    const double Rp = R[p];
    const bool ok_radius = Rp >= 0.0 && !(Rp > max_radius);  // block-uniform
    if (threadIdx.x == 0) {
        nlower = 0;
        if (!ok_radius) atomicOr(err, 1ull);
    }
    __syncthreads();
    if (!ok_radius && !ONE) return;
    if (ok_radius) {
        const float xf[3] = {(float)Xp[0], (float)Xp[1], (float)Xp[2]};
        for (int j = threadIdx.x; j < p; j += NA_BLOCK) {
            // FP32 first: on an axis of up to 2^20 nodes the coordinates of two
            // particles that share a node carry an error below 0.1 each, so a pair 1
            // beyond reach along a non-periodic axis cannot overlap.  Longer axes
            // (from 2^25 nodes the error exceeds the margin) leave it to FP64 below.
            const double Rj = R[j];
            const float reachf = (float)Rj + (float)Rp + 3.0f;
            bool far = false;
            double Xj[3];
#pragma unroll
            for (int d = 0; d < D; ++d) {
                Xj[d] = X[j * D + d];
                far |= !g.per[d] && g.n[d] <= (1 << 20) && fabsf((float)Xj[d] - xf[d]) > reachf;
            }
            if (far) continue;
            double d2 = 0.0;
#pragma unroll
            for (int d = 0; d < D; ++d) {
                double dx = Xj[d] - Xp[d];
                if (g.per[d]) dx -= g.n[d] * rint(dx / g.n[d]);
                d2 += dx * dx;
            }
            const double reach = Rj + Rp + 2.0;
            if (d2 <= reach * reach) {
                const int slot = atomicAdd(&nlower, 1);
                if (slot < 64) lower[slot] = j;
                else atomicOr(err, 2ull);
            }
        }
    }
    __syncthreads();
    const int nl = min(nlower, 64);
    // bounding box of p, node range [floor(X - R) - 1, floor(X + R) + 1] per axis
    int lo[3] = {0, 0, 0}, len[3] = {1, 1, 1}, ref[3] = {0, 0, 0};
    float frac[3] = {0.f, 0.f, 0.f};
    int total = 0;
    if (ok_radius) {
        long long prod = 1;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            lo[d] = (int)floor(Xp[d] - Rp) - 1;
            len[d] = (int)floor(Xp[d] + Rp) + 1 - lo[d] + 1;
            ref[d] = (int)floor(Xp[d]);
            frac[d] = (float)(Xp[d] - (double)ref[d]);
            prod *= len[d];
        }
        // a box within max_radius never exceeds the launch's slices; a centre
        // beyond the int range would, and owns nothing
        total = (int)max(0LL, min(prod, (long long)(ONE ? NA_SLICE : (int)gridDim.y * NA_SLICE)));
    }
    const float Rf = (float)Rp, R2f = Rf * Rf;  // the band of the fused kernel's filter
    const float R2lo = R2f * (1.0f - 2e-5f) - 2e-4f, R2hi = R2f * (1.0f + 2e-5f) + 2e-4f;
    const int pm = g.per[0] | (g.per[1] << 1) | (g.per[2] << 2);
    PRec pr;
    for (int d = 0; d < 3; ++d) pr.X[d] = Xp[d];
    pr.R2 = Rp * Rp;
    pr.shape = 0;  // disks and spheres only
    const long long N = (long long)g.n[0] * g.n[1] * g.n[2];
    int icnt = 0, id[3] = {0, 0, 0}, idd[6] = {0, 0, 0, 0, 0, 0};
    long long su[3] = {0, 0, 0}, sl[3] = {0, 0, 0};
    const int k1 = ONE ? total : min(total, ((int)blockIdx.y + 1) * NA_SLICE);
    for (int k = (ONE ? 0 : (int)blockIdx.y * NA_SLICE) + threadIdx.x; k < k1; k += NA_BLOCK) {
        const int off[3] = {k % len[0], (k / len[0]) % len[1], D == 3 ? k / (len[0] * len[1]) : 0};
        int xyz[3] = {0, 0, 0}, dd[3] = {0, 0, 0};
        float d2 = 0.f;
        bool ok = true;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            int x = lo[d] + off[d];
            dd[d] = x - ref[d];  // offset from floor(X), unwrapped
            const float r = (float)dd[d] - frac[d];
            d2 = fmaf(r, r, d2);
            if (g.per[d]) x = ((x % g.n[d]) + g.n[d]) % g.n[d];
            else if (x < 0 || x >= g.n[d]) ok = false;
            xyz[d] = x;
        }
        if (!ok || d2 > R2hi) continue;
        if (!(d2 < R2lo) && !inside_exact<D>(&pr, xyz[0], xyz[1], xyz[2], g.n[0], g.n[1], g.n[2], pm)) continue;
        bool mine = true;
        for (int i = 0; i < nl && mine; ++i) {
            PRec q;
            const int j = lower[i];
            for (int d = 0; d < 3; ++d) q.X[d] = d < D ? X[j * D + d] : 0.0;
            q.R2 = R[j] * R[j];
            q.shape = 0;
            if (inside_exact<D>(&q, xyz[0], xyz[1], xyz[2], g.n[0], g.n[1], g.n[2], pm)) mine = false;
        }
        if (!mine) continue;
        const long long node = ((long long)xyz[2] * g.n[1] + xyz[1]) * g.n[0] + xyz[0];
        long long ux[3] = {0, 0, 0};
        float uu = 0.f;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const float v = u[d * N + node];
            uu = fmaf(v, v, uu);
            ux[d] = to_fx32(v);
        }
        // the speed bound of the exact sums, as in the fused kernel's
        // divergence test (true for NaN too; to_fx32 would clamp silently)
        if (!(uu < 0.25f)) atomicOr(err, 4ull);
        icnt += 1;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            id[d] += dd[d];
            idd[d] += dd[d] * dd[d];
            su[d] += ux[d];
        }
        idd[3] += dd[0] * dd[1]; idd[4] += dd[0] * dd[2]; idd[5] += dd[1] * dd[2];
        sl[0] += (long long)dd[1] * ux[2] - (long long)dd[2] * ux[1];
        sl[1] += (long long)dd[2] * ux[0] - (long long)dd[0] * ux[2];
        sl[2] += (long long)dd[0] * ux[1] - (long long)dd[1] * ux[0];
    }
    long long v[NPV];
    v[0] = __reduce_add_sync(0xffffffffu, icnt);
#pragma unroll
    for (int d = 0; d < 3; ++d) v[1 + d] = d < D ? __reduce_add_sync(0xffffffffu, id[d]) : 0;
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        const bool need = D == 3 || d == 0 || d == 1 || d == 3;
        v[4 + d] = need ? __reduce_add_sync(0xffffffffu, idd[d]) : 0;
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        v[10 + d] = d < D ? warp_sum_fx(su[d]) : 0;
        v[13 + d] = (D == 3 || d == 2) ? warp_sum_fx(sl[d]) : 0;
    }
    if (lane == 0)
#pragma unroll
        for (int i = 0; i < NPV; ++i) red[warp][i] = v[i];
    __syncthreads();
    if (threadIdx.x < NPV) {
        long long t = 0;
        for (int i = 0; i < NA_BLOCK / 32; ++i) t += red[i][threadIdx.x];
        tot[threadIdx.x] = t;
        if (!ONE && t != 0)
            atomicAdd(reinterpret_cast<unsigned long long*>(scratch + (long long)p * NPV) + threadIdx.x,
                      (unsigned long long)t);
    }
    if (ONE) {
        __syncthreads();
        if (warp == 0) na_finalize<D>(p, Xp, tot, U, W, count, err, lane);
    }
}

// The second pass of sliced particles, one warp each.
template <int D>
__global__ void k_na_finalize(int np, const double* __restrict__ X, long long* scratch, double* U, double* W,
                              int* count) {
    const int p = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (p >= np) return;
    double Xp[3] = {0, 0, 0};
    for (int d = 0; d < D; ++d) Xp[d] = X[p * D + d];
    na_finalize<D>(p, Xp, scratch + (long long)p * NPV, U, W, count,
                   reinterpret_cast<unsigned long long*>(scratch + NA_ERR), threadIdx.x & 31);
}

// The launches of one call; box: nodes of the largest particle's bounding box.
template <int D>
cudaError_t launch_noalloc(const NaGrid& g, const float* u, int np, const double* X, const double* R, double max_radius,
                           long long box, long long* scratch, double* U, double* W, int* count, cudaStream_t st) {
    if (box <= NA_SLICE) {
        const cudaError_t e = cudaMemsetAsync(scratch + NA_ERR, 0, sizeof(long long), st);
        if (e != cudaSuccess) return e;
        k_na_accumulate<D, true><<<np, NA_BLOCK, 0, st>>>(g, u, np, X, R, max_radius, scratch, U, W, count);
        return cudaGetLastError();
    }
    k_na_clear<<<(np * NPV + 255) / 256, 256, 0, st>>>(scratch, np);
    const dim3 grid((unsigned)np, (unsigned)((box + NA_SLICE - 1) / NA_SLICE));
    k_na_accumulate<D, false><<<grid, NA_BLOCK, 0, st>>>(g, u, np, X, R, max_radius, scratch, U, W, count);
    k_na_finalize<D><<<(np + 3) / 4, 128, 0, st>>>(np, X, scratch, U, W, count);
    return cudaGetLastError();
}

// Device address of the scratch array, looked up once per device (with that
// device current) and cached.
std::mutex g_na_mutex;
long long* g_na_ptr[256] = {nullptr};

long long* scratch_address(int dev, cudaError_t* err) {
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (dev < 0 || dev >= 256) {
        *err = cudaErrorInvalidDevice;
        return nullptr;
    }
    if (!g_na_ptr[dev]) {
        void* p = nullptr;
        *err = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (*err != cudaSuccess) return nullptr;
        g_na_ptr[dev] = static_cast<long long*>(p);
    }
    *err = cudaSuccess;
    return g_na_ptr[dev];
}

}  // namespace
}  // namespace lbmpen

using namespace lbmpen;

extern "C" int lbm_rigid_projection_noalloc(int dim, const int* n, const int* periodic, const float* u,
                                            int np, const double* pos, const double* radius,
                                            double max_radius, double* vel, double* omega,
                                            int* count, void* stream) {
    if ((dim != 2 && dim != 3) || !n || !periodic || np < 0) return LBM_ERR_INVALID;
    if (np > NA_MAXP) return LBM_ERR_INVALID;  // beyond the fixed scratch array
    if (np == 0) return LBM_OK;
    if (!u || !pos || !radius || !vel || !omega || !count) return LBM_ERR_INVALID;
    if (!(max_radius >= 0.0) || max_radius > (dim == 3 ? MAX_RADIUS_3D : MAX_RADIUS)) return LBM_ERR_INVALID;
    NaGrid g;
    g.D = dim;
    for (int d = 0; d < 3; ++d) {
        g.n[d] = d < dim ? n[d] : 1;
        g.per[d] = d < dim ? (periodic[d] != 0) : 1;
        if (g.n[d] < 1) return LBM_ERR_INVALID;
        // a particle's box must not wrap onto itself on a periodic axis
        if (d < dim && g.per[d] && (long long)(2.0 * max_radius) + 4 > g.n[d]) return LBM_ERR_INVALID;
    }
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return LBM_ERR_CUDA;
    cudaError_t e;
    long long* scratch = scratch_address(dev, &e);
    if (!scratch) return LBM_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const long long side = (long long)(2.0 * max_radius) + 4;
    if (dim == 2) e = launch_noalloc<2>(g, u, np, pos, radius, max_radius, side * side, scratch, vel, omega, count, st);
    else e = launch_noalloc<3>(g, u, np, pos, radius, max_radius, side * side * side, scratch, vel, omega, count, st);
    if (e != cudaSuccess) return LBM_ERR_CUDA;
    long long err = 0;
    if (cudaMemcpyAsync(&err, scratch + NA_ERR, sizeof err, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return LBM_ERR_CUDA;
    if (err & 1) return LBM_ERR_INVALID;   // a radius above max_radius
    if (err & 4) return LBM_ERR_DIVERGED;  // a velocity component is non-finite or |u| >= 1/2
    if (err & 2) return LBM_ERR_CAPACITY;  // a particle overlaps more than 64 of lower index
    if (err & 8) return LBM_ERR_PARTICLE;  // a particle owns no node, or its nodes have no inertia
    return LBM_OK;
}
