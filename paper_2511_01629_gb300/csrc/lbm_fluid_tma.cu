// TMA-pipelined variant of the fused stream-collide-penalize kernel (D2Q9).
//
// Persistent blocks of one producer warp and NC consumer warps.  The producer
// takes tiles from a work counter (successive claims alternate between the
// two ends of the tile range) and fills a ring of shared-memory stages: the
// tile's populations by cp.async.bulk.tensor (one box of every population
// over the tile rows and one halo row on each side), 32*k nodes wide
// plus a 16-byte halo on both sides so that every box starts on a 16-byte
// boundary, and the tile's candidate particles by one bulk copy of the
// records the particle kernel listed for the tile.  Everything else the
// producer needs comes from a per-block shared table of instance constants,
// or was fetched one tile ahead (the next tile's list count and the values
// its x-edge node pulls across the face, by cp.async), so its own path per
// tile touches no global memory.  The copies of a stage are counted by its
// mbarrier; each consumer lane pulls two adjacent nodes' populations from
// shared memory at x - c_x, collides them with packed FP32x2 arithmetic,
// stores them to HBM with 8-byte coalesced stores, and adds the velocities
// of solid nodes to their particle's sums of Eq. 22.  At a y wall a node's own
// opposite populations, staged too, come back; the rows at a periodic y face
// gather theirs from the previous buffer directly.
//
// Every mbarrier wait is bounded in time; on expiry the kernel records a
// timeout in the status word, waits (bounded) for the copies it issued and
// returns.
#include <cuda.h>

#include <mutex>
#include <type_traits>

#include "lbm_common.cuh"

namespace lbmpen {

namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// Raise the bytes the current phase waits for, without arriving.
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}
// Wait for the phase of the given parity; false once limit_ns has passed.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned long long limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = now_ns();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try_wait(bar, parity)) return true;
        if (now_ns() - t0 > limit_ns) return false;
    }
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int c0, int c1, int c2,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

// One bulk copy global -> shared counted by an mbarrier (16-byte aligned
// addresses, a multiple of 16 bytes).
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// 4-byte asynchronous copy global -> shared (completion: cp_async_wait_all)
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

constexpr int Q = 9;  // D3Q19 takes k_fluid_direct
using L = Lat<Q>;
// Populations with c_x = +1 (equally, -1): the ones an x-edge node pulls
// across its face.
__host__ __device__ constexpr int edge_pops() { return 3; }
constexpr unsigned long long WAIT_LIMIT_NS = 2000000000ull;  // 2 s

// The constants of one instance that a tile needs, copied once per block
// into a shared-memory table (for up to TI_MAX instances) so that neither the
// producer nor the consumers go to global memory for them in the tile loop.
struct __align__(16) TInst {
    const void* f[2];          // population buffers
    long long* tot[3];         // totals of Eq. 22: per parity, scratch
    const PRec* prec;
    int* status;
    int* lcnt[2];              // tile list counts per parity
    const Cand* lrec[2];       // candidate records per parity
    long long qstride;
    int tile0, ntx, pitch, np;
    int n[3], per[3];
    float gdrive[3], sload, sstore, keep, fpref, alpha;
    int free;                  // no body force: fluid nodes take collide2_free
    float ewt[2][edge_pops()];  // moving-wall term of the populations an x-edge node pulls
                               //   across the low (0) / high (1) x face
};
constexpr int TI_MAX = 64;
constexpr int TI_WORDS = (int)(sizeof(TInst) / 16);

__device__ __forceinline__ void make_tinst(TInst& t, const InstDesc& in) {
    for (int b = 0; b < 2; ++b) {
        t.f[b] = in.f[b];
        t.lcnt[b] = in.list_cnt[b];
        t.lrec[b] = static_cast<const Cand*>(in.list_rec[b]);
    }
    t.tot[0] = in.tot[0];
    t.tot[1] = in.tot[1];
    t.tot[2] = in.tot_scratch;
    t.prec = in.prec;
    t.status = in.status;
    t.qstride = in.qstride;
    t.tile0 = in.tile0;
    t.ntx = in.ntile[0];
    t.pitch = in.pitch;
    t.np = in.np;
    for (int d = 0; d < 3; ++d) {
        t.n[d] = in.n[d];
        t.per[d] = in.periodic[d];
        t.gdrive[d] = in.gdrive[d];
    }
    t.sload = in.s_load;
    t.sstore = in.s_store;
    t.keep = in.keep;
    t.fpref = in.fpref;
    t.alpha = in.alpha;
    t.free = in.gdrive[0] == 0.f && in.gdrive[1] == 0.f && in.gdrive[2] == 0.f;
    for (int face = 0; face < 2; ++face)
        for (int k = 0; k < edge_pops(); ++k) t.ewt[face][k] = 0.f;
    for (int face = 0; face < 2; ++face) {  // face 0 is pulled across by c_x = +1, face 1 by c_x = -1
        const int ecx = face == 0 ? 1 : -1;
        for (int k = 0, q = 1; q < Q; ++q)
            if (L::c(q, 0) == ecx) t.ewt[face][k++] = in.wterm[0][face][q];
    }
}

// What finish_pair needs of the instance, read from the shared copy when it does.
struct TileEnv {
    const TInst& ti;
    long long* sums;
    __device__ __forceinline__ int n(int d) const { return ti.n[d]; }
    __device__ __forceinline__ int per(int d) const { return ti.per[d]; }
    __device__ __forceinline__ const PRec* prec() const { return ti.prec; }
    __device__ __forceinline__ float gdrive(int d) const { return ti.gdrive[d]; }
    __device__ __forceinline__ long long* tot() const { return sums; }
};

// Per-tile record the producer writes next to the staged populations.
struct __align__(16) StageHdr {
    TInst ti;   // the tile's instance
    int tile;   // global tile index, -1 = no more work
    int ncand;
    int inst;
    int x0, y0;
    int ex;     // bit 0: the tile holds x = 0, bit 1: it holds x = nx - 1 (the values
                //   these nodes pull across the face are staged, side by side)
};

// The next tile of the producer, prepared one iteration ahead: its place in
// registers; its list count and the values its x-edge nodes pull across the
// faces in flight to the shared prefetch buffer (cp.async) while the producer
// waits for a free stage.
constexpr int EDGE_ITERS = 2;  // edge values per lane: 2 sides x 8 rows x 3 populations at most
struct TileAhead {
    int t, ii, local, x0, y0, ex, np;
    float sload;
    float add[EDGE_ITERS];
    int hsel;  // FP16: bit j set = value j is the upper half of its 4-byte word
};
constexpr int PRE_WORDS = 32 * EDGE_ITERS + 8;  // per prefetch buffer: edge values, the list count
constexpr int PRE_CNT = 32 * EDGE_ITERS;

}  // namespace

// Geometry of the shared-memory ring, identical on host and device.
struct TmaLayout {
    int bw;          // box width (nodes) = tile width + 2 halo
    int stage;       // bytes of all populations of one stage
    int pops_bytes;  // stages * stage
    int hdr_off, cand_off, edge_off, tab_off, pre_off, bar_off, bytes;
};

__host__ __device__ inline TmaLayout tma_layout(int ssize, int tw, int rows, int stages, int ninst) {
    TmaLayout L;
    const int halo = 16 / ssize;
    const int ntab = ninst < TI_MAX ? ninst : TI_MAX;
    L.bw = tw + 2 * halo;
    // one box per tile: all populations, rows y0 - 1 .. y0 + rows, densely packed
    L.stage = ((Q - 1) * L.bw * (rows + 2) * ssize + 127) & ~127;
    L.pops_bytes = stages * L.stage;
    L.hdr_off = L.pops_bytes;
    L.cand_off = L.hdr_off + (int)sizeof(StageHdr) * stages;  // 16-byte aligned (bulk copies)
    L.edge_off = L.cand_off + CAND_BYTES * LIST_CAP * stages;
    L.tab_off = (L.edge_off + (int)sizeof(float) * 2 * rows * edge_pops() * stages + 15) & ~15;
    L.pre_off = L.tab_off + (int)sizeof(TInst) * ntab;
    L.bar_off = L.pre_off + 4 * 2 * PRE_WORDS;
    L.bytes = L.bar_off + 16 * stages + 128;  // + alignment slack of the base
    return L;
}

// The k-th population (0-based) with c_x == ecx.
__device__ __forceinline__ int edge_pop(int ecx, int k) {
    int q = 1;
    for (int m = 0, qq = 1; qq < Q; ++qq)
        if (L::c(qq, 0) == ecx && m++ == k) q = qq;
    return q;
}

// Register budget: two blocks of 9 warps per SM; each lane collides two
// nodes at a time.
template <class S, int TW, int ROWS>
__global__ void __launch_bounds__(288, 2) k_fluid_tma(const InstDesc* __restrict__ insts,
                                                   const CUtensorMap* __restrict__ tmaps,
                                                   const uint16_t* __restrict__ tile_inst, int ntiles,
                                                   int par, Shape sh, int commit, int* tile_ctr,
                                                   int stages, int ninst) {
    constexpr int QS = Q - 1;
    constexpr int H = 16 / (int)sizeof(S);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    // Base of the ring rounded up to 128 bytes by an offset from the shared
    // array itself: a pointer rebuilt from an integer would lose its address
    // space, and every access through it would become a generic load.
    unsigned char* smem = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
    constexpr int rows = ROWS;  // == sh.ty
    constexpr int BW = TW + 2 * H;
    constexpr int SLAB = BW * (ROWS + 2);  // elements between populations in a stage
    const TmaLayout LY = tma_layout((int)sizeof(S), TW, rows, stages, ninst);
    StageHdr* hdr = reinterpret_cast<StageHdr*>(smem + LY.hdr_off);
    Cand* cands = reinterpret_cast<Cand*>(smem + LY.cand_off);
    float* edgev = reinterpret_cast<float*>(smem + LY.edge_off);  // [stages][side][rows][QE]
    TInst* tab = reinterpret_cast<TInst*>(smem + LY.tab_off);
    uint32_t* pre = reinterpret_cast<uint32_t*>(smem + LY.pre_off);  // [2][PRE_WORDS]
    constexpr int QE = edge_pops();
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + LY.bar_off);
    uint64_t* empty = full + stages;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nc = (blockDim.x >> 5) - 1;  // consumer warps
    const int ntab = ninst < TI_MAX ? ninst : TI_MAX;
    if (threadIdx.x == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], nc);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int i = threadIdx.x; i < ntab; i += blockDim.x) make_tinst(tab[i], insts[i]);
    __syncthreads();
    dep_wait();  // the populations, lists and work counter of the previous step
    dep_launch();

    if (warp == 0) {
        // ---------------------------------------------------------- producer
        // the lists and populations were written by plain stores; the copies below
        // read them through the async proxy
        if (lane == 0) asm volatile("fence.proxy.async.global;" ::: "memory");
        // Tiles come from a work counter; claims alternate between the two
        // ends of the tile range (the slower y-face rows come first).  Two
        // claims are in flight, and everything the next tile needs from
        // global memory is loaded one iteration ahead, so the producer's
        // own path per tile touches only shared memory.
        bool ok = true;
        int issued = 0;
        int c_cur = 0, c_nxt = 0;
        if (lane == 0) {
            c_cur = atomicAdd(&tile_ctr[0], 1);
            c_nxt = atomicAdd(&tile_ctr[0], 1);
        }
        // instance of a tile without a memory round trip: votes over the
        // first tiles of up to TI_MAX instances in the table (lanes hold two)
        const int tf0 = lane < ntab ? tab[lane].tile0 : 0x7fffffff;
        const int tf1 = lane + 32 < ntab ? tab[lane + 32].tile0 : 0x7fffffff;
        auto ahead = [&](int c, int buf) {
            TileAhead a;
            a.t = -1;
            a.np = 0;
            a.ex = 0;
            a.sload = 1.f;
#pragma unroll
            for (int j = 0; j < EDGE_ITERS; ++j) a.add[j] = 0.f;
            a.hsel = 0;
            uint32_t* pb = pre + buf * PRE_WORDS;
            const int cc = __shfl_sync(0xffffffffu, c, 0);
            if (cc >= ntiles) return a;
            const int t = (cc & 1) ? ntiles - 1 - (cc >> 1) : (cc >> 1);
            a.t = t;
            a.ii = ninst <= TI_MAX ? __popc(__ballot_sync(0xffffffffu, t >= tf0)) +
                                         __popc(__ballot_sync(0xffffffffu, t >= tf1)) - 1
                                   : (int)tile_inst[t];
            const InstDesc& in = insts[a.ii];
            const bool tb = ninst <= TI_MAX;
            const int tile0 = tb ? tab[a.ii].tile0 : in.tile0;
            const int ntx = tb ? tab[a.ii].ntx : in.ntile[0];
            const int n[2] = {tb ? tab[a.ii].n[0] : in.n[0], tb ? tab[a.ii].n[1] : in.n[1]};
            a.np = tb ? tab[a.ii].np : in.np;
            a.sload = tb ? tab[a.ii].sload : in.s_load;
            a.local = t - tile0;
            a.x0 = (a.local % ntx) * TW;
            a.y0 = a.local / ntx * rows;
            if (lane == 0) {
                if (a.np > 0) cp_async4(pb + PRE_CNT, (tb ? tab[a.ii].lcnt[par] : in.list_cnt[par]) + a.local);
                else pb[PRE_CNT] = 0u;
            }
            a.ex = (a.x0 == 0 ? 1 : 0) | (a.x0 + TW >= n[0] ? 2 : 0);
            if (a.ex) {
                // the values the edge nodes x = 0 (side 0) and x = n - 1 (side 1) pull
                // across their x face in rows whose other sources lie inside the box
                // (rows that do not use them may get any in-bounds value)
                const S* fin = static_cast<const S*>(tb ? tab[a.ii].f[par] : in.f[par]);
                const long long qstr = tb ? tab[a.ii].qstride : in.qstride;
                const int pitch = tb ? tab[a.ii].pitch : in.pitch;
                const bool xper = (tb ? tab[a.ii].per[0] : in.periodic[0]) != 0;
#pragma unroll
                for (int j = 0; j < (2 * ROWS * QE + 31) / 32; ++j) {
                    const int l = lane + 32 * j;
                    if (l >= 2 * rows * QE) continue;
                    const int side = l >= rows * QE ? 1 : 0;
                    if (!((a.ex >> side) & 1)) continue;
                    const int r = (l - side * rows * QE) / QE, k = (l - side * rows * QE) % QE;
                    const int ecx = side ? -1 : 1, xe = side ? n[0] - 1 : 0;
                    const int q = edge_pop(ecx, k);
                    const int y = a.y0 + r, ys = y - L::c(q, 1);
                    const S* src = nullptr;
                    if (!xper) {  // bounce-back at the x wall
                        if (y < n[1]) src = pop(fin, L::opp(q), qstr) + (y * pitch + xe);
                        a.add[j] = tb ? tab[a.ii].ewt[side][k] : in.wterm[0][side][q];
                    } else if (y < n[1] && ys >= 0 && ys < n[1]) {
                        src = pop(fin, q, qstr) + (ys * pitch + (side ? 0 : n[0] - 1));  // periodic wrap
                    }
                    if (src) {
                        const uintptr_t ad = reinterpret_cast<uintptr_t>(src);
                        if (sizeof(S) == 2 && (ad & 2)) a.hsel |= 1 << j;
                        cp_async4(pb + l, reinterpret_cast<const void*>(ad & ~(uintptr_t)3));
                    } else {
                        pb[l] = 0u;
                    }
                }
            }
            cp_async_commit();
            return a;
        };
        TileAhead nx_ = ahead(c_cur, 0);
        for (int it = 0;; ++it) {
            const int s = it % stages;
            const uint32_t ph = (uint32_t)(it / stages) & 1u;
            if (!mbar_wait(&empty[s], ph ^ 1u, WAIT_LIMIT_NS)) {
                ok = false;
                break;
            }
            const TileAhead a = nx_;
            const uint32_t* pb = pre + (it & 1) * PRE_WORDS;
            if (a.t < 0) {
                if (lane == 0) {
                    hdr[s].tile = -1;
                    mbar_arrive(&full[s]);
                }
                break;
            }
            cp_async_wait_all();  // this tile's count and edge values, copied one iteration ago
            __syncwarp();
            const int ncand = min((int)pb[PRE_CNT], LIST_CAP);
            StageHdr& h = hdr[s];
            if (lane == 0) {
                const CUtensorMap* map = tmaps + 2 * a.ii + par;
                unsigned char* dst = smem + s * LY.stage;
                mbar_expect_tx(&full[s], (uint32_t)(QS * LY.bw * (rows + 2) * (int)sizeof(S) + CAND_BYTES * ncand));
                tma_load_3d(dst, map, a.x0 - H, a.y0 - 1, 0, &full[s]);
                if (ncand > 0) {
                    const Cand* lr = ninst <= TI_MAX ? tab[a.ii].lrec[par]
                                                     : static_cast<const Cand*>(insts[a.ii].list_rec[par]);
                    bulk_load(cands + s * LIST_CAP, lr + (long long)a.local * LIST_CAP,
                              (uint32_t)(CAND_BYTES * ncand), &full[s]);
                }
            }
            // the tile's constants, its edge values and its header
            if (ninst <= TI_MAX) {
                if (lane < TI_WORDS)
                    reinterpret_cast<uint4*>(&h.ti)[lane] = reinterpret_cast<const uint4*>(&tab[a.ii])[lane];
            } else if (lane == 0) {
                make_tinst(h.ti, insts[a.ii]);
            }
            if (a.ex) {
                float* ev = edgev + s * 2 * rows * QE;
#pragma unroll
                for (int j = 0; j < (2 * ROWS * QE + 31) / 32; ++j) {
                    const int l = lane + 32 * j;
                    if (l < 2 * rows * QE && ((a.ex >> (l >= rows * QE ? 1 : 0)) & 1)) {
                        const uint32_t w = pb[l];
                        float v;
                        if (sizeof(S) == 2) {
                            const unsigned short hb = (unsigned short)(((a.hsel >> j) & 1) ? (w >> 16) : (w & 0xffffu));
                            v = __half2float(__ushort_as_half(hb)) * a.sload;
                        } else {
                            v = __uint_as_float(w);
                        }
                        ev[l] = v + a.add[j];
                    }
                }
            }
            if (lane == 0) {
                h.tile = a.t;
                h.inst = a.ii;
                h.x0 = a.x0;
                h.y0 = a.y0;
                h.ncand = ncand;
                h.ex = a.ex;
                if (commit && a.np > 0)  // this tile's list of the next step starts empty
                    (ninst <= TI_MAX ? tab[a.ii].lcnt[par ^ 1] : insts[a.ii].list_cnt[par ^ 1])[a.local] = 0;
            }
            __syncwarp();  // the lanes' table copy and edge values are visible to lane 0's arrive
            if (lane == 0) mbar_arrive(&full[s]);
            ++issued;
            // the next tile: its claim has been in flight for a whole tile
            if (lane == 0) {
                c_cur = c_nxt;
                c_nxt = atomicAdd(&tile_ctr[0], 1);
            }
            __syncwarp();  // every lane has read this buffer before it is refilled
            nx_ = ahead(c_cur, (it + 1) & 1);
        }
        cp_async_wait_all();  // no copy of this warp outlives it
        if (!ok) {
            if (lane == 0) atomicOr(insts[0].status, ST_TIMEOUT);
            // let the copies this warp issued land before the block exits
            for (int k = max(0, issued - stages); k < issued; ++k)
                mbar_wait(&full[k % stages], (uint32_t)(k / stages) & 1u, WAIT_LIMIT_NS);
        }
        if (lane == 0) {  // the last block to leave resets the work counter
            __threadfence();
            if (atomicAdd(&tile_ctr[1], 1) == (int)gridDim.x - 1) {
                tile_ctr[0] = 0;
                tile_ctr[1] = 0;
            }
        }
        return;
    }
    // ------------------------------------------------------------- consumers
    const int cw = warp - 1;
    for (int it = 0;; ++it) {
        const int s = it % stages;
        const uint32_t ph = (uint32_t)(it / stages) & 1u;
        if (!mbar_wait(&full[s], ph, WAIT_LIMIT_NS)) {
            if (lane == 0) atomicOr(insts[0].status, ST_TIMEOUT);
            return;
        }
        const int t = hdr[s].tile;
        if (t < 0) return;
        const StageHdr& h = hdr[s];
        const int ncand = h.ncand;
        const Cand* cand = cands + s * LIST_CAP;
        const int nx = h.ti.n[0], ny = h.ti.n[1];
        const float sload = h.ti.sload;
        const CollK ck = make_collk<Q>(CollP{h.ti.keep, h.ti.fpref, h.ti.alpha});
        const int x0 = h.x0, y0 = h.y0;
        const S* stage = reinterpret_cast<const S*>(smem + s * LY.stage);
        const int ex = h.ex;
        const bool free = h.ti.free != 0;
        const TileEnv env{h.ti, h.ti.tot[commit ? par : 2]};
        const float* ev = edgev + s * 2 * rows * QE;
        bool bad = false;
        // FOLD (FP16 storage at tau = 1): the populations stay at the
        // storage scale from the stage to the store (collide2_t1_scaled)
        auto tile_rows = [&](auto fold_tag) {
            constexpr bool FOLD = decltype(fold_tag)::value;
            const float sstore = h.ti.sstore;
            CollK cks = ck;
            if constexpr (FOLD) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    cks.A[i] *= sstore;
                    cks.fA[i] *= sstore;
                    cks.sA[i] *= sstore;
                }
            }
            for (int r = cw; r < rows; r += nc) {
                const int y = y0 + r;
                if (y >= ny) break;
                // every source row lies inside the box (and so in the stage), or beyond
                // a y wall: then the node's own opposite population, staged too,
                // comes back
                const bool lo_y = y < 1, hi_y = y + 1 >= ny;
                const bool rowfast = !(lo_y || hi_y) || !h.ti.per[1];
                const S* rowbase = stage + r * BW + H;
                // element of population q's source row in the stage, relative to rowbase
                auto qoff = [&](int q) { return (q - 1) * SLAB + (1 - L::c(q, 1)) * BW; };
                auto beyond_y = [&](int q) { return L::c(q, 1) > 0 ? lo_y : L::c(q, 1) < 0 && hi_y; };
                S* outrow = static_cast<S*>(const_cast<void*>(h.ti.f[par ^ 1])) + y * h.ti.pitch;
                // two adjacent nodes per lane: packed FP32x2 arithmetic, 8-byte stores
                for (int j = 0; j < TW / 64; ++j) {
                    const int lx = j * 64 + 2 * lane;
                    const int x = x0 + lx;
                    if (x0 + j * 64 >= nx) break;  // ragged tile: nothing left in this row
                    float2 f[QS];
                    if (rowfast) {
#pragma unroll
                        for (int q = 1; q < Q; ++q) {
                            const S* src = rowbase + qoff(q) + lx - L::c(q, 0);
                            if constexpr (FOLD) {
                                if (L::c(q, 0) == 0) f[q - 1] = __half22float2(*reinterpret_cast<const __half2*>(src));
                                else f[q - 1] = make_float2(__half2float(src[0]), __half2float(src[1]));
                            } else {
                                if (L::c(q, 0) == 0) f[q - 1] = smem_pair(src, sload);
                                else
                                    f[q - 1] = make_float2(to_float_scaled(src[0], sload),
                                                           to_float_scaled(src[1], sload));
                            }
                        }
                        if (lo_y || hi_y) {  // bounce-back at the y walls (Eq. 10)
#pragma unroll
                            for (int q = 1; q < Q; ++q) {
                                const int cy = L::c(q, 1);
                                if (!(cy > 0 ? lo_y : cy < 0 && hi_y)) continue;
                                const float wt = __ldg(&insts[h.inst].wterm[1][cy > 0 ? 0 : 1][q]);
                                const float2 v = smem_pair(rowbase + (L::opp(q) - 1) * SLAB + BW + lx, sload);
                                f[q - 1] = make_float2(v.x + wt, v.y + wt);
                                if constexpr (FOLD) f[q - 1] = make_float2(f[q - 1].x * sstore, f[q - 1].y * sstore);
                            }
                        }
                        // the edge nodes' populations from across the x faces (the box
                        // holds zero fill or a neighbour column there); nodes past
                        // nx in a ragged tile are computed but never stored
                        if (ex) {
                            if ((ex & 1) && x == 0) {
                                int k = 0;
#pragma unroll
                                for (int q = 1; q < Q; ++q)
                                    if (L::c(q, 0) == 1) {
                                        const float vv = FOLD ? ev[r * QE + k] * sstore : ev[r * QE + k];
                                        ++k;
                                        if (!beyond_y(q)) f[q - 1].x = vv;
                                    }
                            }
                            const int e = nx - 1 - x;
                            if ((ex & 2) && (e == 0 || e == 1)) {
                                int k = 0;
#pragma unroll
                                for (int q = 1; q < Q; ++q)
                                    if (L::c(q, 0) == -1) {
                                        const float vv = FOLD ? ev[(rows + r) * QE + k] * sstore : ev[(rows + r) * QE + k];
                                        ++k;
                                        if (beyond_y(q)) continue;
                                        if (e == 0) f[q - 1].x = vv;
                                        else f[q - 1].y = vv;
                                    }
                            }
                        }
                    } else {
                        // a row at a periodic y face: every population straight from the
                        // previous buffer (L2 holds it), all loads in flight
                        const S* fin = static_cast<const S*>(h.ti.f[par]);
                        float g[QS];
                        pull_pre_all<Q, S>(insts[h.inst], fin, min(x, nx - 1), y, 0, (int)h.ti.qstride, g);
#pragma unroll
                        for (int q = 0; q < QS; ++q) f[q].x = FOLD ? g[q] * sstore : g[q];
                        pull_pre_all<Q, S>(insts[h.inst], fin, min(x + 1, nx - 1), y, 0, (int)h.ti.qstride, g);
#pragma unroll
                        for (int q = 0; q < QS; ++q) f[q].y = FOLD ? g[q] * sstore : g[q];
                    }
                    bad |= finish_pair<Q, S, FOLD>(env, f, FOLD ? cks : ck, sload, sstore, free, cand, ncand,
                                                   x0 + j * 64, x, y, 0, lane, outrow + x, (int)h.ti.qstride);
                }
            }
        };
        if constexpr (sizeof(S) == 2) {
            if (ck.keep == 0.f) tile_rows(std::true_type{});
            else tile_rows(std::false_type{});
        } else {
            tile_rows(std::false_type{});
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(h.ti.status, ST_DIVERGED);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
    }
}

// ------------------------------------------------------------- host side ---
template <class S, int TW, int ROWS>
static cudaError_t launch_tma_t(const InstDesc* insts, const void* tmaps, const uint16_t* tile_inst,
                                int ntiles, int par, const Shape& sh, int commit, int grid,
                                int* tile_ctr, int stages, int ninst, cudaStream_t st) {
    const TmaLayout LY = tma_layout((int)sizeof(S), TW, ROWS, stages, ninst);
    return launch_dep(k_fluid_tma<S, TW, ROWS>, dim3((unsigned)grid), 32 * (sh.warps + 1), LY.bytes, st, insts,
                      static_cast<const CUtensorMap*>(tmaps), tile_inst, ntiles, par, sh, commit, tile_ctr, stages, ninst);
}

int tma_tile_width() { return 128; }

bool tma_rows_ok(int rows) { return rows == 4 || rows == 8; }

template <class S, int TW, int ROWS>
static int tma_blocks_t(const Shape& sh, int stages, int ninst) {
    const TmaLayout LY = tma_layout((int)sizeof(S), TW, ROWS, stages, ninst);
    auto* const kern = k_fluid_tma<S, TW, ROWS>;
    {
        // the limit belongs to the kernel, not to a context: only raised, so that a
        // context with fewer instances or stages leaves the others' launches valid
        static std::mutex m;
        std::lock_guard<std::mutex> lock(m);
        cudaFuncAttributes at;
        if (cudaFuncGetAttributes(&at, kern) != cudaSuccess) return 0;
        if (at.maxDynamicSharedSizeBytes < LY.bytes &&
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, LY.bytes) != cudaSuccess)
            return 0;
    }
    int nb = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, 32 * (sh.warps + 1), LY.bytes);
    return nb;
}

#define LBM_TMA_DISPATCH(CALL)                              \
    {                                                       \
        if (!fp16 && sh.ty == 4) return CALL(float, 128, 4);  \
        if (!fp16 && sh.ty == 8) return CALL(float, 128, 8);  \
        if (fp16 && sh.ty == 4) return CALL(__half, 128, 4);  \
        if (fp16 && sh.ty == 8) return CALL(__half, 128, 8);  \
    }

int fluid_tma_blocks_per_sm(int fp16, const Shape& sh, int stages, int ninst) {
#define LBM_BLK(SS, TT, RR) tma_blocks_t<SS, TT, RR>(sh, stages, ninst)
    LBM_TMA_DISPATCH(LBM_BLK)
#undef LBM_BLK
    return 0;
}

cudaError_t launch_fluid_tma(int fp16, const InstDesc* insts, const void* tmaps,
                             const uint16_t* tile_inst, int ntiles, int par, const Shape& sh,
                             int commit, int grid, int* tile_ctr, int stages, int ninst, cudaStream_t st) {
#define LBM_LAUNCH(SS, TT, RR)                                                                             \
    launch_tma_t<SS, TT, RR>(insts, tmaps, tile_inst, ntiles, par, sh, commit, grid, tile_ctr, stages, ninst, st)
    LBM_TMA_DISPATCH(LBM_LAUNCH)
#undef LBM_LAUNCH
    return cudaErrorInvalidValue;
}

}  // namespace lbmpen
