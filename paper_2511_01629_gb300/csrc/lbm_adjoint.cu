// Discrete adjoint of the penalized LBM step (reverse mode, hand-written).
//
// The forward step n maps the post-collision populations g^{n-1} and the
// particle state P^n = (X^n, U^{n-1}, W^{n-1}, theta^n, A^n) to g^n and P^{n+1}
// (Eqs. 9-17, 22 and Algorithm 1).  With the solid indicator held fixed (it
// is piecewise constant in X, Eq. 9, so its derivative vanishes almost
// everywhere) every stage is differentiable, and the backward sweep applies
// the transposed Jacobians in reverse order:
//
//   k_adj_particles  Algorithm 1 (sub-steps with the collision forces of
//                    Eqs. 19-21, A^{n+1}, theta^{n+1}) and the projection of
//                    Eq. 22 transposed, FP64, one block per instance;
//   k_adj_fluid      the fused collide (Eqs. 10, 13-17) transposed per node
//                    and streaming transposed: the adjoint of f^{n+1}_q at
//                    x + c_q is pulled to x (or the opposite population at x
//                    where x + c_q lies beyond a wall), FP32, one block per tile.
//
// The adjoint fluid kernel reads the populations entering step n (recorded
// by the recomputation of a checkpointed segment) and recomputes the node's
// forward state (u, p, feq, Pi_neq) from them; it writes the adjoint of the
// pre-collision populations of step n and adds, per particle, the sums of the
// adjoint acceleration and of the alpha derivative over the particle's nodes.
#include "lbm_common.cuh"

namespace lbmpen {

namespace {

// ----------------------------------------------------------- node adjoint --
// Two nodes (packed FP32x2, one per half): given the pre-collision populations
// f (q = 1..Q-1), the local acceleration a and lam = d J / d f*, replace lam by
// d J / d f and return ab = d J / d a and alb = d J / d alpha.  ubp is the part of d J / d u that
// comes from the rigid-body projection (zero on fluid nodes).  The forward
// map is the one of collide2():
//   g_q = keep f_q + omk A_q E_q + fA_q G_q + chi S_q,
//   E_q = p - u.u/2 + c.u + 1.5 (c.u)^2,   G_q = c.a (1 + 3 c.u) - u.a,
//   S_q = 1.5 alpha A_q (c_q^T Pi c_q - tr(Pi)/3),  Pi = sum_q (f_q - A_q E_q) c_q c_q^T,
//   u = m + a/2,  p = (s - kuu u.u) / sum A.
// Opposite velocities share c.u, c.a and c c^T, so with Eb = omk A lam, Gb = fA lam
// (s, d: the pair's sum and difference) a pair adds to d J / d u along c
//   Eb_d + 3 c.u Eb_s + 3 c.a Gb_s
// and to d J / d a along c  Gb_d + 3 c.u Gb_s.
// FREE: no node of the warp is solid and there is no body force, so a = 0 and
// nothing asks for ab or alb: the forcing and penalty terms drop out.
template <int Q, bool FREE>
struct NodeAdj {
    using L = Lat<Q>;
    static constexpr int D = L::D;
    static constexpr int QS = Q - 1;

    // r + s * c for one component of c
    static __device__ __forceinline__ float2 along(float2 r, float2 v, int c) {
        return c == 0 ? r : c > 0 ? add2(r, v) : sub2(r, v);
    }

    // per-pair accumulations of bb, ub, uab, ax
    template <int q>
    static __device__ __forceinline__ void pairs(const float2* lam, const float2* u, const float2* a, const CollK& k,
                                                 const float2* nuA, float2& bb, float2* ub, float2& uab, float2* ax) {
        if constexpr (q < Q) {
            if constexpr (pair_head<Q>(q)) {
                constexpr int qo = L::opp(q);
                constexpr int cls = (Q == 9 ? q >= 5 : q >= 7) ? 1 : 0;
                const float2 ls = add2(lam[q - 1], lam[qo - 1]), ld = sub2(lam[q - 1], lam[qo - 1]);
                const float2 cu3 = mul2(bc2(3.0f), cdot2<Q, q>(u));
                const float oa = k.omk * k.A[cls];
                float2 es = mul2(bc2(oa), ls);
                if constexpr (!FREE) es = fma2(bc2(-2.0f), nuA[q - 1], es);  // both velocities of the pair
                float2 w = fma2(cu3, es, mul2(bc2(oa), ld));
                if constexpr (!FREE) {
                    const float2 gs = mul2(bc2(k.fA[cls]), ls);
                    w = fma2(mul2(bc2(3.0f), cdot2<Q, q>(a)), gs, w);
                    const float2 v = fma2(cu3, gs, mul2(bc2(k.fA[cls]), ld));
                    uab = sub2(uab, gs);
#pragma unroll
                    for (int d = 0; d < D; ++d) ax[d] = along(ax[d], v, L::c(q, d));
                }
                bb = add2(bb, es);
#pragma unroll
                for (int d = 0; d < D; ++d) ub[d] = along(ub[d], w, L::c(q, d));
            }
            pairs<q + 1>(lam, u, a, k, nuA, bb, ub, uab, ax);
        }
    }
    template <int q>
    static __device__ __forceinline__ void finish(float2* lam, const float2* ub, float2 sb, const float2* nu, bool keep,
                                                  const CollK& k) {
        if constexpr (q < Q) {
            if constexpr (pair_head<Q>(q)) {
                constexpr int qo = L::opp(q);
                const float2 cu = cdot2<Q, q>(ub);
                float2 s = sb;
                if constexpr (!FREE) s = add2(sb, nu[q - 1]);
                float2 r = add2(s, cu), o = sub2(s, cu);
                if (keep) {
                    r = fma2(bc2(k.keep), lam[q - 1], r);
                    o = fma2(bc2(k.keep), lam[qo - 1], o);
                }
                lam[q - 1] = r;
                lam[qo - 1] = o;
            }
            finish<q + 1>(lam, ub, sb, nu, keep, k);
        }
    }

    // the penalty of the solid nodes: nu_q = c_q^T Pb c_q (at the pair's head), A_q nu_q and alb
    template <int q>
    static __device__ __forceinline__ void pen_in(const float2* lam, const CollK& k, float2 m, float2* Pb, float2& tr) {
        if constexpr (q < Q) {
            if constexpr (pair_head<Q>(q)) {
                constexpr int qo = L::opp(q);
                constexpr int cls = (Q == 9 ? q >= 5 : q >= 7) ? 1 : 0;
                const float2 w = mul2(mul2(bc2(k.sA[cls]), m), add2(lam[q - 1], lam[qo - 1]));
                tr = fma2(w, bc2(-1.0f / 3.0f), tr);
                constexpr int cx = L::c(q, 0), cy = L::c(q, 1), cz = L::c(q, 2);
                Pb[0] = along(Pb[0], w, cx * cx);
                Pb[1] = along(Pb[1], w, cy * cy);
                Pb[2] = along(Pb[2], w, cz * cz);
                Pb[3] = along(Pb[3], w, cx * cy);
                Pb[4] = along(Pb[4], w, cx * cz);
                Pb[5] = along(Pb[5], w, cy * cz);
            }
            pen_in<q + 1>(lam, k, m, Pb, tr);
        }
    }
    template <int q>
    static __device__ __forceinline__ void pen_out(const float2* lam, const CollK& k, const float2* P, float2 trP,
                                                   const float2* Pb, float2* nu, float2* nuA, float2& al) {
        if constexpr (q < Q) {
            if constexpr (pair_head<Q>(q)) {
                constexpr int qo = L::opp(q);
                constexpr int cls = (Q == 9 ? q >= 5 : q >= 7) ? 1 : 0;
                al = fma2(mul2(bc2(1.5f * k.A[cls]), add2(lam[q - 1], lam[qo - 1])), sub2(pcc2<Q, q>(P), trP), al);
                nu[q - 1] = pcc2<Q, q>(Pb);
                nuA[q - 1] = mul2(bc2(k.A[cls]), nu[q - 1]);
            }
            pen_out<q + 1>(lam, k, P, trP, Pb, nu, nuA, al);
        }
    }

    static __device__ __forceinline__ void run(const float2* f, const float2* a, float2* lam, bool solid0, bool solid1,
                                               const float2* ubp, const CollK& k, float2* ab, float2* alb) {
        constexpr float inv_sa = (float)(1.0 / L::SUMA);
        constexpr float kuu = (float)(1.5 - 0.5 * L::SUMA);
        float2 s, u[3];
        moments2<Q>(f, s, u);
        if constexpr (!FREE)
#pragma unroll
            for (int d = 0; d < D; ++d) u[d] = fma2(bc2(0.5f), a[d], u[d]);
        float2 ub[3] = {bc2(0.f), bc2(0.f), bc2(0.f)}, ax[3] = {bc2(0.f), bc2(0.f), bc2(0.f)};
        float2 bb = bc2(0.f), uab = bc2(0.f), nu[FREE ? 1 : QS], nuA[FREE ? 1 : QS];
        if constexpr (!FREE) {
            float2 uu = mul2(u[0], u[0]);
#pragma unroll
            for (int d = 1; d < D; ++d) uu = fma2(u[d], u[d], uu);
            const float2 p = mul2(fma2(bc2(-kuu), uu, s), bc2(inv_sa));
            const float2 base = fma2(bc2(-0.5f), uu, p);
            float2 P[6], Pb[6], tr = bc2(0.f), al = bc2(0.f);
            pi_neq2<Q>(f, u, base, P);  // xx yy zz xy xz yz
            const float2 trP = mul2(add2(add2(P[0], P[1]), P[2]), bc2(1.0f / 3.0f));
#pragma unroll
            for (int i = 0; i < 6; ++i) Pb[i] = bc2(0.f);
            pen_in<1>(lam, k, make_float2(solid0 ? 1.f : 0.f, solid1 ? 1.f : 0.f), Pb, tr);
#pragma unroll
            for (int d = 0; d < D; ++d) Pb[d] = add2(Pb[d], tr);
            if (D == 2) Pb[2] = tr;  // (no velocity reads it)
            pen_out<1>(lam, k, P, trP, Pb, nu, nuA, al);
            *alb = al;
#pragma unroll
            for (int d = 0; d < D; ++d) ub[d] = ubp[d];
        }
        pairs<1>(lam, u, a, k, nuA, bb, ub, uab, ax);
        // base = p - u.u/2, p = (s - kuu u.u) / sum A
        const float2 sb = mul2(bb, bc2(inv_sa));
        const float2 uub2 = fma2(bc2(-2.0f * kuu), sb, mul2(bc2(-1.0f), bb));  // 2 d J / d (u.u)
#pragma unroll
        for (int d = 0; d < D; ++d) {
            if constexpr (!FREE) {
                ub[d] = fma2(uab, a[d], ub[d]);
                ax[d] = fma2(uab, u[d], ax[d]);
            }
            ub[d] = fma2(uub2, u[d], ub[d]);
            if constexpr (!FREE) ab[d] = fma2(bc2(0.5f), ub[d], ax[d]);
        }
        // u = m + a/2 with m = sum_q f_q c_q, s = sum_q f_q
        if (k.keep != 0.f) finish<1>(lam, ub, sb, nu, true, k);
        else finish<1>(lam, ub, sb, nu, false, k);
    }
};

// Transposed streaming: the adjoint of f*_q at x is the adjoint of f_q at
// x + c_q (wrapped on periodic axes), or of f_opp(q) at x when x + c_q lies
// beyond a wall (the population bounced back at x).
template <int Q, int q>
__device__ __forceinline__ float pull_lam_any(const InstDesc& in, const float* __restrict__ lam, int x, int y, int z,
                                              long long qs) {
    using L = Lat<Q>;
    constexpr int c[3] = {L::c(q, 0), L::c(q, 1), L::c(q, 2)};
    int dst[3] = {x + c[0], y + c[1], z + c[2]};
    bool wall = false;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (c[d] == 0) continue;
        const bool out = dst[d] < 0 || dst[d] >= in.n[d];
        if (out && in.periodic[d]) dst[d] += dst[d] < 0 ? in.n[d] : -in.n[d];
        else if (out) wall = true;
    }
    const int node = (z * in.n[1] + y) * in.pitch + x;
    return __ldg(wall ? pop(lam, L::opp(q), qs) + node : pop(lam, q, qs) + ((dst[2] * in.n[1] + dst[1]) * in.pitch + dst[0]));
}
template <int Q, int q = 1>
__device__ __forceinline__ void pull_lam_all(const InstDesc& in, const float* ls, int x, int y, int z, long long qs,
                                             float* l) {
    if constexpr (q < Q) {
        l[q - 1] = pull_lam_any<Q, q>(in, ls, x, y, z, qs);
        pull_lam_all<Q, q + 1>(in, ls, x, y, z, qs, l);
    }
}

// The adjoint entering nodes x, x + 1 (x even) of a row whose y and z
// neighbours lie inside the box (pull_pair's transpose; EDGE as there).
template <int Q, bool EDGE>
__device__ __forceinline__ void pull_lam_pair(const InstDesc& in, const float* __restrict__ ls, int x, int y, int z,
                                              float2* l) {
    using L = Lat<Q>;
    const int nx = in.n[0], pitch = in.pitch, zs = in.n[1] * pitch;
    const long long qs = in.qstride;
    const int own = z * zs + y * pitch, xl = EDGE ? min(x, (nx - 1) & ~1) : x;
    auto row_of = [&](int q) { return own + L::c(q, 2) * zs + L::c(q, 1) * pitch; };  // within population q
#pragma unroll
    for (int q = 1; q < Q; ++q) {
        const int cx = L::c(q, 0), at = row_of(q) + xl;
        const float* lq = pop(ls, q, qs);
        if (cx == 0) l[q - 1] = __ldg(reinterpret_cast<const float2*>(lq + at));
        else l[q - 1] = make_float2(__ldg(lq + (at + cx)), __ldg(lq + (at + 1 + cx)));
    }
    if constexpr (EDGE) {
        const bool wall = !in.periodic[0], lo = x == 0, hi0 = x == nx - 1, hi1 = x + 1 == nx - 1;
        const long long wq = wall ? qs : 0;  // see pull_pair
        float v[Q];
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const int cx = L::c(q, 0);
            if (cx == 0) continue;
            const float* from = pop(ls, q, qs) + (L::opp(q) - q) * wq +
                                (wall ? own + (cx < 0 ? 0 : nx - 1) : row_of(q) + (cx < 0 ? nx - 1 : 0));
            v[q] = 0.f;
            if (cx < 0 ? lo : hi0 || hi1) v[q] = __ldg(from);
        }
#pragma unroll
        for (int q = 1; q < Q; ++q) {
            const int cx = L::c(q, 0);
            if (cx == 0) continue;
            if (cx < 0 ? lo : hi0) l[q - 1].x = v[q];
            if (cx > 0 && hi1) l[q - 1].y = v[q];
        }
    }
}

}  // namespace

// ------------------------------------------------------------ fluid sweep --
constexpr int ADJ_WARPS = 4;   // warps per block
constexpr int ADJ_BLOCKS = 5;  // resident blocks per SM in 2D (launch bounds)

// lam_mode: 0 = pull the adjoint of step n + 1, 1 = read a field seed [Q][N]
// (the adjoint of the final post-collision populations), 2 = zero.
// A block takes a tile of the forward kernel's shape (the candidate lists are
// per tile) or a part of one, a warp a 64-node segment of a row at a time; a
// lane takes two adjacent nodes, all of their populations and adjoints in
// flight before the first is used (8-byte loads where c_x = 0), and stores
// 8-byte pairs.  The candidates are read where they are: copying them to shared
// memory behind a barrier first cost one box of 400 x 1600 11 % of its backward
// pass.  HBM-bound: two reads and a write per population.  16 boxes of 400 x
// 1600, FP32: about 285 us a step before (one node per lane, scalar arithmetic
// over all velocities, the candidates before the loads), 212 now (983 MB, 4.6
// TB/s; what is left is load latency, at 20 warps per SM).
// Warps that stride over all segments (760 blocks) took 22.4 ms for the 16 boxes.
template <int Q, class S>
__global__ void __launch_bounds__(32 * ADJ_WARPS, Q == 9 ? ADJ_BLOCKS : 3) k_adj_fluid(
    const InstDesc* __restrict__ insts, const AdjFluid* __restrict__ afs, const uint16_t* __restrict__ tile_inst, int ninst,
    int lam_mode, Shape sh) {
    using L = Lat<Q>;
    constexpr int D = L::D;
    constexpr int QS = Q - 1;
    const int lane = threadIdx.x & 31;
    const int tw = sh.tw, rows = sh.ty * sh.tz, segs = (tw + 63) >> 6;
    const int t = blockIdx.x;
    const int ii = ninst > 1 ? (int)tile_inst[t] : 0;
    const InstDesc& in = insts[ii];
    const AdjFluid& af = afs[ii];
    const int local = t - in.tile0;
    const int ntx = in.ntile[0], nty = in.ntile[1];
    const int rest = local / ntx;
    const int x0 = (local - rest * ntx) * tw, y0 = (rest % nty) * sh.ty, z0 = (rest / nty) * sh.tz;
    const int nx = in.n[0], ny = in.n[1], nz = in.n[2];
    const int pitch = in.pitch;
    const long long qs = in.qstride;
    const S* __restrict__ fin = static_cast<const S*>(af.fin);
    const float* __restrict__ lsrc = af.lam_src;
    float* __restrict__ ldst = af.lam_dst;
    const int ncand = in.np > 0 ? min(af.lcnt[local], LIST_CAP) : 0;
    const Cand* cand = static_cast<const Cand*>(af.lrec) + (long long)local * LIST_CAP;
    Geo geo = make_geo(in);
    geo.prec = af.prec;
    const CollK ck = make_collk<Q>(make_collp(in));
    const float gd[3] = {in.gdrive[0], in.gdrive[1], in.gdrive[2]};
    const bool free = gd[0] == 0.f && gd[1] == 0.f && gd[2] == 0.f;
    for (int rs = (threadIdx.x >> 5) + ADJ_WARPS * blockIdx.y; rs < rows * segs; rs += ADJ_WARPS * gridDim.y) {
        const int r = rs / segs, sg = rs - r * segs;
        const int y = y0 + r % sh.ty, z = z0 + r / sh.ty, xb = x0 + 64 * sg;
        if (xb >= nx || y >= ny || z >= nz) continue;  // warp-uniform: beyond the box
        const int x = xb + 2 * lane, wseg = min(64, min(tw - 64 * sg, nx - xb));
        float2 f[QS], lam[QS];
        const int xc0 = min(x, nx - 1), xc1 = min(x + 1, nx - 1);  // lanes past the row read valid nodes
        const bool row_in = y >= 1 && y + 1 < ny && (D == 2 || (z >= 1 && z + 1 < nz));
        const bool edge = xb == 0 || xb + 64 >= nx;
        float g0[QS], g1[QS];
        if (row_in) {
            if (edge) pull_pair<Q, S, true>(in, fin, qs, x, y, z, f);
            else pull_pair<Q, S, false>(in, fin, qs, x, y, z, f);
        } else {
            pull_pre_all<Q, S>(in, fin, xc0, y, z, qs, g0);
            pull_pre_all<Q, S>(in, fin, xc1, y, z, qs, g1);
#pragma unroll
            for (int q = 0; q < QS; ++q) f[q] = make_float2(g0[q], g1[q]);
        }
        if (lam_mode == 0) {
            if (row_in) {
                if (edge) pull_lam_pair<Q, true>(in, lsrc, x, y, z, lam);
                else pull_lam_pair<Q, false>(in, lsrc, x, y, z, lam);
            } else {
                pull_lam_all<Q>(in, lsrc, xc0, y, z, qs, g0);
                pull_lam_all<Q>(in, lsrc, xc1, y, z, qs, g1);
#pragma unroll
                for (int q = 0; q < QS; ++q) lam[q] = make_float2(g0[q], g1[q]);
            }
        } else if (lam_mode == 1) {
            const long long N = (long long)nx * ny * nz, nd = ((long long)z * ny + y) * nx;
#pragma unroll
            for (int q = 1; q < Q; ++q)
                lam[q - 1] = make_float2(__ldg(lsrc + (long long)q * N + nd + xc0), __ldg(lsrc + (long long)q * N + nd + xc1));
        } else {
#pragma unroll
            for (int q = 0; q < QS; ++q) lam[q] = bc2(0.f);
        }
        const bool v0 = 2 * lane < wseg, v1 = 2 * lane + 1 < wseg;
        const int xyz0[3] = {x, y, z}, xyz1[3] = {x + 1, y, z};
        int own0 = -1, own1 = -1, sl0 = -1, sl1 = -1;
        if (ncand > 32) {
            own0 = owner_of<D>(geo, cand, ncand, xyz0, &sl0);
            own1 = owner_of<D>(geo, cand, ncand, xyz1, &sl1);
        } else if (ncand > 0) {
            const unsigned act = segment_candidates<D>(geo, cand, ncand, xb, y, z, 64, lane);
            if (act) {
                own0 = owner_masked<D>(geo, cand, act, xyz0, &sl0);
                own1 = owner_masked<D>(geo, cand, act, xyz1, &sl1);
            }
        }
        if (!v0) own0 = -1;
        if (!v1) own1 = -1;
        const unsigned any = __ballot_sync(0xffffffffu, own0 >= 0 || own1 >= 0);
        float2 ab[3] = {bc2(0.f), bc2(0.f), bc2(0.f)}, alb = bc2(0.f);
        if (free && !any) {
            NodeAdj<Q, true>::run(f, nullptr, lam, false, false, nullptr, ck, nullptr, nullptr);
        } else {
            float2 a[3], ubp[3];
            float an[2][3], un[2][3];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int own = h ? own1 : own0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    an[h][d] = gd[d];
                    un[h][d] = 0.f;
                }
                if (own >= 0) {
                    const Cand& cd = cand[h ? sl1 : sl0];
                    float rr[3] = {0.f, 0.f, 0.f};
#pragma unroll
                    for (int d = 0; d < D; ++d)
                        rr[d] = (float)wrap_int((h ? xyz1 : xyz0)[d] - cd.ref[d], in.n[d], in.periodic[d]) - cd.frac[d];
                    const float* cf = af.coef + 8LL * own;
#pragma unroll
                    for (int d = 0; d < 3; ++d) an[h][d] += cd.a[d];
                    // d U / d u = 1 / count, d W / d u: (I^-1 dW) x r
                    un[h][0] = cf[0] + (cf[4] * rr[2] - cf[5] * rr[1]);
                    un[h][1] = cf[1] + (cf[5] * rr[0] - cf[3] * rr[2]);
                    un[h][2] = D == 3 ? cf[2] + (cf[3] * rr[1] - cf[4] * rr[0]) : 0.f;
                }
            }
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                a[d] = make_float2(an[0][d], an[1][d]);
                ubp[d] = make_float2(un[0][d], un[1][d]);
            }
            NodeAdj<Q, false>::run(f, a, lam, own0 >= 0, own1 >= 0, ubp, ck, ab, &alb);
        }
        float* out = ldst + ((z * ny + y) * pitch + x);
        if (v1) {
#pragma unroll
            for (int q = 1; q < Q; ++q) *reinterpret_cast<float2*>(pop(out, q, qs)) = lam[q - 1];
        } else if (v0) {
#pragma unroll
            for (int q = 1; q < Q; ++q) *pop(out, q, qs) = lam[q - 1].x;
        }
        // per-particle sums of the adjoint acceleration and alpha derivative
        if (!any) continue;
        for (;;) {  // lanes 0..3 add the four sums
            const unsigned pend = __ballot_sync(0xffffffffu, own0 >= 0 || own1 >= 0);
            if (!pend) break;
            const int leader = __ffs(pend) - 1;
            const int p = __shfl_sync(0xffffffffu, own0 >= 0 ? own0 : own1, leader);
            const bool m0 = own0 == p, m1 = own1 == p;
            float v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float2 s = k < 3 ? ab[k] : alb;
                v[k] = (m0 ? s.x : 0.f) + (m1 ? s.y : 0.f);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k < D || k == 3) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
            if (lane < 4 && (lane < D || lane == 3))
                atomicAdd(af.Abar + 4LL * p + lane, (double)(lane == 0 ? v[0] : lane == 1 ? v[1] : lane == 2 ? v[2] : v[3]));
            if (m0) own0 = -1;
            if (m1) own1 = -1;
        }
    }
}

// Adjoint of the initial post-collision populations (transposed streaming of
// the adjoint of step 0), written as [Q][N] with the rest population zero.
template <int Q>
__global__ void k_adj_pull_out(const InstDesc* __restrict__ insts, int inst, const float* __restrict__ lam,
                               float* __restrict__ out) {
    const InstDesc& in = insts[inst];
    const long long N = (long long)in.n[0] * in.n[1] * in.n[2];
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    const int x = (int)(i % in.n[0]), y = (int)((i / in.n[0]) % in.n[1]),
              z = (int)(i / ((long long)in.n[0] * in.n[1]));
    float v[Q - 1];
    pull_lam_all<Q>(in, lam, x, y, z, in.qstride, v);
    out[i] = 0.f;
#pragma unroll
    for (int q = 1; q < Q; ++q) out[(long long)q * N + i] = v[q - 1];
}

// --------------------------------------------------------- particle sweep --
namespace {

// Whether a particle at coordinate Y (radius R) along wall axis d can be within
// the wall range R + delta/2 of either plane -1/2, n - 1/2: an FP32 test with
// a margin (wall_reach, the forward kernel's filter), so that particles far from the
// walls skip the FP64 range tests, whose outcome it cannot change.
__device__ __forceinline__ bool wall_near(const InstDesc& in, int d, double Y, double R) {
    const float reach = wall_reach(in, d, R);
    const float yf = (float)Y;
    return !(yf + 0.5f > reach && (float)in.n[d] - 0.5f - yf > reach);
}

// Difference of particles i and j at positions Y (the lattice's minimum image).
__device__ __forceinline__ void pair_diff(const InstDesc& in, int D, const double* Y, int i, int j, double* dv) {
    for (int d = 0; d < 3; ++d) dv[d] = 0.0;
    for (int d = 0; d < D; ++d) {
        double x = Y[3 * i + d] - Y[3 * j + d];
        if (in.periodic[d]) {
            const double half = 0.5 * in.n[d];
            if (x > half) x -= in.n[d];
            else if (x < -half) x += in.n[d];
        }
        dv[d] = x;
    }
}

// Component c of the collision force on particle i per unit C (Eqs. 19-21 with
// C = 1): pairs with the lattice's minimum image, and mirror images across
// wall planes.
__device__ double unit_force(const InstDesc& in, int D, const double* Y, int i, int c) {
    double G = 0.0;
    const double idl = in.pconst[PCONST_N * i + PC_INVDELTA];
    for (int j = 0; j < in.np; ++j) {
        if (j == i) continue;
        double dv[3];
        pair_diff(in, D, Y, i, j, dv);
        const double range = in.R[i] + in.R[j] + in.delta;
        const double d2 = dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2];
        if (d2 > range * range) continue;
        const double s = (range - sqrt(d2)) * idl;
        G += dv[c] * s * s * in.inv_eps_p;
    }
    if (c < D && !in.periodic[c] && wall_near(in, c, Y[3 * i + c], in.R[i])) {
        const double walls[2] = {-0.5, in.n[c] - 0.5};
        for (int face = 0; face < 2; ++face) {
            const double diff = 2.0 * (Y[3 * i + c] - walls[face]);
            const double range = 2.0 * in.R[i] + in.delta;
            if (fabs(diff) <= range) {
                const double s = (range - fabs(diff)) * idl;
                G += diff * s * s * in.inv_eps_w;
            }
        }
    }
    return G;
}

// Transposed Jacobian of the collision forces at positions Y applied to
// their adjoint v: component c of the adjoint of the position of particle m.  With
// F_i = k_i sum_j phi(d_ij), phi(d) = d s^2, s = (range - |d|)/delta and
// phi'(d) = s^2 1 - (2 s / (delta |d|)) d d^T (even in d):
//   Yb_m = sum_j phi'(d_mj) (k_m v_m - k_j v_j) + walls 2 kw_m psi'(diff) v_m.
__device__ double force_jt(const InstDesc& in, int D, const double* Y, const double* v, int m, int c) {
    const double idl = in.pconst[PCONST_N * m + PC_INVDELTA];
    const double km = in.pconst[PCONST_N * m + PC_CPAIR];  // C_m / eps_p
    double acc = 0.0;
    for (int j = 0; j < in.np; ++j) {
        if (j == m) continue;
        double dv[3];
        pair_diff(in, D, Y, m, j, dv);
        const double range = in.R[m] + in.R[j] + in.delta;
        const double d2 = dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2];
        if (d2 > range * range || d2 == 0.0) continue;
        const double dist = sqrt(d2);
        const double s = (range - dist) * idl;
        const double kj = in.pconst[PCONST_N * j + PC_CPAIR];
        double w[3];
        for (int d = 0; d < 3; ++d) w[d] = km * v[3 * m + d] - kj * v[3 * j + d];
        const double dw = dv[0] * w[0] + dv[1] * w[1] + dv[2] * w[2];
        const double g = 2.0 * s * idl * rcp64(dist);
        acc += s * s * w[c] - g * dv[c] * dw;
    }
    if (c < D && !in.periodic[c] && wall_near(in, c, Y[3 * m + c], in.R[m])) {
        const double kw = in.pconst[PCONST_N * m + PC_CWALL];  // C_m / eps_w
        const double walls[2] = {-0.5, in.n[c] - 0.5};
        for (int face = 0; face < 2; ++face) {
            const double diff = 2.0 * (Y[3 * m + c] - walls[face]);
            const double range = 2.0 * in.R[m] + in.delta;
            if (fabs(diff) <= range) {
                const double s = (range - fabs(diff)) * idl;
                acc += 2.0 * kw * (s * s - 2.0 * s * fabs(diff) * idl) * v[3 * m + c];
            }
        }
    }
    return acc;
}

}  // namespace

// Backward of the particle part of step n for every instance (block = instance).
// An FP64 instruction takes its pipe ~64 cycles whether one lane or 32 are
// active, so a lane takes one component of one particle (a serial loop over
// the components cost three times the chain), and the scratch of the sub-steps
// lies in shared memory where it fits (each of its round trips through L2 was
// a wait of its own).  Bound by that chain: 13.3 us before on one particle.
constexpr int ADJ_SCR = 2048;  // doubles of shared scratch: 64 particles at K = 1
template <int D>
__global__ void __launch_bounds__(128) k_adj_particles(const InstDesc* __restrict__ insts,
                                                       const AdjPart* __restrict__ steps,
                                                       const AdjBufs* __restrict__ bufs) {
    const int ii = blockIdx.x;
    __shared__ __align__(16) InstDesc sdesc;
    __shared__ double scr[ADJ_SCR];
    const AdjPart sp = steps[ii];
    const AdjBufs b = bufs[ii];
    stage_desc(&sdesc, insts[ii]);
    const InstDesc& in = sdesc;
    const int np = in.np;
    if (np == 0) return;
    const int K = in.K, n3 = 3 * np;
    const double h = in.hK;
    const double gC = in.rho_f * in.gmag;
    const int tid = threadIdx.x, nt = blockDim.x;
    double* q = adj_scratch(np, K) <= ADJ_SCR ? scr : b.scratch;
    double* const Xk = q;                 // [K+1][np][3] sub-step positions
    double* const Xs = Xk + (K + 1) * n3;  // [K][np][3] predicted positions
    double* const Gs = Xs + K * n3;       // [K][np][3] unit forces at both
    double* const Ubar = Gs + K * n3;     // (U^n + U^{n-1}) / 2
    double* const Xkb = Ubar + n3;        // adjoint of the current sub-step position
    double* const v = Xkb + n3;           // adjoint of the sub-step force sum
    double* const Ubb = v + n3;           // adjoint of Ubar
    double* const Wnb = Ubb + n3;         // adjoint of W^n
    double* const cc = Wnb + n3;          // h^2 / (4 M)
    if (tid < np) asm volatile("prefetch.global.L1 [%0];" ::"l"(sp.geo + (long long)NPV * tid));
    // 1. fold the fluid sums of step n + 1 into the adjoint of A^{n+1}, of
    //    the density ratios (a = (1 - 1/ratio) g + A on solid nodes) and of alpha
    double al = 0.0;
    for (int e = tid; e < n3; e += nt) {
        const int p = e / 3, d = e - 3 * p;
        const double Ap = b.Ab[e] + b.Abar[4 * p + d];
        const double xb = b.Xb[e], tb = b.Tb[e], wb = b.Wb[e];
        const double un = sp.st1[16 * p + 3 + d], uo = sp.st0[16 * p + 3 + d], x0 = sp.st0[16 * p + d];
        const double irs = in.pconst[PCONST_N * p + PC_INVRHOS], cnt = sp.st1[16 * p + 15];
        if (d == 0) {
            double gsum = 0.0;
            for (int k = 0; k < 3; ++k) gsum += b.Abar[4 * p + k] * (double)in.ggrav[k];
            al += b.Abar[4 * p + 3];
            const double iratio = irs * in.rho_f;
            b.rb[p] += gsum * iratio * iratio;
        }
        // state after step n: X' = Xk_K (wrapped), U' = U^n, W' = W^n,
        // theta' = theta + (W^n + W)/2, A' = 2 (Xk_K - X - Ubar)
        b.Ab[e] = 0.0;
        Xkb[e] = xb + 2.0 * Ap;
        b.Xb[e] = -2.0 * Ap;
        Ubb[e] = -2.0 * Ap;
        Wnb[e] = wb + 0.5 * tb;  // adjoint of W^n
        b.Wb[e] = 0.5 * tb;      // adjoint of W^{n-1}
        Ubar[e] = 0.5 * (un + uo);
        Xk[e] = x0;
        cc[e] = 0.25 * h * h * irs * rcp64(cnt);
    }
    if (al != 0.0) atomicAdd(b.alpha_b, al);
    __syncthreads();
    for (int k = tid; k < 4 * np; k += nt) b.Abar[k] = 0.0;
    // 2. forward sub-steps of Algorithm 1 (positions and unit forces)
    for (int j = 1; j <= K; ++j) {
        const double* Xp = Xk + (j - 1) * n3;
        double* X1 = Xs + (j - 1) * n3;
        for (int e = tid; e < n3; e += nt) X1[e] = Xp[e] + h * Ubar[e];
        __syncthreads();
        for (int e = tid; e < n3; e += nt) {
            const int p = e / 3, d = e - 3 * p;
            const double G = unit_force(in, D, Xp, p, d) + unit_force(in, D, X1, p, d);
            const double Cp = (in.ratio[p] - 1.0) * gC;
            Gs[(j - 1) * n3 + e] = G;
            Xk[j * n3 + e] = X1[e] + cc[e] * Cp * G;
        }
        __syncthreads();
    }
    // 3. reverse sub-steps: Xk_j = Xs_j + c (F1(Xk_{j-1}) + F2(Xs_j)), Xs_j = Xk_{j-1} + h Ubar
    for (int j = K; j >= 1; --j) {
        for (int e = tid; e < n3; e += nt) {
            const int p = e / 3, d = e - 3 * p;
            v[e] = cc[e] * Xkb[e];
            if (d == 0) {
                const double Cp = (in.ratio[p] - 1.0) * gC;
                const double iratio = in.pconst[PCONST_N * p + PC_INVRHOS] * in.rho_f, c = cc[e];
                double rbp = 0.0;  // d c / d ratio = -c / ratio, d C / d ratio = rho_f |g|
                for (int k = 0; k < 3; ++k) {
                    const double g = Gs[(j - 1) * n3 + e + k];
                    if (g != 0.0) rbp += Xkb[e + k] * (-c * iratio * Cp * g + c * gC * g);
                }
                b.rb[p] += rbp;
            }
        }
        __syncthreads();
        for (int e = tid; e < n3; e += nt) {
            const int p = e / 3, d = e - 3 * p;
            const double xsb = Xkb[e] + force_jt(in, D, Xs + (j - 1) * n3, v, p, d);
            Ubb[e] += h * xsb;
            Xkb[e] = xsb + force_jt(in, D, Xk + (j - 1) * n3, v, p, d);
        }
        __syncthreads();
    }
    // 4. Ubar = (U^n + U^{n-1})/2, the projection (Eq. 22) and the outputs
    for (int e = tid; e < n3; e += nt) {
        const int p = e / 3, d = e - 3 * p;
        const double* g = sp.geo + (long long)NPV * p;
        const double icnt = rcp64(g[0]);
        const double Unb = b.Ub[e] + 0.5 * Ubb[e];
        double Wb[3], W[3], Su[3], Sr[3];
        for (int k = 0; k < 3; ++k) {
            Wb[k] = Wnb[3 * p + k];
            W[k] = sp.st1[16 * p + 6 + k];
            Su[k] = g[10 + k];
            Sr[k] = g[1 + k];
        }
        double xb = b.Xb[e] + Xkb[e], mu[3] = {0, 0, 0}, t = 0.0;
        // d W / d X through r = x - X: mu x Su + 2 (mu.W) Sr - mu (Sr.W) - W (mu.Sr)
        if (D == 2) {  // mu and W along z, Su and Sr in the plane
            mu[2] = Wb[2] * rcp64(g[4] + g[5]);
            t = (d == 0 ? -mu[2] * Su[1] : mu[2] * Su[0]) + 2.0 * (mu[2] * W[2]) * (d == 0 ? Sr[0] : Sr[1]);
        } else {
            // I = tr(rr) 1 - rr (symmetric); mu = I^-1 Wnb by cofactors
            const double tr = g[4] + g[5] + g[6];
            const double I00 = tr - g[4], I11 = tr - g[5], I22 = tr - g[6];
            const double I01 = -g[7], I02 = -g[8], I12 = -g[9];
            const double c00 = I11 * I22 - I12 * I12, c01 = I02 * I12 - I01 * I22, c02 = I01 * I12 - I02 * I11;
            const double c11 = I00 * I22 - I02 * I02, c12 = I01 * I02 - I00 * I12, c22 = I00 * I11 - I01 * I01;
            const double idet = rcp64(I00 * c00 + I01 * c01 + I02 * c02);
            mu[0] = (c00 * Wb[0] + c01 * Wb[1] + c02 * Wb[2]) * idet;
            mu[1] = (c01 * Wb[0] + c11 * Wb[1] + c12 * Wb[2]) * idet;
            mu[2] = (c02 * Wb[0] + c12 * Wb[1] + c22 * Wb[2]) * idet;
            const double muW = mu[0] * W[0] + mu[1] * W[1] + mu[2] * W[2];
            const double SrW = Sr[0] * W[0] + Sr[1] * W[1] + Sr[2] * W[2];
            const double muSr = mu[0] * Sr[0] + mu[1] * Sr[1] + mu[2] * Sr[2];
            const int k1 = d == 2 ? 0 : d + 1, k2 = d == 0 ? 2 : d - 1;
            t = mu[k1] * Su[k2] - mu[k2] * Su[k1] + 2.0 * muW * Sr[d] - mu[d] * SrW - W[d] * muSr;
        }
        b.Ub[e] = 0.5 * Ubb[e];
        b.Xb[e] = d < D ? xb + t : 0.0;
        b.coef[8 * p + d] = (float)(Unb * icnt);
        b.coef[8 * p + 3 + d] = (float)mu[d];
    }
}

// After the sweep: fold the fluid sums of step 0 and write, per instance,
// [d alpha] + per particle [d ratio, d X0 (3), d U0 (3), d W0 (3), d theta0 (3), d A0 (3)].
__global__ void k_adj_finish(const InstDesc* __restrict__ insts, const AdjBufs* __restrict__ bufs,
                             const long long* __restrict__ out_off, double* __restrict__ out) {
    const int ii = blockIdx.x;
    const InstDesc& in = insts[ii];
    const AdjBufs b = bufs[ii];
    double* o = out + out_off[ii];
    double al = 0.0;
    for (int p = threadIdx.x; p < in.np; p += blockDim.x) {
        const double iratio = in.pconst[PCONST_N * p + PC_INVRHOS] * in.rho_f;
        double gsum = 0.0;
        double* r = o + 1 + 16LL * p;
        for (int d = 0; d < 3; ++d) {
            const double fl = b.Abar[4 * p + d];
            gsum += fl * (double)in.ggrav[d];
            r[1 + d] = b.Xb[3 * p + d];
            r[4 + d] = b.Ub[3 * p + d];
            r[7 + d] = b.Wb[3 * p + d];
            r[10 + d] = b.Tb[3 * p + d];
            r[13 + d] = b.Ab[3 * p + d] + fl;
        }
        al += b.Abar[4 * p + 3];
        r[0] = b.rb[p] + gsum * iratio * iratio;
    }
    __shared__ double red[128];
    red[threadIdx.x] = al;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int k = 0; k < (int)blockDim.x; ++k) s += red[k];
        o[0] = *b.alpha_b + s;
    }
}

// The particle state of checkpoint s, every instance in one launch (a block
// each; one launch and three copies or clears per instance before).
__global__ void __launch_bounds__(256) k_adj_state(const InstDesc* __restrict__ insts, const AdjSeg* __restrict__ seg,
                                                   int s, AdjStateOp op) {
    const InstDesc& in = insts[blockIdx.x];
    const AdjSeg g = seg[blockIdx.x];
    const int np = in.np;
    double* rec = g.ckst + 16LL * np * s;
    double* arr[5] = {in.X, in.U, in.W, in.theta, in.A};
    for (int p = threadIdx.x; p < np; p += blockDim.x) {
        double* r = rec + 16LL * p;
#pragma unroll
        for (int a = 0; a < 5; ++a)
            for (int d = 0; d < 3; ++d) {
                if (op == ADJ_SAVE) r[3 * a + d] = arr[a][3 * p + d];
                else arr[a][3 * p + d] = r[3 * a + d];
            }
        if (op == ADJ_SAVE) r[15] = (double)in.count[p];
        else in.count[p] = (int)r[15];
    }
    if (op != ADJ_RESTART) return;
    for (int k = threadIdx.x; k < 16 * np; k += blockDim.x) g.rstate[k] = rec[k];
    for (int k = threadIdx.x; k < 2 * NPV * np; k += blockDim.x) g.tot[k] = 0;
    for (int k = threadIdx.x; k < g.ntiles; k += blockDim.x) g.rlcnt[k] = 0;
}

// ------------------------------------------------------------- launchers --
cudaError_t launch_adj_fluid(int Q, int fp16, const InstDesc* insts, const AdjFluid* afs,
                             const uint16_t* tile_inst, int ninst, int ntiles, int lam_mode, const Shape& sh,
                             int num_sms, cudaStream_t st) {
    const int units = sh.ty * sh.tz * ((sh.tw + 63) / 64), per = (units + ADJ_WARPS - 1) / ADJ_WARPS;
    // With few tiles every segment goes to a warp of its own; with two waves of
    // tiles or more one block takes a whole tile and starts up once (backward pass,
    // 1 / 2 / 4 blocks per tile: one 400 x 1600 box, 240 steps 13.4 / 12.2 / 11.9 ms;
    // 48 steps FP32 of 1, 2, 3, 4, 8, 16 of them (800 tiles each): 2.49 / 2.36 / 2.37,
    // 3.58 / 3.49 / 3.57, 4.59 / 4.58 / 4.68, 5.52 / 5.64 / 5.78, 9.18 / 9.64 / 10.64, 16.4 /
    // 17.5 / 20.0 ms; FP16, half as tall tiles, 2.32 / 2.33 / 2.34 at 1600 tiles, 3.44 /
    // 3.49 at 3200; 100 x 200 boxes and D3Q19 do not tell the splits apart).
    const bool many = ntiles >= 2 * ADJ_BLOCKS * num_sms;
    const dim3 grid((unsigned)ntiles, many ? 1u : (unsigned)per);
    auto go = [&](auto kern) { kern<<<grid, 32 * ADJ_WARPS, 0, st>>>(insts, afs, tile_inst, ninst, lam_mode, sh); };
    if (Q == 9) {
        if (fp16) go(k_adj_fluid<9, __half>);
        else go(k_adj_fluid<9, float>);
    } else {
        if (fp16) go(k_adj_fluid<19, __half>);
        else go(k_adj_fluid<19, float>);
    }
    return cudaGetLastError();
}

cudaError_t launch_adj_particles(int D, const InstDesc* insts, const AdjPart* steps, const AdjBufs* bufs,
                                 int ninst, cudaStream_t st) {
    if (D == 2) k_adj_particles<2><<<ninst, 128, 0, st>>>(insts, steps, bufs);
    else k_adj_particles<3><<<ninst, 128, 0, st>>>(insts, steps, bufs);
    return cudaGetLastError();
}

cudaError_t launch_adj_finish(const InstDesc* insts, const AdjBufs* bufs, const long long* out_off,
                              double* out, int ninst, cudaStream_t st) {
    k_adj_finish<<<ninst, 128, 0, st>>>(insts, bufs, out_off, out);
    return cudaGetLastError();
}

cudaError_t launch_adj_pull_out(int Q, const InstDesc* insts, int inst, long long N, const float* lam,
                                float* out, cudaStream_t st) {
    const unsigned blocks = (unsigned)((N + 255) / 256);
    if (Q == 9) k_adj_pull_out<9><<<blocks, 256, 0, st>>>(insts, inst, lam, out);
    else k_adj_pull_out<19><<<blocks, 256, 0, st>>>(insts, inst, lam, out);
    return cudaGetLastError();
}

cudaError_t launch_adj_state(const InstDesc* insts, const AdjSeg* seg, int ninst, int s, AdjStateOp op, cudaStream_t st) {
    k_adj_state<<<ninst, 256, 0, st>>>(insts, seg, s, op);
    return cudaGetLastError();
}

}  // namespace lbmpen
