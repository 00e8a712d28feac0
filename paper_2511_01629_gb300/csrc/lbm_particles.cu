// Per-particle FP64 kernel of lbmpen: the second pass of the rigid-body
// projection (Eq. 22) from the totals that the fluid kernel added up, the
// predictor-corrector of Algorithm 1 with the repulsive collision forces
// (Eqs. 19-21), and the rebuild of each particle's record and tile-list
// entries for the next step.
//
// One launch does all of it, with no barrier between the projection and the
// pair forces: a particle's U^n follows from its totals by a few operations,
// so a block takes the U^n of the few neighbours it needs from their totals
// itself.  What a block reads of other particles (totals, state) is kept per
// step parity, and a block writes only the other parity's.
//
// GB300 runs FP64 at a small fraction of its FP32 rate, and an FP64
// instruction occupies a sub-partition's FP64 pipe for ~64 cycles whether one
// lane or 32 are active, so the serial per-particle arithmetic runs one lane
// per (particle, vector component).  The O(N^2) pair search uses a warp per
// particle and filters pairs in FP32 (positions staged in shared memory)
// before the FP64 evaluation of the few pairs in range.
#include "lbm_common.cuh"

namespace lbmpen {

constexpr int PB = 8;         // particles per block (one per warp)
constexpr int XCHUNK = 1024;  // particle positions staged in shared memory at a time

// Extent of a particle along the unit vector (nx, ny): R for a disk; for an
// ellipse (semi-axes R = a and B = b, orientation (ec, es)) the support
// distance sqrt(a^2 (n.e)^2 + b^2 (n.e_perp)^2).  Used in place of the radius
// in Eqs. 19-20, which the paper states for disks.
__device__ __forceinline__ double extent_along(double R, double B, double ec, double es, double nx,
                                               double ny) {
    if (B == R) return R;
    const double ne = __dadd_rn(__dmul_rn(nx, ec), __dmul_rn(ny, es));
    const double np = __dsub_rn(__dmul_rn(ny, ec), __dmul_rn(nx, es));
    return sqrt(__dadd_rn(__dmul_rn(__dmul_rn(R, R), __dmul_rn(ne, ne)),
                          __dmul_rn(__dmul_rn(B, B), __dmul_rn(np, np))));
}

// Position X^{k} of particle j and, with ub, its Ubar (FP64): before the first
// sub-step from its state and totals of this step, later from the arrays that
// its block wrote.
template <bool FIRST>
__device__ __forceinline__ void pair_operands(const InstDesc& in, int j, int src, int par, int D, bool ub, double* X,
                                              double* Ub) {
    for (int d = 0; d < 3; ++d) Ub[d] = 0.0;
    if (!FIRST) {
        for (int d = 0; d < 3; ++d) {
            X[d] = in.Xk[(long long)src * in.np * 3 + 3 * j + d];
            if (ub) Ub[d] = in.Ubar[3 * j + d];
        }
        return;
    }
    const PState& ps = in.pst[par][j];
    for (int d = 0; d < 3; ++d) X[d] = ps.X[d];
    if (!ub) return;
    const long long* v = in.tot[par] + (long long)NPV * j;
    if (v[0] == 0) return;
    const double inv = rcp64((double)v[0]);
    for (int d = 0; d < D; ++d) Ub[d] = 0.5 * (finalize_u(v[10 + d], inv) + ps.U[d]);
}

// Pair part of Eq. 21 on particle i at two position sets: X^{k} (F1) and
// X^{k} + h Ubar (F2).  The block's particles all belong to one instance;
// its positions are staged in shared memory in chunks and the lanes split
// them: bit k of a lane's mask stands for particle j0 + lane + 32 k.  An FP32
// filter (pair_mask) leaves the pairs within 2 of range at X^{k} (a predicted
// position lies within |h Ubar| < sqrt(3)/2 of it, a larger step is reported
// as ST_DISPLACEMENT); pair_forces evaluates in FP64, in the reference operation
// order, those near the range at X^{k} or at the predicted positions.
static_assert(XCHUNK <= 32 * 32, "a lane's pairs of a chunk fit a mask");
struct PairGeo {
    float n[3];
    bool per[3];
    __device__ __forceinline__ explicit PairGeo(const InstDesc& in) {
        for (int d = 0; d < 3; ++d) {
            n[d] = (float)in.n[d];
            per[d] = in.periodic[d] && in.n[d] > 1;
        }
    }
    __device__ __forceinline__ float dist2(float4 a, float4 b) const {
        float dv[3] = {a.x - b.x, a.y - b.y, a.z - b.z};
#pragma unroll
        for (int d = 0; d < 3; ++d)
            if (per[d]) dv[d] -= n[d] * rintf(dv[d] / n[d]);
        return dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2];
    }
};
// An FP32 position on an axis of n nodes carries an error of 2^-24 n, a predicted
// one twice that: the distance of two is off by up to 4 sqrt(3) 2^-24 n < 5e-7 n.
__device__ __forceinline__ float pair_reach(const InstDesc& in, const PairGeo& g, float4 xi) {
    return xi.w + (float)in.delta + fmaf(5e-7f, fmaxf(fmaxf(g.n[0], g.n[1]), g.n[2]), 0.01f);
}

__device__ __forceinline__ unsigned pair_mask(const InstDesc& in, int i, int lane, const float4* xs, int j0, int nj, float4 xi) {
    const PairGeo g(in);
    const float reach = pair_reach(in, g, xi) + 2.0f;
    unsigned m = 0;
    for (int jj = lane, k = 0; jj < nj; jj += 32, ++k) {
        const float4 b = xs[jj];
        const float lim = reach + b.w;
        if (j0 + jj != i && g.dist2(xi, b) <= lim * lim) m |= 1u << k;
    }
    return m;
}

template <bool FIRST>
__device__ __noinline__ void pair_forces(const InstDesc& in, int i, int src, int par, double h, int D, int lane, const float4* xs,
                            const float4* xs2, int j0, unsigned m, float4 xi, float4 xi2, double cp, double inv_delta,
                            double* f1, double* f2) {
    if (cp == 0.0) return;  // cp = C / eps_p of particle i
    const PairGeo g(in);
    const float reach = pair_reach(in, g, xi);
    // X + h Ubar of a particle in FP32, from its totals (before the first sub-step)
    auto predicted = [&](int j, float4 x) {
        const long long* v = in.tot[par] + (long long)NPV * j;
        const float s = v[0] > 0 ? 9.094947017729282e-13f / (float)v[0] : 0.f;  // 2^-40 / count
        const PState& ps = in.pst[par][j];
        const float hh = 0.5f * (float)h;
        x.x += hh * ((float)v[10] * s + (float)ps.U[0]);
        x.y += hh * ((float)v[11] * s + (float)ps.U[1]);
        if (D == 3) x.z += hh * ((float)v[12] * s + (float)ps.U[2]);
        return x;
    };
    for (; m; m &= m - 1) {
        const int jj = lane + 32 * (__ffs(m) - 1), j = j0 + jj;
        const float4 b = xs[jj];
        const float lim = reach + b.w;
        const float d2 = g.dist2(xi, b);
        const float e2 = FIRST ? g.dist2(predicted(i, xi), predicted(j, b)) : g.dist2(xi2, xs2[jj]);
        const bool near[2] = {d2 <= lim * lim, e2 <= lim * lim};
        if (!near[0] && !near[1]) continue;
        const double Bi = in.pconst[PCONST_N * i + PC_B], Bj = in.pconst[PCONST_N * j + PC_B];
        const bool ell = Bi != in.R[i] || Bj != in.R[j];
        double Xi[3], Xj[3], Ui[3], Uj[3];
        pair_operands<FIRST>(in, i, src, par, D, near[1], Xi, Ui);
        pair_operands<FIRST>(in, j, src, par, D, near[1], Xj, Uj);
        for (int pass = 0; pass < 2; ++pass) {
            if (!near[pass]) continue;
            const double sh = pass ? h : 0.0;
            double dd[3];
            for (int d = 0; d < 3; ++d) {
                const double xi_d = Xi[d] + sh * Ui[d];
                const double xj_d = Xj[d] + sh * Uj[d];
                dd[d] = xi_d - xj_d;
                if (g.per[d]) {
                    const double half = 0.5 * in.n[d];
                    if (dd[d] > half) dd[d] -= in.n[d];
                    else if (dd[d] < -half) dd[d] += in.n[d];
                }
            }
            const double dij = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(dd[0], dd[0]), __dmul_rn(dd[1], dd[1])),
                                              __dmul_rn(dd[2], dd[2])));
            double range = in.R[i] + in.R[j] + in.delta;
            if (ell && dij > 0.0) {  // ellipses (2D): extents along the line of centres
                const double nx = dd[0] / dij, ny = dd[1] / dij;
                const PState &ri = in.pst[par][i], &rj = in.pst[par][j];
                range = extent_along(in.R[i], Bi, ri.ec, ri.es, nx, ny) +
                        extent_along(in.R[j], Bj, rj.ec, rj.es, nx, ny) + in.delta;
            }
            if (dij <= range) {
                const double sc = (range - dij) * inv_delta;
                double* f = pass ? f2 : f1;
                for (int d = 0; d < 3; ++d) f[d] += cp * dd[d] * sc * sc;
            }
        }
    }
}

// Gather the (few) lanes that found a pair into every lane.
__device__ void gather_pairs(const double* f1, const double* f2, double* F1, double* F2) {
    const unsigned act = __ballot_sync(0xffffffffu, f1[0] != 0 || f1[1] != 0 || f1[2] != 0 ||
                                                        f2[0] != 0 || f2[1] != 0 || f2[2] != 0);
    double g1[3] = {0, 0, 0}, g2[3] = {0, 0, 0};
    for (int l = 0; l < 32; ++l) {
        if (!(act & (1u << l))) continue;
        for (int d = 0; d < 3; ++d) {
            g1[d] += __shfl_sync(0xffffffffu, f1[d], l);
            g2[d] += __shfl_sync(0xffffffffu, f2[d], l);
        }
    }
    for (int d = 0; d < 3; ++d) {
        F1[d] = g1[d];
        F2[d] = g2[d];
    }
}

// Wall part of Eq. 21 (mirror images across the planes -1/2 and n - 1/2),
// component d of the force on a particle at coordinate Xi along axis d; Ri is
// the particle's extent along axis d (its radius, for a disk).
__device__ void wall_force_d(const InstDesc& in, int d, double Xi, double& F, double cw, double inv_delta,
                             double Ri) {
    if (cw == 0.0) return;  // cw = C / eps_w of the particle
    const float reach = wall_reach(in, d, Ri);
    if (in.periodic[d] || in.n[d] <= 1) return;
    const float xf = (float)Xi;  // skip walls farther than (2R + delta)/2
    if (xf + 0.5f > reach && (float)in.n[d] - 0.5f - xf > reach) return;
    const double walls[2] = {-0.5, in.n[d] - 0.5};
    for (int face = 0; face < 2; ++face) {
        const double Xim = 2.0 * walls[face] - Xi;
        const double diff = Xi - Xim;
        const double dprime = fabs(diff);
        const double range = 2.0 * Ri + in.delta;
        if (dprime <= range) {
            const double sc = (range - dprime) * inv_delta;
            F += cw * diff * sc * sc;
        }
    }
}

// Tiles along one axis that hold nodes of the node interval [X-R-1, X+R+1]:
// tiles a0 .. a0+na-1 and b0 .. b0+nb-1 (disjoint).  On a periodic axis the
// interval may wrap; it is split at the face before mapping to tiles, since
// the last tile of a ragged axis does not continue into the first one.
struct AxisTiles {
    int a0, na, b0, nb;
};

__device__ AxisTiles axis_tiles_f(float X, float R, int n, int T, int ntile, int periodic) {
    int lo = (int)floorf(X - R) - 1, hi = (int)floorf(X + R) + 1;
    AxisTiles t{0, 1, 0, 0};
    if (!periodic) {
        lo = min(max(lo, 0), n - 1);  // in range wherever a failed run may have put X
        hi = max(min(hi, n - 1), lo);
        t.a0 = lo / T;
        t.na = hi / T - t.a0 + 1;
        return t;
    }
    if (hi - lo + 1 >= n) {
        t.a0 = 0;
        t.na = ntile;
        return t;
    }
    int alo, bhi;
    if (lo < 0) {
        alo = lo + n;
        bhi = hi;
    } else if (hi >= n) {
        alo = lo;
        bhi = hi - n;
    } else {
        t.a0 = lo / T;
        t.na = hi / T - t.a0 + 1;
        return t;
    }
    const int ta0 = alo / T, tb1 = bhi / T;
    if (tb1 >= ta0) {  // the two pieces share a tile: take the whole axis
        t.a0 = 0;
        t.na = ntile;
        return t;
    }
    t.a0 = ta0;
    t.na = ntile - ta0;
    t.b0 = 0;
    t.nb = tb1 + 1;
    return t;
}

__device__ __forceinline__ int axis_tile(const AxisTiles& t, int i) {
    return i < t.na ? t.a0 + i : t.b0 + (i - t.na);
}

// Component d of a particle's record for the next fluid step: the reference
// node floor(X), the offset from it, the acceleration term of the penalty
// force, and the tiles of the bounding box [X - R - 1, X + R + 1] along d (its
// one-node margin covers the float rounding).
struct RecComp {
    int ref;
    float frac, a;
    AxisTiles t;
};

__device__ __forceinline__ RecComp record_component(const InstDesc& in, int d, int D, const Shape& sh, double X,
                                                    double A, float Rf, float gfac) {
    const int T = d == 0 ? sh.tw : (d == 1 ? sh.ty : sh.tz);
    RecComp r;
    r.ref = d < D ? __double2int_rd(X) : 0;
    r.frac = (float)(X - (double)r.ref);
    r.a = fmaf(gfac, in.ggrav[d], (float)A);
    r.t = d >= D ? AxisTiles{0, 1, 0, 0}
                 : axis_tiles_f((float)r.ref + r.frac, Rf, in.n[d], T, in.ntile[d], in.periodic[d]);
    return r;
}

// The size and shape fields of particle p's record (host-computed, RecConst)
// and its tile count (nt tiles of the bounding box).
__device__ __forceinline__ void record_radius(const InstDesc& in, PRec& pr, const RecConst& rc, int nt) {
    pr.R2 = rc.R2;
    pr.R2lo = rc.R2lo;
    pr.R2hi = rc.R2hi;
    pr.ntiles = nt;
    pr.shape = rc.shape;
    pr.rows2 = rc.rows2;
    pr.b2 = rc.b2;
    pr.ia2 = rc.ia2;
    pr.ib2 = rc.ib2;
    pr.qlo = rc.qlo;
    pr.qhi = rc.qhi;
    pr.pad2[0] = pr.pad2[1] = 0.f;
    if (nt > in.maxk) atomicOr(in.status, ST_CAPACITY);
}

// Orientation fields of a record: cos and sin of theta (the z component of
// the orientation in 2D) for an ellipse; (1, 0) otherwise.
__device__ __forceinline__ void record_orientation(PRec& pr, bool ellipse, double theta) {
    double c = 1.0, s = 0.0;
    if (ellipse) sincos(theta, &s, &c);
    pr.ec = c;
    pr.es = s;
    pr.fc = (float)c;
    pr.fs = (float)s;
}

// Record of particle p from its state (X, A, theta) and constants (R, B,
// 1 - rho_f/rho_s), with the tiles of its bounding box (slots k enumerate them
// x-fastest; no tile is listed twice).  One thread.
__device__ PRec make_record_from(const InstDesc& in, int p, int D, const Shape& sh, AxisTiles* at,
                                 const double* Xp, const double* Ap, double R, double B, double theta,
                                 float gfac) {
    PRec pr;
    int nt = 1;
    for (int d = 0; d < 3; ++d) {
        const RecComp r = record_component(in, d, D, sh, Xp[d], Ap[d], (float)R, gfac);
        pr.X[d] = Xp[d];
        pr.ref[d] = r.ref;
        pr.frac[d] = r.frac;
        pr.a[d] = r.a;
        at[d] = r.t;
        nt *= r.t.na + r.t.nb;
    }
    record_radius(in, pr, in.rconst[p], nt);
    record_orientation(pr, B != R, theta);
    in.prec_out[p] = pr;
    return pr;
}

// The candidate record of a particle (Cand) from its record's fields.
__device__ __forceinline__ Cand make_cand(const PRec& pr, int p) {
    Cand cd;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        cd.ref[d] = pr.ref[d];
        cd.frac[d] = pr.frac[d];
        cd.a[d] = pr.a[d];
    }
    cd.R2lo = pr.R2lo;
    cd.R2hi = pr.R2hi;
    cd.p = p;
    cd.k = 0;
    cd.rows2 = pr.rows2;
    cd.pad = 0;
    cd.shape = pr.shape;
    return cd;
}

__device__ Cand make_record(const InstDesc& in, int p, int D, const Shape& sh, AxisTiles* at, int lpar) {
    double X[3], A[3];
    for (int d = 0; d < 3; ++d) {
        X[d] = in.X[3 * p + d];
        A[d] = in.A[3 * p + d];
    }
    const double R = in.pconst[PCONST_N * p + PC_R];
    const PRec pr = make_record_from(in, p, D, sh, at, X, A, R, in.pconst[PCONST_N * p + PC_B], in.theta[3 * p + 2],
                                     (float)in.pconst[PCONST_N * p + PC_GFAC]);
    PState& ps = in.pst[lpar][p];
    for (int d = 0; d < 3; ++d) {
        ps.X[d] = X[d];
        ps.U[d] = in.U[3 * p + d];
    }
    ps.ec = pr.ec;
    ps.es = pr.es;
    in.Xp[lpar][p] = make_float4((float)X[0], (float)X[1], (float)X[2], (float)R);
    return make_cand(pr, p);
}

// List entries of particle p in the tiles of its bounding box (lanes share):
// the entry p << KBITS | k and, in the same slot, the 64-byte candidate record
// cd that the fluid kernel copies.
__device__ void append_tiles(const InstDesc& in, int p, const AxisTiles* at, Cand cd, int lpar, int lane, int nl) {
    const int cnt[3] = {at[0].na + at[0].nb, at[1].na + at[1].nb, at[2].na + at[2].nb};
    const int nt = cnt[0] * cnt[1] * cnt[2];
    Cand* rec = static_cast<Cand*>(in.list_rec[lpar]);
    for (int k = lane; k < nt && k < in.maxk; k += nl) {
        const int kx = k % cnt[0], ky = (k / cnt[0]) % cnt[1], kz = k / (cnt[0] * cnt[1]);
        const int tc[3] = {axis_tile(at[0], kx), axis_tile(at[1], ky), axis_tile(at[2], kz)};
        const int local = (tc[2] * in.ntile[1] + tc[1]) * in.ntile[0] + tc[0];
        const int pos = atomicAdd(&in.list_cnt[lpar][local], 1);
        if (pos < LIST_CAP) {
            // the slot is informational (a particle may cover more than MAXK
            // tiles): only its low KBITS bits go into the entry, below p
            in.list_ent[lpar][(long long)local * LIST_CAP + pos] = ((uint32_t)p << KBITS) | (uint32_t)(k & (MAXK - 1));
            cd.k = k;
            rec[(long long)local * LIST_CAP + pos] = cd;
        } else {
            atomicOr(in.status, ST_CAPACITY);
        }
    }
}

// Algorithm 1 for particle i, component d (one lane per component; the lanes
// of particle slot sl are sl + PB * d, and lanes with valid = false take part
// in the shuffles only): wall forces, the corrected position, and on the last
// sub-step A^{n+1}, theta^{n+1}, U^{n-1} <- U^n and the record for the next
// step.  Each lane evaluates the expressions of a serial loop over d.
// The operands of update_lane, loaded in one batch before the pair search so
// that their latency overlaps it (on the first sub-step before the fluid kernel
// has ended; project_lane adds what its totals give).
struct LaneIn {
    double X0, Ub, Un, invrhos, cw, idl, Ri, Bi, gfac, invc, Acor, ec, es;
    int cnt;
    RecConst rc;
};

__device__ __forceinline__ LaneIn load_lane(const InstDesc& in, int i, int d, bool valid, int src, int par, int first) {
    if (!valid) {  // in-range operands for the shuffle-only lanes
        i = 0;
        d = 0;
    }
    const long long j = 3LL * i + d;
    LaneIn L;
    const PState& ps = in.pst[par][i];
    // orientation theta^n of this step's record
    L.ec = first ? ld_l2(&ps.ec) : ps.ec;
    L.es = first ? ld_l2(&ps.es) : ps.es;
    if (first) {
        L.X0 = ld_l2(ps.X + d);
        L.Ub = ld_l2(ps.U + d);  // U^{n-1} until project_lane
    }
    const double* pc = in.pconst + PCONST_N * i;
    L.invrhos = pc[PC_INVRHOS];
    L.cw = pc[PC_CWALL];
    L.idl = pc[PC_INVDELTA];
    L.Ri = pc[PC_R];
    L.Bi = pc[PC_B];
    L.gfac = pc[PC_GFAC];
    L.rc = in.rconst[i];
    if (first) {
        L.Acor = 0.0;
    } else {
        L.X0 = in.Xk[(long long)src * in.np * 3 + j];
        L.Ub = in.Ubar[j];
        L.Un = in.Un[j];
        L.invc = in.invc[i];
        L.cnt = in.count[i];
        L.Acor = in.Acor[j];
    }
    return L;
}

// The translation of Eq. 22 into the operands of the first sub-step, from the
// totals of this step.
__device__ __forceinline__ void project_lane(const InstDesc& in, int i, int d, bool valid, int par, int D, LaneIn& L) {
    if (!valid) {
        i = 0;
        d = 0;
    }
    const long long j = 3LL * i + d;
    const long long* v = in.tot[par] + (long long)NPV * i;
    const long long n = v[0], su = v[10 + d];
    const double Uold = L.Ub;
    L.cnt = (int)n;
    L.invc = 0.0;
    L.Un = Uold;
    L.Ub = 0.0;
    if (n != 0) {
        L.invc = rcp64((double)n);
        L.Un = d < D ? finalize_u(su, L.invc) : 0.0;
        L.Ub = d < D ? 0.5 * (L.Un + Uold) : 0.0;
    }
    if (valid) {
        in.Un[j] = L.Un;
        if (n == 0 && d == 0) atomicOr(in.status, ST_PARTICLE);
        if (!(fabs(L.Ub) < 0.5)) atomicOr(in.status, ST_DISPLACEMENT);
        if (d == 0) in.count[i] = (int)n;
        if (in.K > 1) {  // the later sub-steps read these
            in.Ubar[j] = L.Ub;
            if (d == 0) in.invc[i] = L.invc;
        }
    }
}

// Rotation of particle i, component d: W^n (first sub-step, Eq. 22) and, on
// the last one, theta^{n+1} (reading: trapezoid of W) with the record's
// orientation.  Runs on its own warp beside update_lane.
__device__ __forceinline__ void rotate_lane(const InstDesc& in, int i, int d, int par, int first, int last, int D,
                                            double Th, double Wo) {
    const long long j = 3LL * i + d;
    double Wn;
    if (first) {
        double* geo = in.adj_geo ? in.adj_geo + (long long)NPV * i : nullptr;
        const long long* v = in.tot[par] + (long long)NPV * i;
        Wn = D == 2 ? finalize_rotation<2>(v, in.pst[par][i].X, d, geo) : finalize_rotation<3>(v, in.pst[par][i].X, d, geo);
        in.Wn[j] = Wn;
    } else {
        Wn = in.Wn[j];
    }
    if (!last) return;
    const double Tn = Th + 0.5 * (Wn + Wo);
    in.theta[j] = Tn;
    in.W[j] = Wn;
    if (in.rec_state) {
        in.rec_state[16LL * i + 6 + d] = Wn;
        in.rec_state[16LL * i + 9 + d] = Tn;
    }
    if (d == 2) {
        const double* pc = in.pconst + PCONST_N * i;
        PRec& pr = in.prec_out[i];
        record_orientation(pr, pc[PC_B] != pc[PC_R], Tn);
        PState& ps = in.pst[par ^ 1][i];
        ps.ec = pr.ec;
        ps.es = pr.es;
    }
}

__device__ __forceinline__ void update_lane(const InstDesc& in, int i, int d, int sl, bool valid, const double* F1in,
                            const double* F2in, int src, int par, double h, int first, int last, int D,
                            const Shape& sh, AxisTiles* at, Cand& cd, const LaneIn& L) {
    if (!valid) {  // in-range operands for the shuffle-only lanes; nothing is stored
        i = 0;
        d = 0;
    }
    const int dst = src ^ 1;
    const long long j = 3LL * i + d;
    const double X0 = L.X0, Ub = L.Ub;
    double F1 = F1in ? F1in[d] : 0.0, F2 = F2in ? F2in[d] : 0.0;
    const double Ri = L.Ri, Bi = L.Bi;
    const double invM = L.invrhos * L.invc;  // 1 / (rho_s n)
    const double Xst = fma(h, Ub, X0);
    // extent along axis d: the radius, or for an ellipse at theta^n (this
    // step's record) its support distance normal to the walls of axis d
    double Rd = Ri;
    if (Bi != Ri && d < 2)
        Rd = d == 0 ? extent_along(Ri, Bi, L.ec, L.es, 1.0, 0.0) : extent_along(Ri, Bi, L.ec, L.es, 0.0, 1.0);
    wall_force_d(in, d, X0, F1, L.cw, L.idl, Rd);
    wall_force_d(in, d, Xst, F2, L.cw, L.idl, Rd);
    const double c = 0.25 * h * h * invM;  // (1 / 2M) h^2 / 2
    const double cor = c * (F1 + F2);      // this sub-step's correction
    const double Xn = Xst + cor;
    // A^{n+1} = 2 (X^{n+1} - X^n - Ubar) is twice the sum of the corrections;
    // summed directly, since the difference of positions cancels catastrophically
    const double acc = first ? cor : L.Acor + cor;
    const float Rf = (float)Ri;
    if (!last) {
        if (valid) {
            in.Acor[j] = acc;
            in.Xk[(long long)dst * in.np * 3 + j] = Xn;
            float* xf = in.Xf + ((long long)dst * in.np + i) * 4;
            float* xsf = in.Xsf + ((long long)dst * in.np + i) * 4;
            xf[d] = (float)Xn;
            xsf[d] = (float)fma(h, Ub, Xn);
            if (d == 0) {
                xf[3] = Rf;
                xsf[3] = Rf;
            }
        }
        return;
    }
    bool left = false;
    const double An = 2.0 * acc;
    double xn = Xn;
    if (d < D) {
        if (in.periodic[d]) {
            if (xn >= in.n[d]) xn -= in.n[d];
            else if (xn < 0.0) xn += in.n[d];
        } else if (xn < -0.5 || xn > in.n[d] - 0.5) {
            left = true;
        }
    }
    const RecComp r = record_component(in, d, D, sh, xn, An, Rf, (float)L.gfac);
    const int ct = r.t.na + r.t.nb;
    const int nt = __shfl_sync(0xffffffffu, ct, sl) * __shfl_sync(0xffffffffu, ct, sl + PB) *
                   __shfl_sync(0xffffffffu, ct, sl + 2 * PB);
    if (!valid) return;
    at[d] = r.t;  // shared: what append_tiles needs
    cd.ref[d] = r.ref;
    cd.frac[d] = r.frac;
    cd.a[d] = r.a;
    if (d == 0) {
        cd.R2lo = L.rc.R2lo;
        cd.R2hi = L.rc.R2hi;
        cd.p = i;
        cd.rows2 = L.rc.rows2;
        cd.pad = 0;
        cd.shape = L.rc.shape;
    }
    in.A[j] = An;
    in.X[j] = xn;
    in.U[j] = L.Un;
    PState& ps = in.pst[par ^ 1][i];
    ps.X[d] = xn;
    ps.U[d] = L.Un;
    float* xp = reinterpret_cast<float*>(in.Xp[par ^ 1] + i);
    xp[d] = (float)xn;
    if (d == 0) xp[3] = Rf;
    if (left) atomicOr(in.status, ST_PARTICLE);
    if (in.rec_state) {  // adjoint recording: the state this step hands to the next
        double* q = in.rec_state + 16LL * i;
        q[d] = xn;
        q[3 + d] = L.Un;
        q[12 + d] = An;
        if (d == 0) q[15] = (double)L.cnt;
    }
    PRec& pr = in.prec_out[i];
    pr.X[d] = xn;
    pr.ref[d] = r.ref;
    pr.frac[d] = r.frac;
    pr.a[d] = r.a;
    if (d == 0) record_radius(in, pr, L.rc, nt);
}

// ------------------------------------------------------------- the kernel --
// Default bound on a barrier wait (2 s); a context may set another
// (lbm_set_particle_wait_limit), 0 included: then a block that does not find
// the barrier open on its first look gives up at once.
constexpr unsigned long long PWAIT_NS = 2000000000ull;

__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// Barrier over all blocks of the particle kernel (launched only when they are
// all resident).  Bounded: after limit_ns it records a timeout and returns
// false, and the kernel stops.  Every block arrives before it waits, so the
// last arrival always resets the count, timeouts included.
__device__ bool grid_sync(GridBar* gb, int* status, unsigned long long limit_ns) {
    if (gridDim.x == 1) {  // one block: the block barrier is the grid barrier
        __syncthreads();
        return true;
    }
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        volatile unsigned* vgen = &gb->gen;
        const unsigned g = *vgen;  // generation before this block arrives
        __threadfence();
        if (atomicAdd(&gb->count, 1) == gridDim.x - 1) {
            gb->count = 0;
            __threadfence();
            atomicAdd(&gb->gen, 1u);
        } else {
            const unsigned long long t0 = gtimer();
            while (*vgen == g) {
                if (gtimer() - t0 >= limit_ns) {
                    ok = 0;
                    atomicOr(status, ST_TIMEOUT);
                    break;
                }
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// Phase k (1..K): sub-step k of Algorithm 1 for the block's particles (slot s
// is particle i0 + s; np of its instance), positions of buffer src -> src ^ 1
// (the first from the state).  The block's warps find the pair forces (one
// particle each); warp 0 does the FP64 update, one lane per particle component,
// warp 1 the rotation, and warp 2 clears the totals that the next step adds to.
// The first phase runs up to its wait beside the fluid kernel: that kernel lets
// this one start once the previous step's particle kernel has ended, so all but
// the totals is there (state, positions, the pairs that may be in range; read
// by ld_l2).
template <bool FIRST>
__device__ __forceinline__ void phase_substep(const InstDesc& in, int i0, int D, int src, int par, int last, const Shape& sh,
                              float4* xs, float4* xs2, double (*sF)[6], AxisTiles (*sAT)[3], Cand* sC) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double h = in.hK;
    const int i = i0 + warp;
    const bool mine = i < in.np;
    // warps 0 and 1: particle slot and component of the lane
    const int usl = lane & (PB - 1), ud = lane / PB;
    const bool uvalid = ud < 3 && i0 + usl < in.np;
    LaneIn li;
    double th = 0.0, wo = 0.0;
    if (warp == 0) li = load_lane(in, i0 + usl, ud, uvalid, src, par, FIRST);
    if (warp == 1 && uvalid) {
        const double *pt = in.theta + 3 * (i0 + usl) + ud, *pw = in.W + 3 * (i0 + usl) + ud;
        th = FIRST ? ld_l2(pt) : *pt;
        wo = FIRST ? ld_l2(pw) : *pw;
    }
    const bool pairs = in.np > 1;  // one particle: nothing to search
    const bool one = in.np <= XCHUNK;
    const float4* Xfb = FIRST ? in.Xp[par] : reinterpret_cast<const float4*>(in.Xf) + (long long)src * in.np;
    const float4* Xsb = reinterpret_cast<const float4*>(in.Xsf) + (long long)src * in.np;
    float4 xi = make_float4(0.f, 0.f, 0.f, 0.f), xi2 = xi;
    double cp = 0.0, idl = 0.0;
    // the positions of a chunk into shared memory, every load in flight at
    // once, and the pairs of the warp's particle that may be in range
    auto chunk = [&](int j0) {
        const int nj = min(XCHUNK, in.np - j0);
        constexpr int PER = XCHUNK / 256;  // blockDim.x == 256
        float4 ra[PER], rb[PER];
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int k = threadIdx.x + 256 * u;
            if (k < nj) {
                ra[u] = FIRST ? ld_l2(Xfb + j0 + k) : Xfb[j0 + k];
                if (!FIRST) rb[u] = Xsb[j0 + k];
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < PER; ++u) {
            const int k = threadIdx.x + 256 * u;
            if (k < nj) {
                xs[k] = ra[u];
                if (!FIRST) xs2[k] = rb[u];
            }
        }
        __syncthreads();
        return mine ? pair_mask(in, i, lane, xs, j0, nj, xi) : 0u;
    };
    unsigned m = 0;
    if (pairs) {
        if (mine) {  // issued before the staging barrier, so the loads overlap it
            xi = FIRST ? ld_l2(Xfb + i) : Xfb[i];
            if (!FIRST) xi2 = Xsb[i];
            cp = in.pconst[PCONST_N * i + PC_CPAIR];
            idl = in.pconst[PCONST_N * i + PC_INVDELTA];
        }
        if (one) m = chunk(0);
    }
    if (FIRST) {
        dep_wait();  // the totals of this step
        dep_launch();
        if (warp == 0) project_lane(in, i0 + usl, ud, uvalid, par, D, li);
    }
    if (pairs) {
        double f1[3] = {0, 0, 0}, f2[3] = {0, 0, 0};
        for (int j0 = 0; j0 < in.np; j0 += XCHUNK) {
            if (!one) m = chunk(j0);
            if (__any_sync(0xffffffffu, m != 0)) pair_forces<FIRST>(in, i, src, par, h, D, lane, xs, xs2, j0, m, xi, xi2, cp, idl, f1, f2);
        }
        if (mine) {  // (no lane found a pair: the sums are zero)
            double F1[3], F2[3];
            gather_pairs(f1, f2, F1, F2);
            if (lane == 0)
                for (int d = 0; d < 3; ++d) {
                    sF[warp][d] = F1[d];
                    sF[warp][3 + d] = F2[d];
                }
        }
        __syncthreads();
    }
    if (warp == 0) {
        update_lane(in, i0 + usl, ud, usl, uvalid, pairs ? sF[usl] : nullptr, pairs ? sF[usl] + 3 : nullptr, src, par, h,
                    FIRST, last, D, sh, sAT[usl], sC[usl], li);
    } else if (warp == 1) {
        if (uvalid) rotate_lane(in, i0 + usl, ud, par, FIRST, last, D, th, wo);
    } else if (FIRST && warp == 2) {
        for (int k = lane; k < PB * NPV; k += 32)
            if (i0 + k / NPV < in.np) in.tot[par ^ 1][(long long)NPV * i0 + k] = 0;
    }
}

// The later sub-steps (K > 1), out of line: their registers stay out of the K = 1 path.
__device__ __noinline__ void phase_later(const InstDesc& in, int i0, int D, int src, int par, int last, const Shape& sh,
                                         float4* xs, float4* xs2, double (*sF)[6], AxisTiles (*sAT)[3], Cand* sC) {
    phase_substep<false>(in, i0, D, src, par, last, sh, xs, xs2, sF, sAT, sC);
}

// Particle part of one time step for the block's 8 particles (one instance),
// phases first..last, phase k = sub-step k of Algorithm 1, the first after the
// projection of Eq. 22; after the last sub-step the warps append their
// particle to the next step's tile lists.  With more than one phase (K > 1)
// the blocks meet at grid barriers between phases (the launch guarantees they
// are all resident); with K = 1 there is no barrier.
template <int D>
__global__ void __launch_bounds__(256, 1) k_particles(const InstDesc* __restrict__ insts,
                                                   const PartRef* __restrict__ refs, int ninst, int K, int first, int last, int lpar,
                                                   Shape sh, GridBar* gb, unsigned long long wait_ns) {
    __shared__ double sF[PB][6];
    __shared__ AxisTiles sAT[PB][3];
    __shared__ Cand sC[PB];
    __shared__ float4 xs[XCHUNK];
    __shared__ float4 xs2[XCHUNK];
    __shared__ __align__(16) InstDesc sdesc;
    // blocks never straddle instances; one instance needs no look at the table
    PartRef r0{0, (int)blockIdx.x * PB};
    if (ninst > 1) r0 = refs[blockIdx.x * PB];
    stage_desc(&sdesc, insts[r0.inst]);
    const InstDesc& in = sdesc;
    const int par = lpar ^ 1, i0 = r0.p;
    for (int ph = first; ph <= last; ++ph) {
        if (ph > first && !grid_sync(gb, in.status, wait_ns)) return;
        if (ph == 1) phase_substep<true>(in, i0, D, 0, par, K == 1, sh, xs, xs2, sF, sAT, sC);
        else phase_later(in, i0, D, (ph - 1) & 1, par, ph == K, sh, xs, xs2, sF, sAT, sC);
    }
    if (last == K) {
        __syncthreads();  // records and tile ranges of the block's particles are ready
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (warp < PB && i0 + warp < in.np) append_tiles(in, i0 + warp, sAT[warp], sC[warp], lpar, lane, 32);
    }
}

// Publish every particle from its current state (after creation, particle
// insertion, a shape change or a state load).  Lists must be zeroed first.
__global__ void k_publish(const InstDesc* __restrict__ insts, const PartRef* __restrict__ refs,
                          int ntotal, int D, int lpar, Shape sh) {
    const int gp = blockIdx.x * blockDim.x + threadIdx.x;
    if (gp >= ntotal) return;
    const PartRef r = refs[gp];
    if (r.inst < 0) return;
    AxisTiles at[3];
    const Cand cd = make_record(insts[r.inst], r.p, D, sh, at, lpar);
    append_tiles(insts[r.inst], r.p, at, cd, lpar, 0, 1);
}

// Blocks of the kernel of dimension D that are resident at once (its grid barriers need all).
int particle_blocks_resident(int D, int num_sms) {
    int nb = 0;
    const cudaError_t e = D == 2 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_particles<2>, 256, 0)
                                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_particles<3>, 256, 0);
    if (e != cudaSuccess) return 0;
    return nb * num_sms;
}

// The particle part of a step: one launch with grid barriers when all blocks
// fit on the GPU at once, else one launch per phase.
cudaError_t launch_particles(const InstDesc* insts, const PartRef* refs, int ntotal, int ninst, int D, int K,
                             int lpar, const Shape& sh, GridBar* gb, bool fused, cudaStream_t st,
                             long long wait_ns) {
    const int blocks = (ntotal + PB - 1) / PB;
    const unsigned long long lim = wait_ns < 0 ? PWAIT_NS : (unsigned long long)wait_ns;
    const auto kern = D == 2 ? k_particles<2> : k_particles<3>;
    if (fused || K == 1)
        return launch_dep(kern, dim3((unsigned)blocks), 256, 0, st, insts, refs, ninst, K, 1, K, lpar, sh, gb, lim);
    for (int ph = 1; ph <= K; ++ph)
        kern<<<blocks, 256, 0, st>>>(insts, refs, ninst, K, ph, ph, lpar, sh, gb, lim);
    return cudaGetLastError();
}

cudaError_t launch_publish(const InstDesc* insts, const PartRef* refs, int ntotal, int D, int lpar,
                           const Shape& sh, cudaStream_t st) {
    k_publish<<<(ntotal + 63) / 64, 64, 0, st>>>(insts, refs, ntotal, D, lpar, sh);
    return cudaGetLastError();
}

}  // namespace lbmpen
