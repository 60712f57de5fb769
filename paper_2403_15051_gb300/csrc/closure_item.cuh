// The closure of the FDLB stage as device code shared by the closure kernel and the
// persistent step kernel.  Results per cell do not depend on how cells are grouped into items,
// nor on the number of warps above four, so both kernels produce identical records.
#pragma once

#include "device_common.cuh"
#include "kernels.cuh"
#include "kernels_decl.h"

namespace fdlb {

constexpr int kClosureThreads = 128;  // the closure kernel's block; the order of the wall sums
constexpr int kClosureWarps = kClosureThreads / 32;

// ------------------------------------------------------------------------------ closure
// Per cell, once per stage.  A cell item covers up to kClosureCells own cells and the two
// stencil cells on each side ("reach", at most 32 cells); one lane per reach cell for the
// macroscopic fields, so that no arithmetic is spread thinly over lanes:
//  * n, u, T (Eq. macro_def) of every reach cell from the FP64 raw sums, in the wide type
//    (FP64, or double-float for FP32 populations); q and P_12 of the own cells;
//  * warps 1..3 meanwhile sum the FM bands (Eq. fm, n = 0 outside the domain) from the slice
//    densities staged in shared memory; chi = chi_SET(pi sigma^3 nbar / 6) (Eqs. chi, chi_ret),
//    or chi at the local density;
//  * the J1 gradients (Eq. j1) from the differences of neighbouring reach cells (clo_pair_terms), the
//    covariant strain;
//  * mu, Pr, tau (Eqs. viscosity, prandtl, tau) and the Shakhov coefficient; the recurrences of the
//    expansion coefficients of the equilibria (Sec. III.C) and the per-axis vectors g_2, g_R, g_3.
// chi and nbar of the own cells also go to a small side buffer, from which ca_kernel forms the
// FP64 closure record of the moments and closure queries.
// Wall items (kind 1 + side, part): the block sums the outgoing flux of one part of the momenta
// at one wall; the stage kernel forms n_w from the parts (diffuse walls, zero net mass flux).
// Output: the per-cell collision record in the populations' precision, [20 scalars | g_2 | g_R
// | g_3].
__host__ __device__ inline int closure_tab_elems(int nR, int n2, int n3) {
    return (2 * (nR + n2 + n3) + 3) / 4 * 4 + (nR + n2 + n3) * kMaxE + 4 * kMaxE + 2;
}
// dynamic shared memory: [staged band rows | tables | band-union densities]
__host__ __device__ inline size_t closure_smem_bytes(int nR, int n2, int n3, int max_union, int wst_elems, int tsize) {
    return (size_t)wst_elems * tsize + ((size_t)closure_tab_elems(nR, n2, n3) + (size_t)max_union) * tsize + 16;
}

// The five-point derivative stencil of cell c in the mapped coordinate (gradients of Eq. j1; fourth
// order: central in the interior, one-sided at the two cells next to each wall) as weights of the four
// differences y[base + p + 1] - y[base + p] of its ascending cells: the weights of the values sum to
// zero, so weight p is the sum of the value weights above position p.
template <typename R>
__device__ __forceinline__ void stencil5_pairs(int c, int N, int& base, R (&w)[4]) {
    const R k = R(1) / R(12);
    if (c >= 2 && c <= N - 3) {
        base = c - 2;
        w[0] = w[3] = -k;
        w[1] = w[2] = R(7) * k;
    } else if (c < 2) {
        base = 0;
        w[0] = (c == 0 ? R(25) : R(3)) * k;
        w[1] = (c == 0 ? R(-23) : R(13)) * k;
        w[2] = (c == 0 ? R(13) : R(-5)) * k;
        w[3] = (c == 0 ? R(-3) : R(1)) * k;
    } else {
        base = N - 5;
        w[0] = (c == N - 1 ? R(-3) : R(1)) * k;
        w[1] = (c == N - 1 ? R(13) : R(-5)) * k;
        w[2] = (c == N - 1 ? R(-23) : R(13)) * k;
        w[3] = (c == N - 1 ? R(25) : R(3)) * k;
    }
}

template <typename T>
__device__ __forceinline__ T inst_param(double d, float f) {
    if constexpr (sizeof(T) == 4) return f;
    else return d;
}


template <typename T>
struct ClosureTabs {
    T *ha, *hb, *ihb, *h0t, *GR, *G2, *G3, *pRt, *wRt, *w2t, *w3t;
};

// The closure's tables in shared memory (closure_tab_elems elements from `base`), filled by the
// block's threads; the caller synchronises.  The two spans of the device table that hold them (nodes
// and weights from o_pR; equilibrium tables and recurrence from o_GR) are contiguous, so the copy is
// one loop whose loads are all in flight: table by table, each with its own wait on L2, the copy took
// 5000 cycles before every closure (cylinder, 16 x 8 x 8).
template <typename T>
__device__ ClosureTabs<T> closure_tables(T* base, const void* tabTv, const MomSet& M, int tid, int NT) {
    const int nR = M.nR, n2 = M.n2, n3 = M.n3, ng = nR + n2 + n3;
    const int nA = 2 * ng, oB = (nA + 3) / 4 * 4, nB = ng * kMaxE + 3 * kMaxE + 1;  // (rows of GR on 16 bytes)
    ClosureTabs<T> t;
    t.pRt = base;
    t.wRt = t.pRt + nR;
    t.w2t = t.wRt + nR + n2;
    t.w3t = t.w2t + n2 + n3;
    t.GR = base + oB;
    t.G2 = t.GR + nR * kMaxE;
    t.G3 = t.G2 + n2 * kMaxE;
    t.ha = t.G3 + n3 * kMaxE;
    t.hb = t.ha + kMaxE;
    t.h0t = t.hb + kMaxE + 1;
    t.ihb = base + oB + nB;  // 1 / hb
    const T* tabT = reinterpret_cast<const T*>(tabTv);
#pragma unroll 4
    for (int e = tid; e < oB + nB; e += NT) base[e] = tabT[e < oB ? M.o_pR + e : M.o_GR + e - oB];
    for (int e = tid; e <= kMaxE; e += NT) {
        const T h = tabT[M.o_hb + e];
        t.ihb[e] = h != T(0) ? T(1) / h : T(0);
    }
    return t;
}

// One thread's share of part `part` (of P) of the outgoing flux through a wall (side 0: inner,
// 1: outer): the sum over the outgoing momenta (half of the radial nodes; of the reduced pair phi's
// alone, the mass flux) of |p_R| times the WENO5 value at the wall face, from the wall cell, its
// neighbours and the cubic extrapolation outside, in the stage kernel's form (f itself, epsilon
// scaled by w^2).  `wall` points at the populations of the wall cell (cell 0 or N-1), `st` is the step
// to the next cell inward (the rows may be in global or shared memory).  `tl` is the thread's index in
// a block of kClosureThreads threads, whose order of the sums this follows.
template <typename T>
__device__ T wall_flux_partial(const T* wall, long long st, const MomSet& M, const ClosureTabs<T>& tb, int side, int part,
                               int P, int tl) {
    const int nR = M.nR, n2 = M.n2, QR = nR / 2, NT = kClosureThreads;
    const int Nout = QR * n2 * (M.reduced ? 1 : M.n3);
    const int mlo = (int)((long long)Nout * part / P), mhi = (int)((long long)Nout * (part + 1) / P);
    const T sg = side == 0 ? T(-3) : T(3), dL = side == 0 ? T(0.3) : T(0.1), dR = side == 0 ? T(0.1) : T(0.3);
    T acc = T(0);
    for (int m0 = mlo + tl; m0 < mhi; m0 += 4 * NT) {
        // four momenta per pass so that their sixteen loads are in flight together
        T fv[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int mo = m0 + u * NT;
            if (mo < mhi) {
                const int k = mo / (QR * n2), rem = mo % (QR * n2);
                const int m = k * nR * n2 + (side == 0 ? QR * n2 : 0) + rem;
#pragma unroll
                for (int r = 0; r < 4; ++r) fv[u][r] = wall[m + r * st];
            }
        }
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
            const int mo = m0 + u * NT;
            if (mo >= mhi) break;
            const int k = mo / (QR * n2), rem = mo % (QR * n2), i = (side == 0 ? QR : 0) + rem / n2, j = rem % n2;
            const T wm = mul_rn(mul_rn(tb.wRt[i], tb.w3t[k]), tb.w2t[j]), ew = mul_rn(mul_rn(T(4e-6), wm), wm);
            const T e4 = sizeof(T) == 4 ? fmax(ew, T(1e-37)) : ew;
            const T f0 = fv[0][0], f1 = fv[0][1], f2 = fv[0][2], f3 = fv[0][3];
#pragma unroll
            for (int r = 0; r < 4; ++r) {  // the next pass's populations move up
                fv[0][r] = fv[1][r];
                fv[1][r] = fv[2][r];
                fv[2][r] = fv[3][r];
            }
            const T g1 = fma(T(4), f0, fma(T(-6), f1, fma(T(4), f2, -f3)));
            const T g2 = fma(T(10), f0, fma(T(-20), f1, fma(T(15), f2, mul_rn(T(-4), f3))));
            const T vh = side == 0 ? weno5_one(g2, g1, f0, f1, f2, sg, dL, dR, e4) : weno5_one(f2, f1, f0, g1, g2, sg, dL, dR, e4);
            acc = fma(fabs(tb.pRt[i]), vh, acc);
        }
    }
    return acc;
}

// A part of the wall flux from its four warp sums, in the closure kernel's order.
template <typename T>
__device__ __forceinline__ T wall_part_sum(const T* r) {
    return (r[0] + r[1]) + (r[2] + r[3]);
}

// A part of the wall flux by one warp, in the order of the closure kernel's block of kClosureThreads
// threads: lane L takes the momenta of its threads L, L + 32, L + 64, L + 96 and the four warp sums are
// combined as there.  Lane 0 returns the part.
template <typename T>
__device__ T wall_part_of_warp(const T* fin, const MomSet& M, const ClosureTabs<T>& tb, const InstDev& I, int side, int part,
                               int P, int lane) {
    const T* wall = fin + I.f_off + (side == 0 ? 0LL : (long long)(I.n_cells - 1) * M.Np);
    T r0 = T(0), r1 = T(0), r2 = T(0), r3 = T(0);
#pragma unroll 1
    for (int vw = 0; vw < kClosureWarps; ++vw) {
        r0 = r1;
        r1 = r2;
        r2 = r3;
        r3 = warp_sum(wall_flux_partial<T>(wall, side == 0 ? (long long)M.Np : -(long long)M.Np, M, tb, side, part, P,
                                           32 * vw + lane));
    }
    const T r[kClosureWarps] = {r0, r1, r2, r3};
    return wall_part_sum(r);
}

struct NoExtra {
    __device__ void operator()(int, int) const {}
};
struct NoHook {
    __device__ void operator()() const {}
};

// ---- the per-cell steps of the closure.  The item chain below (closure_cells) and the two
// kernels of the batch form (closure_band_kernel, closure_records_kernel) are made of these
// functions, so a cell's record is the same whichever form computes it.

// Raw sums of global cell `gc` over its slices, in the wide type: FP64, or for FP32 populations
// the double-float pairs the stage kernel stores beside the FP64 sums (no FP64 arithmetic).
template <typename T>
__device__ __forceinline__ void clo_load_sums(const ClosureArgs& A, long long gc, Wide<T> (&sv)[kSums]) {
    const int slices = A.slices;
    if constexpr (sizeof(T) == 4) {
        const float2* src = reinterpret_cast<const float2*>(A.sumsw) + gc * slices * kSums;
#pragma unroll
        for (int q = 0; q < kSums; ++q) {
            const float2 p = src[q];
            sv[q] = Wide<T>{p.x, p.y};
        }
        for (int sl = 1; sl < slices; ++sl)
#pragma unroll
            for (int q = 0; q < kSums; ++q) {
                const float2 p = src[sl * kSums + q];
                sv[q] = w_add(sv[q], Wide<T>{p.x, p.y});
            }
    } else {
        const double* src = A.sums + gc * slices * kSums;
#pragma unroll
        for (int q = 0; q < kSums; ++q) sv[q] = w_from(src[q], (T*)nullptr);
        for (int sl = 1; sl < slices; ++sl)
#pragma unroll
            for (int q = 0; q < kSums; ++q) sv[q] = w_add(sv[q], w_from(src[sl * kSums + q], (T*)nullptr));
    }
}

// n, u, T of a cell (Eq. macro_def) in the wide type, and the heat flux q in the populations'
// precision (it enters only the Shakhov factor and the diagnostics).
template <typename T>
__device__ __forceinline__ void clo_fields(const Wide<T> (&sv)[kSums], Wide<T>& n, Wide<T> (&u)[3], Wide<T>& Tc,
                                           T (&q)[3]) {
    using W = Wide<T>;
    n = sv[0];
    const W tr = w_add(w_add(sv[4], sv[5]), sv[6]);
    u[0] = w_div(sv[1], n);
    u[1] = w_div(sv[2], n);
    u[2] = w_div(sv[3], n);
    T tuu;  // |u|^2, rounded once
    if constexpr (sizeof(T) == 8) {
        tuu = fma(u[0].v, u[0].v, fma(u[1].v, u[1].v, mul_rn(u[2].v, u[2].v)));
        Tc.v = fma(-n.v, tuu, tr.v) / mul_rn(T(3), n.v);
    } else {
        const W uu = w_add(w_add(w_mul(u[0], u[0]), w_mul(u[1], u[1])), w_mul(u[2], u[2]));
        Tc = w_div(w_sub(tr, w_mul(n, uu)), w_scale(n, T(3)));
        tuu = w_hi(uu);
    }
    const T tn = w_hi(n), t0 = w_hi(u[0]), t1 = w_hi(u[1]), t2 = w_hi(u[2]), ttr = w_hi(tr);
    const T nuu = mul_rn(tn, tuu);
    const T s4 = w_hi(sv[4]), s5 = w_hi(sv[5]), s6 = w_hi(sv[6]), s7 = w_hi(sv[7]), s8 = w_hi(sv[8]), s9 = w_hi(sv[9]);
    const T m0 = fma(s4, t0, fma(s7, t1, mul_rn(s8, t2)));
    const T m1 = fma(s7, t0, fma(s5, t1, mul_rn(s9, t2)));
    const T m2 = fma(s8, t0, fma(s9, t1, mul_rn(s6, t2)));
    // (S3_a - 2 m_a - u_a tr S2 + 2 n u^2 u_a) / 2
    q[0] = mul_rn(T(0.5), fma(mul_rn(T(2), nuu), t0, fma(-t0, ttr, fma(T(-2), m0, w_hi(sv[10])))));
    q[1] = mul_rn(T(0.5), fma(mul_rn(T(2), nuu), t1, fma(-t1, ttr, fma(T(-2), m1, w_hi(sv[11])))));
    q[2] = mul_rn(T(0.5), fma(mul_rn(T(2), nuu), t2, fma(-t2, ttr, fma(T(-2), m2, w_hi(sv[12])))));
}

// The FM band sum of one row (Eq. fm; a whole warp, every lane returns the sum): weights Wr[k]
// times densities dn(k), k < kmax, lane-strided into four accumulators (accumulator a takes
// k = lane + 32 a + 128 j in increasing j), then a butterfly.  The first loop takes two strides at
// a time so that sixteen loads per lane are in flight; the order of every accumulator is the same.
// Every term is an explicit fused multiply-add, so the sum does not depend on how the compiler
// contracts the expression in a given caller (clo_band_row2 must reproduce it bit for bit).
template <typename T, typename Dens>
__device__ __forceinline__ T clo_band_row(const T* Wr, const Dens& dn, int kmax, int lane) {
    T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0);
    int k = lane;
    for (; k + 224 < kmax; k += 256) {
        T w[8], d[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            w[u] = Wr[k + 32 * u];
            d[u] = dn(k + 32 * u);
        }
        a0 = fma(w[0], d[0], a0);
        a1 = fma(w[1], d[1], a1);
        a2 = fma(w[2], d[2], a2);
        a3 = fma(w[3], d[3], a3);
        a0 = fma(w[4], d[4], a0);
        a1 = fma(w[5], d[5], a1);
        a2 = fma(w[6], d[6], a2);
        a3 = fma(w[7], d[7], a3);
    }
    for (; k + 96 < kmax; k += 128) {
        a0 = fma(Wr[k], dn(k), a0);
        a1 = fma(Wr[k + 32], dn(k + 32), a1);
        a2 = fma(Wr[k + 64], dn(k + 64), a2);
        a3 = fma(Wr[k + 96], dn(k + 96), a3);
    }
    for (; k < kmax; k += 32) a0 = fma(Wr[k], dn(k), a0);
    return warp_sum((a0 + a1) + (a2 + a3));
}

// Two band rows at once by one warp, each summed exactly as clo_band_row sums it, with the loads
// of both rows in flight together.  clo_band_row's eight-wide pass is two of its four-wide passes
// in the same order, so strides of 128 alone reproduce it; a row that has left a pass adds zeros
// there, which leaves its accumulators unchanged.
template <typename T, typename DensA, typename DensB>
__device__ __forceinline__ void clo_band_row2(const T* WrA, const DensA& dnA, int kmaxA, const T* WrB, const DensB& dnB,
                                              int kmaxB, int lane, T& totA, T& totB) {
    T a0 = T(0), a1 = T(0), a2 = T(0), a3 = T(0), b0 = T(0), b1 = T(0), b2 = T(0), b3 = T(0);
    int ka = lane, kb = lane;
    for (;;) {
        const bool pa = ka + 96 < kmaxA, pb = kb + 96 < kmaxB;
        if (!pa && !pb) break;
        T wa[4], da[4], wb[4], db[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            wa[u] = pa ? WrA[ka + 32 * u] : T(0);
            da[u] = pa ? dnA(ka + 32 * u) : T(0);
            wb[u] = pb ? WrB[kb + 32 * u] : T(0);
            db[u] = pb ? dnB(kb + 32 * u) : T(0);
        }
        a0 = fma(wa[0], da[0], a0);
        a1 = fma(wa[1], da[1], a1);
        a2 = fma(wa[2], da[2], a2);
        a3 = fma(wa[3], da[3], a3);
        b0 = fma(wb[0], db[0], b0);
        b1 = fma(wb[1], db[1], b1);
        b2 = fma(wb[2], db[2], b2);
        b3 = fma(wb[3], db[3], b3);
        ka += pa ? 128 : 0;
        kb += pb ? 128 : 0;
    }
    for (;;) {
        const bool pa = ka < kmaxA, pb = kb < kmaxB;
        if (!pa && !pb) break;
        const T wa = pa ? WrA[ka] : T(0), da = pa ? dnA(ka) : T(0);
        const T wb = pb ? WrB[kb] : T(0), db = pb ? dnB(kb) : T(0);
        a0 = fma(wa, da, a0);
        b0 = fma(wb, db, b0);
        ka += pa ? 32 : 0;
        kb += pb ? 32 : 0;
    }
    totA = warp_sum((a0 + a1) + (a2 + a3));
    totB = warp_sum((b0 + b1) + (b2 + b3));
}

// R rows of at most 32 U columns (U <= 4) by one warp, each summed exactly as clo_band_row sums it, with
// the loads of all rows in flight together; every lane passes the row pointers and extents.
template <typename T, int R, int U>
__device__ __forceinline__ void clo_band_rows(const T* const (&Wr)[R], const T* const (&nd)[R], const int (&kmax)[R],
                                              int slices, int lane, T (&tot)[R]) {
    T w[R][4], d[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = lane + 32 * u;
            w[r][u] = d[r][u] = T(0);
            if (u < U && k < kmax[r]) {
                w[r][u] = Wr[r][k];
                d[r][u] = nd[r][(long long)k * slices];
                for (int sl = 1; sl < slices; ++sl) d[r][u] += nd[r][(long long)k * slices + sl];
            }
        }
#pragma unroll
    for (int r = 0; r < R; ++r) {
        // four accumulators where all four columns are in the row, else one
        T a0 = fma(w[r][0], d[r][0], T(0)), a1 = T(0), a2 = T(0), a3 = T(0);
        if (U == 4 && lane + 96 < kmax[r]) {
            a1 = fma(w[r][1], d[r][1], T(0));
            a2 = fma(w[r][2], d[r][2], T(0));
            a3 = fma(w[r][3], d[r][3], T(0));
        } else {
            a0 = fma(w[r][1], d[r][1], a0);
            if (U == 4) a0 = fma(w[r][2], d[r][2], a0);
        }
        tot[r] = warp_sum((a0 + a1) + (a2 + a3));
    }
}

// chi = chi_SET(eta), eta = etafac x (Eqs. chi, chi_ret), in the wide type, rounded once: J1
// scales with b rho chi, and near finely resolved walls J1 is large enough that a few roundings of
// chi show in the right-hand side.
template <typename T>
__device__ __forceinline__ T clo_chi(T etafac, T x) {
    using W = Wide<T>;
    const W eta = w_scale(w_from_t(x), etafac);
    const W om = w_sub(w_from_t(T(1)), eta);
    const W om3 = w_mul(w_mul(om, om), om);
    return w_hi(w_div(w_sub(w_from_t(T(2)), eta), w_scale(om3, T(2))));
}

// The reach cells' fields as a block holds them (shared memory, reach-local index).
template <typename T>
struct ReachView {
    const Wide<T>* n;
    const Wide<T>* Tc;
    const Wide<T>* u[3];
    const T* nb;
};

// Whether one of four values is below -1/8, on the bits: negative values order like their bit patterns, above
// the positive ones (an FP64 comparison would be another dependent FP64 operation).  A NaN may fall on either side.
__device__ __forceinline__ bool steep_drop(float a, float b, float c, float d) {
    return max(max(__float_as_uint(a), __float_as_uint(b)), max(__float_as_uint(c), __float_as_uint(d))) > 0xBE000000u;
}
__device__ __forceinline__ bool steep_drop(double a, double b, double c, double d) {
    return max(max((unsigned)__double2hiint(a), (unsigned)__double2hiint(b)),
               max((unsigned)__double2hiint(c), (unsigned)__double2hiint(d))) >= 0xBFC00000u;
}

// ln(n'^2 chi' T') - ln(n^2 chi T) factor by factor, each logarithm as that of a rise (beside the code of the usual
// case, whose instructions a short launch fetches cold).  n1, T1: the second cell's; dn, dT, deta: the differences.
template <typename T>
__device__ __noinline__ T clo_steep_log(T n0, T n1, T dn, T T0, T T1, T dT, T eta, T deta) {
    T sum = T(0);
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        // n and 1 / (1 - eta) enter with their powers, T and 2 - eta once
        const T p = k == 0 ? n0 : k == 1 ? T0 : k == 2 ? T(2) - eta : T(1) - eta;
        const T s = k == 0 ? n1 : k == 1 ? T1 : p - deta;
        const T dv = k == 0 ? dn : k == 1 ? dT : -deta;
        const T r = dv < T(0) ? log1p(ratio_fast(-dv, s)) : -log1p(ratio_fast(dv, p));  // ln(p / s)
        sum = fma(k == 0 ? T(-2) : k == 3 ? T(3) : T(-1), r, sum);
    }
    return sum;
}

// The terms of the J1 gradients (Eq. j1) of the neighbouring reach cells lt and lt + 1: the
// differences of ln(n^2 chi T), ln T and the three velocities.  A derivative stencil is a weighted sum
// of four such differences (stencil5_pairs), so each is formed once per pair of cells instead of once
// per cell and stencil position, with two logarithms instead of four: the ratio of n^2 chi T is the
// product of 1 + x over the factors' relative differences, and its deviation from one is carried as
// E <- E + x + E x; ln chi(eta) = ln(2 - eta) - ln 2 - 3 ln(1 - eta) from the packing-fraction difference
// alone (no rounding noise of chi itself).  The factors' differences are taken in the wide type, but a
// product well below one leaves E near -1, known to the absolute accuracy of one only (FP32: 1.3e-2 of
// the logarithm at a density ratio of 1e-3, minus infinity from 2e-4 on).  So where a factor drops by
// more than an eighth (the product of the rest is then above 0.39, and the error within three roundings),
// and where one is negative, the factors' logarithms are taken one by one, each as that of a rise.  The gradients of two cells'
// closure in FP64 took 20800 cycles with twenty logarithms per cell, a third of the whole chain in FP32.
template <typename T>
__device__ __forceinline__ void clo_pair_terms(const ReachView<T>& R, int lt, T etaf, bool chi_local, T (&d)[5]) {
    const Wide<T> nw = R.n[lt], Tw = R.Tc[lt];
    const T dn = w_hi(w_sub(R.n[lt + 1], nw));
    const T a = ratio_fast(dn, w_hi(nw)), b = ratio_fast(w_hi(w_sub(R.Tc[lt + 1], Tw)), w_hi(Tw));
    const T eta = mul_rn(etaf, chi_local ? w_hi(nw) : R.nb[lt]);
    const T deta = mul_rn(etaf, chi_local ? dn : R.nb[lt + 1] - R.nb[lt]);
    const T x = ratio_fast(-deta, T(2) - eta);               // (2 - eta') / (2 - eta) - 1
    const T y = ratio_fast(deta, (T(1) - eta) - deta);        // (1 - eta) / (1 - eta') - 1
    T E = fma(a, a, mul_rn(T(2), a));                                // (1 + a)^2 - 1
    E = fma(E, b, E + b);
    E = fma(E, x, E + x);
    E = fma(E, y, E + y);
    E = fma(E, y, E + y);
    E = fma(E, y, E + y);
    d[0] = log1p(E);
    d[1] = log1p(b);
    if (__builtin_expect(steep_drop(a, b, x, y), 0)) {
        d[0] = clo_steep_log<T>(w_hi(nw), w_hi(R.n[lt + 1]), dn, w_hi(Tw), w_hi(R.Tc[lt + 1]), w_hi(w_sub(R.Tc[lt + 1], Tw)), eta, deta);
    }
    d[2] = w_hi(w_sub(R.u[0][lt + 1], R.u[0][lt]));
    d[3] = w_hi(w_sub(R.u[1][lt + 1], R.u[1][lt]));
    d[4] = w_hi(w_sub(R.u[2][lt + 1], R.u[2][lt]));
}

// The collision record's 20 scalars of an own cell, in two independent halves (entry 0, the density of
// f^MB, follows with the equilibrium vectors).  The transport half: u, 1/T, 1/tau (Eq. tau, mu from Eq. viscosity), the Shakhov coefficient (Eq. prandtl), q and
// -b rho chi.  With x = b rho chi and P(x) = 1 + 4/5 x + 4/25 (1 + 12/pi) x^2, mu is mu0 P / chi and the
// Prandtl number 2/3 P / Q, so the two share P and 1/tau = n sqrt(T) chi (16 sigma^2 sqrt(pi) / 5) / P.
template <typename T>
__device__ __forceinline__ void clo_record_transport(T* ct, Wide<T> nw, T cu0, T cu1, T cu2, T cT, T cchi, const T (&q)[3],
                                                     const InstDev& I) {
    using C = T;
    const C cn = w_hi(nw);
    const C in = ratio_fast(C(1), cn), iT = ratio_fast(C(1), cT);
    const C sg = inst_param<C>(I.sigma, I.f_sigma);
    const C x = mul_rn(mul_rn(inst_param<C>(I.bfac, I.f_bfac), cn), cchi);
    constexpr double pi = 3.14159265358979323846;
    const C P = fma(x, fma(C(4.0 / 25.0 * (1.0 + 12.0 / pi)), x, C(0.8)), C(1));
    const C Q = fma(x, fma(C(9.0 / 25.0 * (1.0 + 32.0 / (9.0 * pi))), x, C(1.2)), C(1));
    const C Pr1 = fma(C(-2.0 / 3.0), ratio_fast(P, Q), C(1));  // 1 - Pr
    ct[1] = cu0;
    ct[2] = cu1;
    ct[3] = cu2;
    ct[4] = iT;
    ct[5] = ratio_fast(mul_rn(mul_rn(mul_rn(cn, sqrt(cT)), cchi), mul_rn(mul_rn(C(5.671852322897651), sg), sg)), P);
    ct[6] = mul_rn(mul_rn(mul_rn(Pr1, iT), iT), in);
    ct[7] = q[0];
    ct[8] = q[1];
    ct[9] = q[2];
    ct[10] = -x;
}

// The gradient half: X = d ln(n^2 chi T), Y = d ln T, the radial velocity's derivative, the covariant
// strain (cylinder / sphere) and its divergence (Eq. j1).  Products the stage kernel would otherwise
// form per cell and thread are stored in place of their factors that it uses nowhere else:
// 0.4 S_11 / T in place of S_11, 2 S_01 / T in place of S_01, 1 / (2T) in the spare slot 18.
// gp[v]: the pair terms of the reach (32 per term); base - h0: the stencil's first pair.
template <typename T>
__device__ __forceinline__ void clo_record_gradients(T* ct, int c, int N, int h0, const T (*gp)[32], T cu0, T cu1, T cu2,
                                                     T cT, T geo0, T geo1, const InstDev& I) {
    using C = T;
    const C iT = ratio_fast(C(1), cT), iR = ratio_fast(C(1), geo0);
    const C sc = mul_rn(geo1, inst_param<C>(1.0 / I.ds, I.f_ids));
    int base;
    C w[4];
    stencil5_pairs<C>(c, N, base, w);
    base -= h0;
    C g[5];
#pragma unroll
    for (int v = 0; v < 5; ++v)
        g[v] = mul_rn(sc, fma(w[3], gp[v][base + 3], fma(w[2], gp[v][base + 2], fma(w[1], gp[v][base + 1], mul_rn(w[0], gp[v][base])))));
    const C S11 = mul_rn(cu0, iR), S22 = I.geometry == 0 ? C(0) : S11;
    const C S01 = mul_rn(C(0.5), fma(-cu1, iR, g[3]));
    const C S02 = mul_rn(C(0.5), I.geometry == 0 ? g[4] : fma(-cu2, iR, g[4]));
    const C div = I.geometry == 0 ? g[2] + S11 : fma(C(2), S11, g[2]);
    ct[11] = g[0];
    ct[12] = g[1];
    ct[13] = g[2];
    ct[14] = mul_rn(mul_rn(T(0.4), iT), S11);
    ct[15] = S22;
    ct[16] = mul_rn(mul_rn(T(2), iT), S01);
    ct[17] = S02;
    ct[18] = mul_rn(T(0.5), iT);
    ct[19] = div;
}

// Expansion coefficients of one equilibrium factor of an own cell (Sec. III.C); job 0 / 1: the
// half-range axis on the half line of sign + / -, job 2 / 3: the full-range axes 2 / 3.  cT, tm1
// = T - 1 (without cancellation), ur = u_R, ua = u_2 (job 2) or u_3 (job 3).
template <typename T>
__device__ __forceinline__ void clo_eq_coeffs(int job, T cT, T tm1, T ur, T ua, const ClosureTabs<T>& tb,
                                              const MomSet& M, T (&ev)[kMaxE + 1]) {
    using C = T;
    const T *ha = tb.ha, *hb = tb.hb, *ihb = tb.ihb, *h0t = tb.h0t;
#pragma unroll
    for (int l = 0; l <= kMaxE; ++l) ev[l] = C(0);
    if (job < 2) {
        // half range, half line of sign s (job 0: +, 1: -), v = s u_R.  The recurrence of the
        // coefficients,
        //   e_0 = h_0 (1 + erf(v / sqrt(2T))) / 2,
        //   b_{l+1} e_{l+1} = (v - a_l) e_l + (T - 1) b_l e_{l-1}
        //                     + T h_l(0) [G_v(0) - sum_{k<l} h_k(0) e_k / sqrt(2 pi)],
        // is run for the deviation d_l = e_l - r_l from the rest state (v = 0, T = 1: r_0 = h_0 / 2,
        // r_l = 0 for l >= 1), where every term is small and nothing cancels: with
        // D = sqrt(2 pi) G_v(0) - 1 = (expm1(-z^2) - (T - 1)/(1 + sqrt T)) / sqrt T, z = v / sqrt(2T),
        // and h_0(0) r_0 = 1,
        //   d_0 = h_0 erf(z) / 2,
        //   b_1 d_1 = v r_0 + (v - a_0) d_0 + h_0 [(T - 1) + T D] / sqrt(2 pi),
        //   b_{l+1} d_{l+1} = (v - a_l) d_l + (T - 1) b_l e_{l-1}
        //                     + T h_l(0) [D - sum_{k<l} h_k(0) d_k] / sqrt(2 pi).
        const C v = job == 0 ? ur : -ur;
        const C sT = sqrt(cT), z = mul_rn(ur, rsqrt(mul_rn(C(2), cT)));  // (odd in z: the two halves share erf)
        const C D = (expm1(mul_rn(-z, z)) - tm1 / (C(1) + sT)) / sT;
        const C ez = erf(z);
        const C is2pi = C(0.39894228040143267794);
        const C r0 = mul_rn(h0t[0], C(0.5));
        C d[kMaxE + 1];
#pragma unroll
        for (int l = 0; l <= kMaxE; ++l) d[l] = C(0);
        d[0] = mul_rn(r0, job == 0 ? ez : -ez);
        C run = C(0);  // sum_{k<l} h_k(0) d_k
#pragma unroll
        for (int l = 0; l < kMaxE; ++l) {
            if (l < M.NR) {
                C val;
                if (l == 0) {
                    val = fma(v - ha[0], d[0], fma(v, r0, mul_rn(mul_rn(h0t[0], fma(cT, D, tm1)), is2pi)));
                } else {
                    const C em1 = (l == 1 ? r0 : C(0)) + d[l > 0 ? l - 1 : 0];
                    val = fma(v - ha[l], d[l], fma(mul_rn(tm1, hb[l]), em1, mul_rn(mul_rn(cT, h0t[l]), mul_rn(D - run, is2pi))));
                }
                run = fma(h0t[l], d[l], run);
                d[l + 1] = mul_rn(val, ihb[l + 1]);
            }
        }
#pragma unroll
        for (int l = 0; l <= kMaxE; ++l) ev[l] = d[l];
        ev[0] += r0;
    } else {
        // full range: e_l = E[He_l(X)], X ~ N(u, T): e_{l+1} = u e_l + l (T - 1) e_{l-1}
        const int Nax = job == 2 ? M.N2 : M.N3;
        ev[0] = C(1);
        ev[1] = Nax >= 1 ? ua : C(0);
#pragma unroll
        for (int l = 1; l < kMaxE; ++l)
            if (l < Nax) ev[l + 1] = fma(ua, ev[l], mul_rn(mul_rn(C(l), tm1), ev[l - 1]));
    }
}

// The expansion coefficients of an item's own cells, [job][l][cell]: consecutive cells on consecutive
// banks for the lane-per-cell writes.
constexpr int kEcsCells = kClosureCells + 1;
template <typename T>
struct EqCoeffs {
    T v[4][kMaxE][kEcsCells];
};

// The per-axis equilibrium vectors g_R, g_2, g_3 of an own cell into its record, and the density
// stored for f^MB, by eight lanes (sub = 0..7, aligned in the warp; every lane of the warp calls, `on`
// false where there is no cell): two lanes for each job of clo_eq_coeffs (equal shares for equal
// orders), each holding the job's coefficients and summing its stored entries in the wide type as it
// forms them.  The rounded vectors need not sum to exactly one per axis, and for FP32 populations that
// bias, times dt / tau every step, would make the total mass drift: the density for f^MB = n g_R g_2 g_3
// is the wide n divided by the wide product of the three sums; lane sub = 0 returns it.  ec: the item's
// coefficients, t: the cell's place in them; cT its temperature (the reduced pair's chi factor).  (Entries
// by one thread each and then a thread per cell reading them all back cost 4000 cycles of 17600 in the
// cylinder's closure.)
template <typename T>
__device__ __forceinline__ T clo_equilibrium(bool on, int sub, T* ct, Wide<T> n, T cT, const EqCoeffs<T>& ec, int t,
                                             const ClosureTabs<T>& tb, const MomSet& M) {
    using W = Wide<T>;
    const int nR = M.nR, n2 = M.n2, QR = nR / 2;
    const int job = sub >> 1;
    const int len = job < 2 ? QR : job == 2 ? n2 : M.n3;
    const int N = job < 2 ? M.NR : job == 2 ? M.N2 : M.N3;
    const T* G = job < 2 ? tb.GR + job * QR * kMaxE : job == 2 ? tb.G2 : tb.G3;
    T* dst = ct + (job < 2 ? rec_off_gR(n2) + job * QR : job == 2 ? rec_off_g2() : rec_off_g3(nR, n2));
    const bool pair = job == 3 && M.reduced;  // the pair's factors: int g_z = 1 (phi), int p_z^2 g_z = T (chi)
    W sum = w_from_t(T(0));
    if (on) {
        // (the expansion orders are at most kMaxE - 1: the coefficients beyond are zero)
        T e[kMaxE];
#pragma unroll
        for (int l = 0; l < kMaxE; ++l) e[l] = l <= N ? ec.v[job][l][t] : T(0);
        for (int k = sub & 1; k < len; k += 2) {
            T g[kMaxE];
            if constexpr (sizeof(T) == 4) {
                const float4 x = reinterpret_cast<const float4*>(G + k * kMaxE)[0], y = reinterpret_cast<const float4*>(G + k * kMaxE)[1];
                g[0] = x.x; g[1] = x.y; g[2] = x.z; g[3] = x.w; g[4] = y.x; g[5] = y.y; g[6] = y.z; g[7] = y.w;
            } else {
#pragma unroll
                for (int l = 0; l < kMaxE; ++l) g[l] = G[k * kMaxE + l];
            }
            T acc = T(0);
#pragma unroll
            for (int l = 0; l < kMaxE; ++l)
                if (l <= N) acc = fma(g[l], e[l], acc);
            if (pair) acc = k == 0 ? T(1) : cT;
            dst[k] = acc;
            if (!pair || k == 0) sum = w_add(sum, w_from_t(acc));  // (the pair's mass is phi's)
        }
    }
    sum = w_add(sum, w_shfl_xor(sum, 1));
    const W r2 = w_shfl_xor(sum, 2);
    // lanes 0..3: g_R's two halves added; lanes 4..7: the product of the two full-range sums
    const W s = job < 2 ? w_add(sum, r2) : w_mul(sum, r2);
    const W p23 = w_shfl_xor(s, 4);
    return w_hi(w_div(n, w_mul(s, p23)));
}

// Reach of an item of own cells [c0, c0 + cnt) of an instance of N cells: the own cells, two on
// each side (the gradient stencils), and the five cells next to a wall.
__device__ __forceinline__ void clo_reach(int c0, int cnt, int N, int& h0, int& h1) {
    h0 = max(0, min(c0 - 2, N - 5));
    h1 = min(N, max(c0 + cnt + 2, 5));
}

// Closure of the own cells [c0, c0 + cnt) of one instance (cnt <= kClosureCells): the collision
// records go to `recb` (the record of cell c0, stride A.rec_stride), chi and nbar to A.cw.
// Every thread of the block calls it (it holds block barriers); the block has at least
// kClosureWarps warps, and warps beyond them run extra(w, nw) (the w-th of nw such warps)
// while the closure's own run the chains of step 3; every thread runs before_loads() once the item's
// constants (geometry, band extents and rows) are requested and before it reads what the previous
// kernel wrote, and after_loads() once the item's global loads are issued.  `wst` holds A.wst_elems staged band elements, `nbuf`
// A.max_union densities.  Returns false on every thread when the band-row copy never
// completed (A.err is set).
template <typename T, typename Extra, typename BeforeLoads, typename AfterLoads>
__device__ bool closure_cells(const ClosureArgs& A, const MomSet& M, const ClosureTabs<T>& tb, const InstDev& I, int c0,
                              int cnt, T* recb, T* wst, T* nbuf, uint64_t* cbar, uint32_t& phase, const Extra& extra,
                              const BeforeLoads& before_loads, const AfterLoads& after_loads) {
    using W = Wide<T>;
    __shared__ W sw_n[32], sw_T[32], sw_u[3][32];  // reach cells, wide
    __shared__ T snb[32];                          // reach cells: band density
    __shared__ int sblo[32], scnt[32];             // reach cells: first band column, stored extent
    __shared__ T sq[3][32];                        // own cells: q
    __shared__ EqCoeffs<T> ecs;                    // own cells: expansion coefficients
    __shared__ T sgp[5][32];                       // gradient terms per pair of neighbouring reach cells
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, NT = blockDim.x;
    const T* band = reinterpret_cast<const T*>(A.band);
    const T* dens = reinterpret_cast<const T*>(A.dens);
    const T* geoT = reinterpret_cast<const T*>(A.geoT);
    const int slices = A.slices;
    const int N = I.n_cells;
    int h0, h1;
    clo_reach(c0, cnt, N, h0, h1);
    const int nh = h1 - h0;
    const int rs = A.rec_stride;
    const ReachView<T> RV{sw_n, sw_T, {sw_u[0], sw_u[1], sw_u[2]}, snb};
    // ---- 1. the constants: the geometry of the own cells (lane per cell of warp 0) and, by bulk
    // copies issued by warp 0, the band rows of the reach cells (their stored extents); then, past
    // before_loads(), every load of the previous kernel's output at once: the raw sums of the reach
    // cells (lane per cell of warp 0) and the densities of the union of the bands (all threads)
    W sv[kSums];
    T geo0 = T(1), geo1 = T(0);
    if (warp == 0 && lane < cnt) {
        const T* gc = geoT + (long long)(I.cell_off + c0 + lane) * kGeo;
        geo0 = gc[0];
        geo1 = gc[1];
    }
    int jlo = 0, nu = 0;
    const bool staged = !I.chi_local && nh * I.band_w <= A.wst_elems;
    if (!I.chi_local) {
        const int2* bl = reinterpret_cast<const int2*>(A.band_lo) + I.cell_off;
        const int2 first = bl[h0], last = bl[h1 - 1];
        jlo = first.x;
        // columns grow with the row, and extents are rounded up by at most 3
        const int jhi = min(N - 1, last.x + last.y - 1 + 3);
        nu = min(jhi - jlo + 1, A.max_union);
        if (warp == 0) {
            int2 mine = make_int2(0, 0);
            if (lane < nh) mine = bl[h0 + lane];
            if (lane < nh) {
                sblo[lane] = mine.x;
                scnt[lane] = mine.y;
            }
            if (staged) {
                // one bulk copy per row, of its stored extent (a multiple of 16 bytes)
                int bytes = lane < nh ? mine.y * (int)sizeof(T) : 0;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) bytes += __shfl_xor_sync(0xffffffffu, bytes, o);
                if (lane == 0) {
                    fence_proxy_async();
                    mbar_expect_tx(cbar, (uint32_t)bytes);
                }
                __syncwarp();
                if (lane < nh && mine.y > 0)
                    bulk_g2s(wst + (long long)lane * I.band_w, band + I.band_off + (long long)(h0 + lane) * I.band_w,
                             (uint32_t)(mine.y * sizeof(T)), cbar);
            }
        }
    }
    before_loads();
    if (warp == 0 && lane < nh) clo_load_sums<T>(A, (long long)I.cell_off + h0 + lane, sv);
    if (!I.chi_local) {
        const T* nd = dens + ((long long)I.cell_off + jlo) * slices;
        for (int j0 = tid; j0 < nu; j0 += 4 * NT) {
            // four loads in flight per thread
            T v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = min(j0 + u * NT, nu - 1);
                v[u] = nd[(long long)j * slices];
                for (int sl = 1; sl < slices; ++sl) v[u] += nd[(long long)j * slices + sl];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (j0 + u * NT < nu) nbuf[j0 + u * NT] = v[u];
        }
    }
    after_loads();
    if (staged) {
        const bool ok = mbar_wait_bounded(cbar, phase);
        // every thread takes the same exit: a block-wide vote on the outcome
        if (__syncthreads_or(!ok)) {
            if (tid == 0) atomicOr(A.err, 2);
            mbar_wait_bounded(cbar, phase);  // bounded wait for the copy still in flight
            return false;
        }
        phase ^= 1u;
    } else {
        __syncthreads();  // staged: the vote above is the barrier
    }
    // ---- 2. warp 0: n, u, T of the reach cells (wide), q of the own cells; the other warps: FM
    // band sums of the reach cells from shared memory
    if (warp == 0) {
        if (lane < nh) {
            const int c = h0 + lane;
            W n, u[3], Tc;
            T q[3];
            clo_fields<T>(sv, n, u, Tc, q);
            sw_n[lane] = n;
            sw_u[0][lane] = u[0];
            sw_u[1][lane] = u[1];
            sw_u[2][lane] = u[2];
            sw_T[lane] = Tc;
            if (c >= c0 && c < c0 + cnt) {
                sq[0][c - c0] = q[0];
                sq[1][c - c0] = q[1];
                sq[2][c - c0] = q[2];
            }
        }
    } else if (!I.chi_local) {
        // one warp per row, every warp but the first (the row's sum does not depend on which)
        for (int t = warp - 1; t < nh; t += NT / 32 - 1) {
            const int c = h0 + t;
            const int lo = sblo[t];
            const int kmax = min(min(scnt[t], N - lo), nu - (lo - jlo));
            const T* Wr = staged ? wst + (long long)t * I.band_w : band + I.band_off + (long long)c * I.band_w;
            const T* nb = nbuf + (lo - jlo);
            const T tot = clo_band_row<T>(Wr, [&](int k) { return nb[k]; }, kmax, lane);
            if (lane == 0) snb[t] = tot;
        }
    }
    __syncthreads();
    // ---- 3. concurrent chains.  Warp 0: the gradient terms (lane per pair of neighbouring reach
    // cells), then the own cells' gradients and strain.  Warp 3: chi, transport and Shakhov coefficient
    // (lane per own cell).  Warps 1 and 2: the expansion coefficients of the equilibria (Sec. III.C),
    // lane per (own cell, axis half): warp 1 the half-range axis (+ and -), warp 2 the axes 2 and 3.
    const T etaf = inst_param<T>(I.etafac, I.f_etafac);
    if (warp == 0) {
        if (lane < nh - 1) {
            T d[5];
            clo_pair_terms<T>(RV, lane, etaf, I.chi_local != 0, d);
#pragma unroll
            for (int v = 0; v < 5; ++v) sgp[v][lane] = d[v];
        }
        __syncwarp();
        if (lane < cnt) {
            const int lt = c0 + lane - h0;
            clo_record_gradients<T>(recb + (long long)lane * rs, c0 + lane, N, h0, sgp, w_hi(sw_u[0][lt]), w_hi(sw_u[1][lt]),
                                    w_hi(sw_u[2][lt]), w_hi(sw_T[lt]), geo0, geo1, I);
        }
    } else if (warp <= 2) {
        for (int e = lane; e < 2 * cnt; e += 32) {
            const int t = e % cnt, job = 2 * (warp - 1) + e / cnt, lt = c0 + t - h0;
            const T cT = w_hi(sw_T[lt]);
            const T tm1 = w_hi(w_sub(sw_T[lt], w_from_t(T(1))));  // T - 1 without cancellation
            T ev[kMaxE + 1];
            clo_eq_coeffs<T>(job, cT, tm1, w_hi(sw_u[0][lt]), w_hi(sw_u[job == 2 ? 1 : 2][lt]), tb, M, ev);
#pragma unroll
            for (int l = 0; l < kMaxE; ++l) ecs.v[job][l][t] = ev[l];
        }
    } else if (warp == 3) {
        if (lane < cnt) {
            const int lt = c0 + lane - h0;
            const T q[3] = {sq[0][lane], sq[1][lane], sq[2][lane]};
            const T nb = I.chi_local ? w_hi(sw_n[lt]) : snb[lt], chi = clo_chi<T>(etaf, nb);
            clo_record_transport<T>(recb + (long long)lane * rs, sw_n[lt], w_hi(sw_u[0][lt]), w_hi(sw_u[1][lt]),
                                    w_hi(sw_u[2][lt]), w_hi(sw_T[lt]), chi, q, I);
            T* cw = reinterpret_cast<T*>(A.cw) + (long long)(I.cell_off + c0 + lane) * 2;
            cw[0] = chi;
            cw[1] = nb;
        }
    } else {
        extra(warp - kClosureWarps, NT / 32 - kClosureWarps);
    }
    __syncthreads();
    // ---- 4. the equilibrium vectors and the normalised density (eight lanes per own cell)
    for (int e = tid; e < (8 * cnt + 31) / 32 * 32; e += NT) {
        const int t = min(e >> 3, cnt - 1), lt = c0 + t - h0;
        const bool on = (e >> 3) < cnt;
        const T nf = clo_equilibrium<T>(on, e & 7, recb + (long long)t * rs, sw_n[lt], w_hi(sw_T[lt]), ecs, t, tb, M);
        if (on && (e & 7) == 0) recb[(long long)t * rs] = nf;
    }
    __syncthreads();  // shared arrays are reused by the next call
    return true;
}

}  // namespace fdlb
