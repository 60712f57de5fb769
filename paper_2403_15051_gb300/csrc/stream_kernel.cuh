// The fused stage kernel: one SSP-RK3 stage for a run of radial cells x one momentum slice.
//
// Per work item (instance, first cell c0, cells Be, slice sl) a team (the block, or for small momentum
// sets a warp of it) marches along the radius with the rows (the slice's populations of a cell) in a
// ring in shared memory:
//  1. the TMA engine copies the rows of cells c0-3 .. c0+G+2 and the first G collision records (written
//     by the closure kernel; a block's first rows before its dependency wait, the records after it);
//     then, while each group of G cells is computed, the next group's rows and records;
//  2. rows beyond the walls are filled as the march reaches them: incoming directions carry n_w times
//     the wall Maxwellian, outgoing directions the cubic extrapolation of the four cells next to
//     the wall (each thread its own momenta);
//  3. per population: WENO5 face values of f/w upwinded by sign(p_R), conservative advection
//     with the face areas and cell volume (Sec. II.B/C), the curvature force with the K matrices
//     (Sec. III.B), the Shakhov + J1 collision (Eqs. j0, j1), the RK combination and the store;
//  4. the 13 raw sums of the new populations per cell: per-thread partials, a transposing warp
//     reduction in the populations' precision, across the warps one group later in a
//     fixed tree (double-float for FP32 populations, FP64 for FP64), stored as FP64 sums and, for
//     FP32 populations, as the double-float pairs the closure reads.
// A cell's results do not depend on the item it is in, nor on G.
//
// Thread mapping: a "vector" is VW momenta with the same (k, i) and consecutive j, which are
// contiguous in the [k][i][j] layout.  A thread owns up to NV vectors for the whole kernel, so
// every shared-memory access is a VW-wide load: the five WENO rows, the column of the K^h
// contraction (shared by the VW momenta), the row of the K_2 contraction and, from K_2 stored
// transposed, each input's coefficients for the vector's outputs.  All momenta of a vector share
// p_R and hence the upwind direction.  A vector's momenta are processed in pairs of lanes (packed
// FP32x2 operations for FP32 populations), every operation written out, so that a lane's result
// does not depend on the pairing.
#pragma once

#include <type_traits>

#include "device_common.cuh"
#include "kernels_decl.h"

namespace fdlb {

// Outgoing-direction ghost values (cubic extrapolation in the cell index) from the four
// populations next to a wall, f0 being the wall cell.
template <typename T>
__device__ __forceinline__ void wall_ghosts(T f0, T f1, T f2, T f3, T& g1, T& g2) {
    g1 = fma(T(4), f0, fma(T(-6), f1, fma(T(4), f2, -f3)));
    g2 = fma(T(10), f0, fma(T(-20), f1, fma(T(15), f2, mul_rn(T(-4), f3))));
}

// VW consecutive elements (16-byte aligned for VW * sizeof(T) >= 16; 8-byte for float2).
template <typename T, int VW>
__device__ __forceinline__ void ld_vec(const T* p, T (&o)[VW]) {
    if constexpr (sizeof(T) == 4 && VW % 4 == 0) {
#pragma unroll
        for (int h = 0; h < VW / 4; ++h) {
            const float4 x = reinterpret_cast<const float4*>(p)[h];
            o[4 * h] = x.x; o[4 * h + 1] = x.y; o[4 * h + 2] = x.z; o[4 * h + 3] = x.w;
        }
    } else if constexpr (sizeof(T) == 4 && VW == 2) {
        const float2 x = *reinterpret_cast<const float2*>(p);
        o[0] = x.x; o[1] = x.y;
    } else if constexpr (sizeof(T) == 8 && VW >= 2) {
#pragma unroll
        for (int h = 0; h < VW / 2; ++h) {
            const double2 x = *reinterpret_cast<const double2*>(p + 2 * h);
            o[2 * h] = x.x; o[2 * h + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < VW; ++e) o[e] = p[e];
    }
}

template <typename T, int VW>
__device__ __forceinline__ void ldg_vec(const T* p, T (&o)[VW]) {
    if constexpr (sizeof(T) == 4 && VW % 4 == 0) {
#pragma unroll
        for (int h = 0; h < VW / 4; ++h) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p) + h);
            o[4 * h] = x.x; o[4 * h + 1] = x.y; o[4 * h + 2] = x.z; o[4 * h + 3] = x.w;
        }
    } else if constexpr (sizeof(T) == 4 && VW == 2) {
        const float2 x = __ldg(reinterpret_cast<const float2*>(p));
        o[0] = x.x; o[1] = x.y;
    } else if constexpr (sizeof(T) == 8 && VW >= 2) {
#pragma unroll
        for (int h = 0; h < VW / 2; ++h) {
            const double2 x = __ldg(reinterpret_cast<const double2*>(p + 2 * h));
            o[2 * h] = x.x; o[2 * h + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < VW; ++e) o[e] = __ldg(p + e);
    }
}

// The same through L2 only (data written earlier in the same launch by other blocks).
template <typename T, int VW>
__device__ __forceinline__ void ldcg_vec(const T* p, T (&o)[VW]) {
    if constexpr (sizeof(T) == 4 && VW % 4 == 0) {
#pragma unroll
        for (int h = 0; h < VW / 4; ++h) {
            const float4 x = __ldcg(reinterpret_cast<const float4*>(p) + h);
            o[4 * h] = x.x; o[4 * h + 1] = x.y; o[4 * h + 2] = x.z; o[4 * h + 3] = x.w;
        }
    } else if constexpr (sizeof(T) == 4 && VW == 2) {
        const float2 x = __ldcg(reinterpret_cast<const float2*>(p));
        o[0] = x.x; o[1] = x.y;
    } else if constexpr (sizeof(T) == 8 && VW >= 2) {
#pragma unroll
        for (int h = 0; h < VW / 2; ++h) {
            const double2 x = __ldcg(reinterpret_cast<const double2*>(p + 2 * h));
            o[2 * h] = x.x; o[2 * h + 1] = x.y;
        }
    } else {
#pragma unroll
        for (int e = 0; e < VW; ++e) o[e] = __ldcg(p + e);
    }
}

template <typename T, int VW>
__device__ __forceinline__ void st_vec(T* p, const T (&o)[VW]) {
    if constexpr (sizeof(T) == 4 && VW % 4 == 0) {
#pragma unroll
        for (int h = 0; h < VW / 4; ++h)
            reinterpret_cast<float4*>(p)[h] = make_float4(o[4 * h], o[4 * h + 1], o[4 * h + 2], o[4 * h + 3]);
    } else if constexpr (sizeof(T) == 4 && VW == 2) {
        *reinterpret_cast<float2*>(p) = make_float2(o[0], o[1]);
    } else if constexpr (sizeof(T) == 8 && VW >= 2) {
#pragma unroll
        for (int h = 0; h < VW / 2; ++h) *reinterpret_cast<double2*>(p + 2 * h) = make_double2(o[2 * h], o[2 * h + 1]);
    } else {
#pragma unroll
        for (int e = 0; e < VW; ++e) p[e] = o[e];
    }
}

// A vector as (VW + 1) / 2 pairs of lanes: (e0, e1), (e2, e3), ...; for VW = 1 one pair whose
// second lane repeats the first (computed alongside and never stored).  The loads go through the
// VW-wide forms above, whose registers the pairs then name without a move.
template <typename T, int VW>
__device__ __forceinline__ void pairs_of(const T (&v)[VW], Pair<T> (&o)[(VW + 1) / 2]) {
#pragma unroll
    for (int h = 0; h < (VW + 1) / 2; ++h) o[h] = p_make(v[2 * h], v[VW == 1 ? 0 : 2 * h + 1]);
}
template <typename T, int VW>
__device__ __forceinline__ void ld_pairs(const T* p, Pair<T> (&o)[(VW + 1) / 2]) {
    T v[VW];
    ld_vec<T, VW>(p, v);
    pairs_of<T, VW>(v, o);
}
template <typename T, int VW>
__device__ __forceinline__ void ldg_pairs(const T* p, Pair<T> (&o)[(VW + 1) / 2]) {
    T v[VW];
    ldg_vec<T, VW>(p, v);
    pairs_of<T, VW>(v, o);
}
template <typename T, int VW>
__device__ __forceinline__ void ldcg_pairs(const T* p, Pair<T> (&o)[(VW + 1) / 2]) {
    T v[VW];
    ldcg_vec<T, VW>(p, v);
    pairs_of<T, VW>(v, o);
}
template <typename T, int VW>
__device__ __forceinline__ void st_pairs(T* p, const Pair<T> (&o)[(VW + 1) / 2]) {
    T v[VW];
#pragma unroll
    for (int h = 0; h < (VW + 1) / 2; ++h) {
        v[2 * h] = o[h].x;
        if (2 * h + 1 < VW) v[2 * h + 1] = o[h].y;
    }
    st_vec<T, VW>(p, v);
}

// Sizes of the stage (NR_, N2_, N3_: compile-time axis sizes, 0: taken from M at run time) and its team:
// a warp of the block where A.teams > 1 (generic kernels), else the block.  The sphere couples every
// axis: one slice (KS = n3), unless K_3 f comes from its own contraction kernel (A.k3f).
#define FDLB_STAGE_SIZES                                                                                         \
    constexpr bool kTeam = NR_ == 0;                                                                             \
    const bool warps_apart = kTeam && A.teams > 1;                                                               \
    const int NT = warps_apart ? 32 : (int)blockDim.x;                                                           \
    const int lane = threadIdx.x & 31;                                                                           \
    const int tid = warps_apart ? lane : (int)threadIdx.x;                                                       \
    const int warp = warps_apart ? 0 : (int)threadIdx.x >> 5, nwarps = NT >> 5;                                  \
    const int nR = NR_ ? NR_ : M.nR, n2 = N2_ ? N2_ : M.n2, n3 = N3_ ? N3_ : M.n3;                               \
    const int KS = M.KS;                                                                                         \
    const int Ms = nR * n2 * KS, Np = nR * n2 * n3;                                                              \
    const int n2v = n2 / VW;                                                                                     \
    const int Vs = Ms / VW;                                                                                      \
    const int rs = record_stride(nR, n2, n3);                                                                    \
    const int gwstride = nR + n2 + n3;                                                                           \
    (void)tid, (void)warp, (void)nwarps, (void)Np, (void)n2v, (void)Vs, (void)rs, (void)gwstride, (void)lane

// Where a team's data lie in shared memory: the copy barrier, the wall densities, the rows (fs), the
// records, the wall Maxwellians [2][nR + n2 + n3], the cells' geometry and the per-warp sums
// [cell][warp][16]; of the block: the tables (p2 first and K_2 transposed, [b][j], for aligned vector
// loads: the coefficients of input b for a vector's outputs; K^h with row stride kr_stride, K_3 with row
// stride n3 + 1); skr: K^h f of the own cells (mma.sync path).
template <typename T>
struct StagePtrs {
    uint64_t* bar;
    T *nw, *fs, *rec, *gw, *geo, *red, *skr;
    T *p2, *K2, *KR, *K3, *pR, *p3, *wR, *w2, *w3;
};
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_table_ptrs(StagePtrs<T>& S, T* base, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    S.p2 = base;
    S.K2 = S.p2 + p2_span(n2);
    S.KR = S.K2 + kr_offset(n2, (int)sizeof(T));
    S.K3 = S.KR + (A.krf ? 0 : nR) * kr_stride(nR);
    S.pR = S.K3 + n3 * (n3 + 1);
    S.p3 = S.pR + nR;
    S.wR = S.p3 + n3;
    S.w2 = S.wR + nR;
    S.w3 = S.w2 + n2;
}
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ StagePtrs<T> march_ptrs(unsigned char* smem, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    const MarchSmem P = march_smem_plan(A.G, Ms, nR, n2, n3, nwarps, (int)sizeof(T), A.krf ? 1 : 0);
    unsigned char* t = smem + P.teams + (warps_apart ? (threadIdx.x >> 5) * P.team_bytes : 0);
    StagePtrs<T> S;
    S.bar = reinterpret_cast<uint64_t*>(t);
    S.nw = reinterpret_cast<T*>(t + 16);
    S.fs = reinterpret_cast<T*>(t + P.fs);
    S.rec = reinterpret_cast<T*>(t + P.rec);
    S.gw = reinterpret_cast<T*>(t + P.gw);
    S.geo = reinterpret_cast<T*>(t + P.geo);
    S.red = reinterpret_cast<T*>(t + P.red);
    S.skr = nullptr;
    stage_table_ptrs<T, GEOM, VW, NV, NR_, N2_, N3_>(S, reinterpret_cast<T*>(smem), A, M);
    return S;
}
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ StagePtrs<T> tile_ptrs(unsigned char* smem, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    const StreamSmem P = stream_smem_plan(A.B, Ms, nR, n2, n3, nwarps, (int)sizeof(T), A.mma ? 1 : 0, A.krf ? 1 : 0);
    StagePtrs<T> S;
    S.bar = reinterpret_cast<uint64_t*>(smem);
    S.fs = reinterpret_cast<T*>(smem + P.fs);
    S.rec = reinterpret_cast<T*>(smem + P.rec);
    S.geo = reinterpret_cast<T*>(smem + P.geo);
    S.red = reinterpret_cast<T*>(smem + P.red);
    S.skr = reinterpret_cast<T*>(smem + P.kr);
    stage_table_ptrs<T, GEOM, VW, NV, NR_, N2_, N3_>(S, reinterpret_cast<T*>(smem + P.tabs), A, M);
    S.gw = S.w3 + n3;
    S.nw = nullptr;
    return S;
}

template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void team_sync(const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    if (warps_apart) __syncwarp();
    else __syncthreads();
}

// Tables of the stage (nodes, weights, K matrices) into shared memory and the copy barrier;
// the caller synchronises the block.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_tables(const StagePtrs<T>& S, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    if (tid == 0) {
        mbar_init(S.bar, 1);
        fence_mbar_init();
    }
    const T* __restrict__ tab = reinterpret_cast<const T*>(A.tabT);
    const int bt = threadIdx.x, BT = blockDim.x;
    if (!A.krf)
#pragma unroll 4
        for (int e = bt; e < nR * nR; e += BT) S.KR[(e / nR) * kr_stride(nR) + e % nR] = tab[M.o_KR + e];
#pragma unroll 2
    for (int e = bt; e < n2 * n2; e += BT) S.K2[(e % n2) * n2 + e / n2] = tab[M.o_K2 + e];  // transposed
    if (GEOM == 1)
#pragma unroll 2
        for (int e = bt; e < n3 * n3; e += BT) S.K3[(e / n3) * (n3 + 1) + e % n3] = tab[M.o_K3 + e];
    // nodes and weights, [pR | wR | p2 | w2 | p3 | w3] from o_pR
    for (int e = bt; e < 2 * (nR + n2 + n3); e += BT) {
        const T x = tab[M.o_pR + e];
        T* d = e < 2 * nR ? (e < nR ? S.pR + e : S.wR + e - nR)
                          : e < 2 * (nR + n2) ? (e < 2 * nR + n2 ? S.p2 + e - 2 * nR : S.w2 + e - 2 * nR - n2)
                                              : (e < 2 * (nR + n2) + n3 ? S.p3 + e - 2 * (nR + n2) : S.w3 + e - 2 * (nR + n2) - n3);
        *d = x;
    }
}

// What a thread keeps while it walks along the radius: its vectors (kk << 20 | i << 10 | jb, -1 if none),
// their radial and third-axis momenta, WENO's epsilon and the value at the left face of the next cell.
template <typename T, int VW, int NV>
struct StageWalk {
    int vcode[NV];
    T pr[NV], p3[NV];
    Pair<T> e4w[NV][(VW + 1) / 2], vl[NV][(VW + 1) / 2];
};

template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_walk_init(StageWalk<T, VW, NV>& W, const StagePtrs<T>& S, int sl, const StageArgs& A,
                                                const MomSet& M) {
    FDLB_STAGE_SIZES;
#pragma unroll
    for (int g = 0; g < NV; ++g) {
        const int v = tid + g * NT;
        W.vcode[g] = -1;
        W.pr[g] = W.p3[g] = T(0);
#pragma unroll
        for (int h = 0; h < (VW + 1) / 2; ++h) W.e4w[g][h] = W.vl[g][h] = p_splat(T(0));
        if (v < Vs) {
            const int kk = v / (nR * n2v), rem = v % (nR * n2v), i = rem / n2v, jb = rem % n2v;
            const int k = sl * KS + kk;
            W.vcode[g] = (kk << 20) | (i << 10) | jb;
            W.pr[g] = S.pR[i];
            W.p3[g] = S.p3[k];
            const T wik = mul_rn(S.wR[i], S.w3[k]);
#pragma unroll
            for (int h = 0; h < (VW + 1) / 2; ++h) {
                const int ja = jb * VW + 2 * h, jc = VW == 1 ? ja : ja + 1;
                // WENO5 of f / w (Sec. II.C) taken on f itself: with eps scaled by w^2 the face value
                // of f is w times that of f / w, and the flux needs no division by the weight.  In
                // FP32 eps w^2 is kept above the float range's floor (weights below ~1e-16 at large
                // radial orders, whose populations are negligible, reconstruct with linear weights)
                const T wa = mul_rn(wik, S.w2[ja]), wc = mul_rn(wik, S.w2[jc]);
                const T ea = mul_rn(mul_rn(T(4e-6), wa), wa), ec = mul_rn(mul_rn(T(4e-6), wc), wc);
                W.e4w[g][h] = sizeof(T) == 4 ? p_make(fmax(ea, T(1e-37)), fmax(ec, T(1e-37))) : p_make(ea, ec);
            }
        }
    }
}

// A vector's face value between two cells: nw times the wall Maxwellian, or WENO5 on the window of rows
// at r0 .. r4 (element offsets of the vector in the rows), ascending.
template <typename T, int VW>
__device__ __forceinline__ void stage_wall_face(Pair<T> (&v)[(VW + 1) / 2], T nw, const T* gw, int nR, int n2, int i, int jb, int k) {
    const Pair<T> gik = p_splat(mul_rn(mul_rn(nw, gw[i]), gw[nR + n2 + k]));
#pragma unroll
    for (int h = 0; h < (VW + 1) / 2; ++h) {
        const int ja = jb * VW + 2 * h, jc = VW == 1 ? ja : ja + 1;
        v[h] = p_mul(gik, p_make(gw[nR + ja], gw[nR + jc]));
    }
}
template <typename T, int VW>
__device__ __forceinline__ void stage_weno_face(Pair<T> (&v)[(VW + 1) / 2], const T* r0p, const T* r1p, const T* r2p, const T* r3p,
                                                const T* r4p, bool pos, const Pair<T> (&e4w)[(VW + 1) / 2]) {
    using V2 = Pair<T>;
    constexpr int NP = (VW + 1) / 2;
    const V2 s3 = p_splat(pos ? T(3) : T(-3)), ns3 = p_splat(pos ? T(-3) : T(3));
    const V2 dL = p_splat(pos ? T(0.1) : T(0.3)), dR = p_splat(pos ? T(0.3) : T(0.1));
    V2 r0[NP], r1[NP], r2[NP], r3[NP], r4[NP];
    ld_pairs<T, VW>(r0p, r0);
    ld_pairs<T, VW>(r1p, r1);
    ld_pairs<T, VW>(r2p, r2);
    ld_pairs<T, VW>(r3p, r3);
    ld_pairs<T, VW>(r4p, r4);
#pragma unroll
    for (int h = 0; h < NP; ++h) v[h] = weno5_pair(r0[h], r1[h], r2[h], r3[h], r4[h], s3, ns3, dL, dR, e4w[h]);
}

// The values at the left face of cell c0; o[0 .. 5]: element offsets in fs of the rows of cells
// c0-3 .. c0+2.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_first_face(StageWalk<T, VW, NV>& W, const StagePtrs<T>& S, int c0, int sl, const int (&o)[6],
                                                 T nwL, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
#pragma unroll
    for (int g = 0; g < NV; ++g) {
        if (W.vcode[g] < 0) continue;
        const int i = (W.vcode[g] >> 10) & 1023, jb = W.vcode[g] & 1023, k = sl * KS + (W.vcode[g] >> 20);
        const bool pos = W.pr[g] > T(0);
        if (c0 == 0 && pos) {
            stage_wall_face<T, VW>(W.vl[g], nwL, S.gw, nR, n2, i, jb, k);
        } else {
            const T* b = S.fs + (tid + g * NT) * VW;
            stage_weno_face<T, VW>(W.vl[g], b + (pos ? o[0] : o[1]), b + (pos ? o[1] : o[2]), b + (pos ? o[2] : o[3]),
                                   b + (pos ? o[3] : o[4]), b + (pos ? o[4] : o[5]), pos, W.e4w[g]);
        }
    }
}

// Two rows beyond a wall from the four rows next to it, r[0] the wall cell's (element offsets in fs),
// into o1 (next to the wall) and, unless it is negative, o2: n_w times the wall Maxwellian for directions into the domain, the
// cubic extrapolation for directions out of it.  Each thread fills its own vectors, which alone it reads.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_ghosts(const StageWalk<T, VW, NV>& W, const StagePtrs<T>& S, int side, int sl, T nw,
                                             const int (&r)[4], int o1, int o2, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    const T* gw = S.gw + side * gwstride;
#pragma unroll
    for (int g = 0; g < NV; ++g) {
        if (W.vcode[g] < 0) continue;
        const int i = (W.vcode[g] >> 10) & 1023, jb = W.vcode[g] & 1023, k = sl * KS + (W.vcode[g] >> 20);
        T* b = S.fs + (tid + g * NT) * VW;
        const bool in = side == 0 ? W.pr[g] > T(0) : W.pr[g] < T(0);
#pragma unroll
        for (int e = 0; e < VW; ++e) {
            T g1, g2;
            if (in)
                g1 = g2 = mul_rn(mul_rn(mul_rn(nw, gw[i]), gw[nR + jb * VW + e]), gw[nR + n2 + k]);
            else
                wall_ghosts(b[r[0] + e], b[r[1] + e], b[r[2] + e], b[r[3] + e], g1, g2);
            b[o1 + e] = g1;
            if (o2 >= 0) b[o2 + e] = g2;
        }
    }
}

// Whether K_2's coefficients come with the launch (StageArgs::K2).
template <typename T, int VW, int N2_>
constexpr bool kK2Const = VW == N2_ && N2_ * N2_ * sizeof(T) <= kK2Bytes;
__device__ __forceinline__ float2 k2_pair(const StageArgs& A, int e, float) { return make_float2(A.K2.f[e], A.K2.f[e + 1]); }
__device__ __forceinline__ double2 k2_pair(const StageArgs& A, int e, double) { return make_double2(A.K2.d[e], A.K2.d[e + 1]); }

// Cell c of the walk: advection, force, collision, RK combination and store of the thread's vectors, the
// warp's raw sums to red[0 .. 15].  o[0 .. 5]: element offsets in fs of the rows of cells c-2 .. c+3
// (kLinear: one row after another from o[0] on); ct
// the cell's record; geo its A_+/V, A_-/V and force factor; skr its K^h f (mma.sync path) or null.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_, bool kCoherent, bool kLinear>
__device__ __forceinline__ void stage_cell(StageWalk<T, VW, NV>& W, const StagePtrs<T>& S, const InstDev& I, int c, int sl,
                                           const int (&o)[6], const T* ct, const T* geo, const T* skr, T nwR, T* red,
                                           const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    using V2 = Pair<T>;
    constexpr int NP = (VW + 1) / 2;
    const T* __restrict__ f_n = reinterpret_cast<const T*>(A.f_n);
    T* __restrict__ f_out = reinterpret_cast<T*>(A.f_out);
    const int krs = kr_stride(nR);
    const T dt = sizeof(T) == 4 ? (T)I.f_dt : (T)I.dt;
    const T ca_ = sizeof(T) == 4 ? (T)A.fa : (T)A.a, cb_ = sizeof(T) == 4 ? (T)A.fb : (T)A.b;
    T sc[20];
#pragma unroll
    for (int q = 0; q < 20; q += 4) {
        T t4[4];
        ld_vec<T, 4>(ct + q, t4);
        sc[q] = t4[0]; sc[q + 1] = t4[1]; sc[q + 2] = t4[2]; sc[q + 3] = t4[3];
    }
    const T n = sc[0], u0 = sc[1], u1 = sc[2], u2 = sc[3], iT = sc[4], itau = sc[5], cS = sc[6];
    const T q0 = sc[7], q1 = sc[8], q2 = sc[9], nbr = sc[10], X = sc[11], Y = sc[12];
    const T S00 = sc[13], J2c = sc[14], S22 = sc[15], g1c = sc[16], S02 = sc[17], hiT = sc[18], dv = sc[19];
    // collision terms of the cell that do not depend on the momentum (see below; the closure
    // stores -b rho chi, 0.4 S_11 / T, 2 S_01 / T and 1 / (2T) as they are used here)
    const T fiT = mul_rn(T(0.2), iT), F3 = mul_rn(mul_rn(cS, fiT), q1);
    const T* g2c = ct + rec_off_g2();
    const T* gRc = ct + rec_off_gR(n2);
    const T* g3c = ct + rec_off_g3(nR, n2);
    const T Ap = geo[0], Am = geo[1], kf = geo[2];
    const T* fc = S.fs + (kLinear ? o[0] + 2 * Ms : o[2]);  // row of cell c
    T acc[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) acc[q] = T(0);
#pragma unroll
    for (int g = 0; g < NV; ++g) {
        const int cd = W.vcode[g];
        if (cd < 0) continue;
        const int kk = cd >> 20, i = (cd >> 10) & 1023, jb = cd & 1023;
        const int k = sl * KS + kk;
        const int vb = ((kk * nR + i) * n2v + jb) * VW;  // element offset in the slice
        const long long gidx = I.f_off + (long long)c * Np + (long long)sl * Ms + vb;
        const T pr = W.pr[g], p3v = W.p3[g];
        // f_n for the RK combination, requested first so that its latency overlaps the update.
        // f_n: read-only for the stage kernel; written earlier in the same launch for the
        // persistent step kernel, which reads it coherently (L2)
        V2 fnv[NP];
        const bool use_fn = A.mode == 0 && ca_ != T(0);
        if (use_fn) {
            if constexpr (kCoherent)
                ldcg_pairs<T, VW>(f_n + gidx, fnv);
            else
                ldg_pairs<T, VW>(f_n + gidx, fnv);
        }
        // advection: WENO5 value at the right face, upwind by sign(p_R): rows of cells c-2..c+2
        // (p_R > 0) or c-1..c+3 (p_R < 0)
        V2 vr[NP];
        const bool pos = pr > T(0);
        if (c == I.n_cells - 1 && !pos) {
            stage_wall_face<T, VW>(vr, nwR, S.gw + gwstride, nR, n2, i, jb, k);
        } else if constexpr (kLinear) {
            const T* b = fc + (pos ? -2 * Ms : -Ms) + vb;
            stage_weno_face<T, VW>(vr, b, b + Ms, b + 2 * Ms, b + 3 * Ms, b + 4 * Ms, pos, W.e4w[g]);
        } else {
            const T* b = S.fs + vb;
            stage_weno_face<T, VW>(vr, b + (pos ? o[0] : o[1]), b + (pos ? o[1] : o[2]), b + (pos ? o[2] : o[3]),
                                   b + (pos ? o[3] : o[4]), b + (pos ? o[4] : o[5]), pos, W.e4w[g]);
        }
        // curvature force: K^h along i (one column shared by the vector), K_2 along j; each
        // output sums its terms in the order of the contracted index
        V2 KRf[NP], K2f[NP], K3f[NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) KRf[h] = K2f[h] = K3f[h] = p_splat(T(0));
        if (skr) {
            ld_pairs<T, VW>(skr + vb, KRf);
        } else if (A.krf) {
            // from the contraction kernel, in the layout of f
            ldg_pairs<T, VW>(reinterpret_cast<const T*>(A.krf) + gidx, KRf);
        } else {
            const T* col = fc + kk * nR * n2 + jb * VW;
            const T* kr = S.KR + i * krs;
            if constexpr (sizeof(T) == 4) {
                // four entries of the K^h row per vector load (the rows' stride is a multiple of four)
#pragma unroll 2
                for (int a4 = 0; a4 < nR; a4 += 4) {
                    T kq[4];
                    ld_vec<T, 4>(kr + a4, kq);
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        if (NR_ % 4 != 0 || NR_ == 0)
                            if (a4 + t >= nR) break;
                        V2 cv[NP];
                        ld_pairs<T, VW>(col + (a4 + t) * n2, cv);
                        const V2 kv = p_splat(kq[t]);
#pragma unroll
                        for (int h = 0; h < NP; ++h) KRf[h] = p_fma(kv, cv[h], KRf[h]);
                    }
                }
            } else {
#pragma unroll 8
                for (int a = 0; a < nR; ++a) {
                    V2 cv[NP];
                    ld_pairs<T, VW>(col + a * n2, cv);
                    const V2 kv = p_splat(kr[a]);
#pragma unroll
                    for (int h = 0; h < NP; ++h) KRf[h] = p_fma(kv, cv[h], KRf[h]);
                }
            }
        }
        {
            // K_2 from its transpose: input b's coefficients for the vector's outputs
            const T* row = fc + (kk * nR + i) * n2;
            const T* k2 = S.K2 + jb * VW;
            if constexpr (kK2Const<T, VW, N2_>) {
                // a whole p_2 row per thread: every coefficient is the same for all threads, an operand from
                // the launch's constants (from shared memory these coefficients alone were 64 of a cell's 281
                // wavefronts per warp, on the busiest unit of the kernel)
                T rv[VW];
                ld_vec<T, VW>(row, rv);
#pragma unroll
                for (int b = 0; b < VW; ++b) {
                    const V2 fv1 = p_splat(rv[b]);
#pragma unroll
                    for (int h = 0; h < NP; ++h)
                        K2f[h] = p_fma(k2_pair(A, b * VW + 2 * h, T(0)), fv1, K2f[h]);
                }
            } else
#pragma unroll 2
            for (int b4 = 0; b4 < n2v; ++b4) {
                T rv[VW];
                ld_vec<T, VW>(row + b4 * VW, rv);
#pragma unroll
                for (int t = 0; t < VW; ++t) {
                    V2 kq[NP];
                    ld_pairs<T, VW>(k2 + (b4 * VW + t) * n2, kq);
                    const V2 fv1 = p_splat(rv[t]);
#pragma unroll
                    for (int h = 0; h < NP; ++h) K2f[h] = p_fma(kq[h], fv1, K2f[h]);
                }
            }
        }
        if (GEOM == 1 && A.k3f) {
            // sliced along p_3: from the contraction kernel, in the layout of f
            ldg_pairs<T, VW>(reinterpret_cast<const T*>(A.k3f) + gidx, K3f);
        } else if (GEOM == 1) {
            const T* k3 = S.K3 + k * (n3 + 1);
            const T* c3 = fc + i * n2 + jb * VW;
#pragma unroll 4
            for (int b = 0; b < n3; ++b) {
                V2 cv[NP];
                ld_pairs<T, VW>(c3 + b * nR * n2, cv);
                const V2 kv = p_splat(k3[b]);
#pragma unroll
                for (int h = 0; h < NP; ++h) K3f[h] = p_fma(kv, cv[h], K3f[h]);
            }
        }
        // collision: -(f - f^S)/tau + J1[f^MB] (Eqs. j0, j1).  With x = p - u and
        // x1 = p_2 - u_2 the only coordinate that varies along the vector, the Shakhov
        // factor f^S / f^MB = 1 + c_S (|x|^2 / (5 T) - 1) x.q is a cubic in x1 and J1 / f^MB
        // (which holds |x|^2 / (2T) - 5/2 and the strain x.S.x / T) a quadratic: their
        // coefficients are formed once per vector, then two Horner evaluations per momentum.
        V2 fv[NP], g2v[NP], p2v[NP], p2q[NP];
        ld_pairs<T, VW>(fc + vb, fv);
        ld_pairs<T, VW>(g2c + jb * VW, g2v);
        ld_pairs<T, VW>(S.p2 + jb * VW, p2v);
#pragma unroll
        for (int h = 0; h < NP; ++h) p2q[h] = p_mul(p2v[h], p2v[h]);
        const T x0 = pr - u0, x2 = p3v - u2;
        T xsA = fma(x0, x0, mul_rn(x2, x2));
        const T xqA = fma(x0, q0, mul_rn(x2, q2));
        if (N3_ == 0 && M.reduced) {
            // cylinder with p_z integrated out (p_3 = u_3 = 0 here): the p_z^2 in |x|^2
            // becomes T for phi (k = 0), 3T for chi (k = 1); chi's T factor is in g_3
            xsA += (k == 0 ? T(1) : T(3)) / iT;
        }
        const T stA = fma(x0, fma(x0, S00, mul_rn(mul_rn(T(2), x2), S02)), mul_rn(mul_rn(x2, x2), S22));
        const T fmbA = mul_rn(mul_rn(n, gRc[i]), g3c[k]);
        const T Yd = fma(mul_rn(T(0.6), x0), Y, mul_rn(T(0.4), dv));
        const T J0 = mul_rn(nbr, fma(x0, X, fma(Yd, fma(hiT, xsA, T(-2.5)), mul_rn(mul_rn(T(0.4), iT), stA))));
        const T J1 = mul_rn(mul_rn(mul_rn(nbr, T(0.4)), g1c), x0);
        const T J2 = mul_rn(nbr, fma(Yd, hiT, J2c));
        const T b0 = fma(fiT, xsA, T(-1)), cb0 = mul_rn(cS, b0);
        const T F0 = fma(cb0, xqA, T(1)), F1 = mul_rn(cb0, q1), F2 = mul_rn(mul_rn(cS, fiT), xqA);
        // the advection and force terms enter negated: -(p_R A+/V vr - p_R A-/V vl) (face
        // values are of f) and -frc, each formed with one rounding like its positive
        const V2 npAp = p_splat(-mul_rn(pr, Ap)), pAm = p_splat(mul_rn(pr, Am));
        const V2 pu1 = p_splat(u1), pfmbA = p_splat(fmbA), pitau = p_splat(itau);
        const V2 pF0 = p_splat(F0), pF1 = p_splat(F1), pF2 = p_splat(F2), pF3 = p_splat(F3);
        const V2 pJ0 = p_splat(J0), pJ1 = p_splat(J1), pJ2 = p_splat(J2);
        V2 out[NP];
#pragma unroll
        for (int h = 0; h < NP; ++h) {
            const V2 nadv = p_fma(npAp, vr[h], p_mul(pAm, W.vl[g][h]));
            W.vl[g][h] = vr[h];
            V2 nfrc;
            if (GEOM == 0) {
                // -kf (p_2^2 K^h f - p_R K_2 f)
                nfrc = p_mul(p_splat(-kf), p_fma(p2q[h], KRf[h], p_mul(p_splat(-pr), K2f[h])));
            } else {
                // -((kf p_2^2 + kf p_3^2) K^h f - kf p_R (K_2 f + K_3 f))
                const V2 na = p_fma(p_splat(-kf), p2q[h], p_splat(-mul_rn(mul_rn(kf, p3v), p3v)));
                nfrc = p_fma(na, KRf[h], p_mul(p_splat(mul_rn(kf, pr)), p_add(K2f[h], K3f[h])));
            }
            const V2 x1 = p_sub(p2v[h], pu1);
            const V2 fmb = p_mul(pfmbA, g2v[h]);
            const V2 fS = p_mul(fmb, p_fma(p_fma(p_fma(pF3, x1, pF2), x1, pF1), x1, pF0));
            const V2 j1 = p_fma(p_fma(pJ2, x1, pJ1), x1, pJ0);
            out[h] = p_fma(fmb, j1, p_fma(p_sub(fS, fv[h]), pitau, p_add(nadv, nfrc)));
        }
        if (A.mode == 0) {
            // a f_n + b (f + dt L) with a = 1 - b, written as f_n + b ((f - f_n) + dt L):
            // exactly affine whatever the rounding of b (in FP32, fl(1/3) + fl(2/3)
            // exceeds one by 3e-8, which would scale the state by that much every step)
            const V2 pdt = p_splat(dt);
            if (use_fn) {
                const V2 pcb = p_splat(cb_);
#pragma unroll
                for (int h = 0; h < NP; ++h) out[h] = p_fma(pcb, p_fma(pdt, out[h], p_sub(fv[h], fnv[h])), fnv[h]);
            } else {
#pragma unroll
                for (int h = 0; h < NP; ++h) out[h] = p_fma(pdt, out[h], fv[h]);
            }
        }
        st_pairs<T, VW>(f_out + gidx, out);
        // raw sums: power sums over the vector's p_2 (per lane of the pairs, then the two
        // lanes), then the 13 moments
        V2 ps1 = p_mul(out[0], p2v[0]);
        V2 ps0 = out[0], ps2 = p_mul(out[0], p2q[0]), ps3 = p_mul(ps1, p2q[0]);
#pragma unroll
        for (int h = 1; h < NP; ++h) {
            const V2 o1 = p_mul(out[h], p2v[h]);
            ps0 = p_add(ps0, out[h]);
            ps1 = p_add(ps1, o1);
            ps2 = p_fma(out[h], p2q[h], ps2);
            ps3 = p_fma(o1, p2q[h], ps3);
        }
        const T s0 = VW == 1 ? ps0.x : ps0.x + ps0.y, s1 = VW == 1 ? ps1.x : ps1.x + ps1.y;
        const T s2 = VW == 1 ? ps2.x : ps2.x + ps2.y, s3 = VW == 1 ? ps3.x : ps3.x + ps3.y;
        const T prs0 = mul_rn(pr, s0), p3s0 = mul_rn(p3v, s0), rr = fma(pr, pr, mul_rn(p3v, p3v));
        const T e10 = fma(rr, s0, s2);  // sum out (p_R^2 + p_2^2 + p_3^2)
        if (N3_ == 0 && M.reduced && k == 1) {
            // chi = int p_z^2 f: it enters S2_zz and the p_z^2 p_a part of S3_a only
            acc[6] += s0;
            acc[10] += prs0;
            acc[11] += s1;
            continue;
        }
        acc[0] += s0;
        acc[1] += prs0;
        acc[2] += s1;
        acc[3] += p3s0;
        acc[4] = fma(pr, prs0, acc[4]);
        acc[5] += s2;
        acc[6] = fma(p3v, p3s0, acc[6]);
        acc[7] = fma(pr, s1, acc[7]);
        acc[8] = fma(pr, p3s0, acc[8]);
        acc[9] = fma(p3v, s1, acc[9]);
        acc[10] = fma(pr, e10, acc[10]);
        acc[11] += fma(rr, s1, s3);
        acc[12] = fma(p3v, e10, acc[12]);
    }
    // warp sums of the 13 raw moments of this cell (lane L holds sum L/2)
    if (A.mode == 0) {
        const T s = warp_sum16_transposed(acc, lane);
        if (!(lane & 1) && (lane >> 1) < kSums) red[warp * 16 + (lane >> 1)] = s;
    }
}

// The raw sums of `cnt` cells from c on, from the per-warp sums red[cell][warp][16]: over the warps in a
// fixed pairwise tree, to FP64.  FP32 partials: a double-float tree (error-free first level, ~44 bits
// after), converted once (exact); the FP64 pipe is slow on this part.  FP64 partials: FP64.  The tree
// over 16 slots (at most 512 threads), the slots beyond the team's warps zero, is taken over the smallest
// power of two of slots that holds the warps, since the levels above add exact zeros (the same sums bit
// for bit, without their instructions).
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_sums(const T* red, const InstDev& I, int c, int cnt, int sl, const StageArgs& A,
                                           const MomSet& M) {
    FDLB_STAGE_SIZES;
    auto tree = [&](auto kWc, int cl, int q) -> double {
        constexpr int kW = decltype(kWc)::value;
        if constexpr (sizeof(T) == 4) {
            Wide<float> v[kW];
#pragma unroll
            for (int ww = 0; ww < kW; ++ww) v[ww] = w_from_t(ww < nwarps ? (float)red[(cl * nwarps + ww) * 16 + q] : 0.f);
#pragma unroll
            for (int h = kW / 2; h > 0; h >>= 1)
#pragma unroll
                for (int ww = 0; ww < h; ++ww) v[ww] = w_add(v[ww], v[ww + h]);
            // the pair itself for the closure (its split of the sum: hi = fl(s), lo = s - hi)
            const long long cs = (long long)(I.cell_off + c + cl) * M.slices + sl;
            reinterpret_cast<float2*>(A.sumsw_out)[cs * kSums + q] = make_float2(v[0].hi, v[0].lo);
            return (double)v[0].hi + (double)v[0].lo;
        } else {
            double v[kW];
#pragma unroll
            for (int ww = 0; ww < kW; ++ww) v[ww] = ww < nwarps ? (double)red[(cl * nwarps + ww) * 16 + q] : 0.0;
#pragma unroll
            for (int h = kW / 2; h > 0; h >>= 1)
#pragma unroll
                for (int ww = 0; ww < h; ++ww) v[ww] = v[ww] + v[ww + h];
            return v[0];
        }
    };
    for (int e = tid; e < cnt * kSums; e += NT) {
        const int cl = e / kSums, q = e % kSums;
        double s;
        if (kTeam && nwarps == 1)
            s = tree(std::integral_constant<int, 1>{}, cl, q);
        else if (nwarps <= 4)
            s = tree(std::integral_constant<int, 4>{}, cl, q);
        else if (nwarps <= 8)
            s = tree(std::integral_constant<int, 8>{}, cl, q);
        else
            s = tree(std::integral_constant<int, 16>{}, cl, q);
        const long long cs = (long long)(I.cell_off + c + cl) * M.slices + sl;
        A.sums_out[cs * kSums + q] = s;
        if (q == 0) reinterpret_cast<T*>(A.dens_out)[cs] = (T)s;
    }
}

// The wall Maxwellians of an item's instance into shared memory; the caller synchronises.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_maxwellians(const StagePtrs<T>& S, int q, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    const T* gwi = reinterpret_cast<const T*>(A.gwT) + (long long)q * 2 * gwstride;
    for (int e = tid; e < 2 * gwstride; e += NT) S.gw[e] = gwi[e];
}

// Its wall densities, from the parts of the outgoing fluxes.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void stage_walls(const StagePtrs<T>& S, int q, const InstDev& I, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    if (tid < 2) {
        const T* pp = reinterpret_cast<const T*>(A.nwp) + ((long long)q * 2 + tid) * A.wall_parts;
        T part[kWallParts], sum = T(0);  // every load in flight; summed in order
#pragma unroll
        for (int p = 0; p < kWallParts; ++p) part[p] = p < A.wall_parts ? pp[p] : T(0);
#pragma unroll
        for (int p = 0; p < kWallParts; ++p)
            if (p < A.wall_parts) sum += part[p];
        S.nw[tid] = mul_rn(sum, sizeof(T) == 4 ? (T)(tid ? I.f_nw_iden[1] : I.f_nw_iden[0])
                                               : (T)(tid ? I.nw_iden[1] : I.nw_iden[0]));
    }
}

// Completion of the staged copy; false (on every thread of the team, A.err set) when it never completes.
// With the bulk engine the outcome is voted on, which is also the team's barrier after the copy.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ bool stage_wait(const StagePtrs<T>& S, const StageArgs& A, const MomSet& M, uint32_t& phase) {
    FDLB_STAGE_SIZES;
    if (!A.use_bulk) {
        team_sync<T, GEOM, VW, NV, NR_, N2_, N3_>(A, M);
        return true;
    }
    const bool bad = !mbar_wait_bounded(S.bar, phase);
    // every thread takes the same exit: a vote of the team on the outcome
    bool any;
    if (warps_apart) {
        any = __any_sync(0xffffffffu, bad);
        __syncwarp();
    } else {
        any = __syncthreads_or(bad) != 0;
    }
    if (any) {
        if (tid == 0) atomicOr(A.err, 1);
        mbar_wait_bounded(S.bar, phase);  // bounded wait for the copy still in flight
        return false;
    }
    phase ^= 1u;
    return true;
}

// Requests the rows of cells [lo, hi) of the item's slice (those inside the domain) and `nrec` records
// from cell crec on (into `rec`), and L2 prefetches of f_n for cells [plo, phi): the bulk engine, one
// completion on the copy barrier; else plain loads.  Row r goes to ring slot (r - base) mod R.
// part: 1 the rows (announcing the records too), 2 the records, 3 both.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void march_request(const StagePtrs<T>& S, const InstDev& I, int sl, int base, int R, int lo, int hi,
                                              int crec, int nrec, T* rec, int plo, int phi, int part, const StageArgs& A,
                                              const MomSet& M) {
    FDLB_STAGE_SIZES;
    lo = max(lo, 0);
    hi = min(hi, I.n_cells);
    const T* fin = reinterpret_cast<const T*>(A.f_in) + I.f_off + (long long)sl * Ms;
    const T* rsrc = reinterpret_cast<const T*>(A.rec) + (long long)(I.cell_off + crec) * rs;
    if (A.use_bulk) {
        if (tid == 0) {
            const uint32_t row = (uint32_t)(Ms * sizeof(T));
            if (part & 1) {
                fence_proxy_async();
                mbar_expect_tx(S.bar, (uint32_t)max(hi - lo, 0) * row + (uint32_t)(nrec * rs * sizeof(T)) + (uint32_t)A.tx_extra);
                int slot = (lo - base) % R;
                if (M.slices == 1 && hi - lo <= R - slot) {  // rows next to one another on both sides: one copy
                    if (hi > lo) bulk_g2s(S.fs + slot * Ms, fin + (long long)lo * Np, (uint32_t)(hi - lo) * row, S.bar);
                } else {
                    for (int r = lo; r < hi; ++r) {
                        bulk_g2s(S.fs + slot * Ms, fin + (long long)r * Np, row, S.bar);
                        if (++slot == R) slot = 0;
                    }
                }
            }
            if ((part & 2) && nrec > 0) bulk_g2s(rec, rsrc, (uint32_t)(nrec * rs * sizeof(T)), S.bar);
            // f_n (read once per population at the end of its update, from HBM) into L2 ahead of its use
            if ((part & 1) && A.mode == 0 && (sizeof(T) == 4 ? A.fa : (float)A.a) != 0.f) {
                const T* fn = reinterpret_cast<const T*>(A.f_n) + I.f_off + (long long)sl * Ms;
                if (M.slices == 1) {
                    if (phi > plo) bulk_prefetch_l2(fn + (long long)plo * Np, (uint32_t)(phi - plo) * row);
                } else {
                    for (int r = plo; r < phi; ++r) bulk_prefetch_l2(fn + (long long)r * Np, row);
                }
            }
        }
    } else {
        if (part & 1) {
            int slot = (lo - base) % R;
            for (int r = lo; r < hi; ++r) {
                for (int e = tid; e < Ms; e += NT) S.fs[slot * Ms + e] = ldg_t(fin + (long long)r * Np + e);
                if (++slot == R) slot = 0;
            }
        }
        if (part & 2)
            for (int e = tid; e < nrec * rs; e += NT) rec[e] = rsrc[e];
    }
}

template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void march_body(const StageArgs& A, const MomSet& M) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FDLB_STAGE_SIZES;
    const StagePtrs<T> S = march_ptrs<T, GEOM, VW, NV, NR_, N2_, N3_>(smem_raw, A, M);
    const int G = A.G, R = march_ring(G);
    stage_tables<T, GEOM, VW, NV, NR_, N2_, N3_>(S, A, M);
    const int nit = A.n_items[1], teams = warps_apart ? A.teams : 1;
    const int it0 = A.n_items[0] + blockIdx.x * teams + (warps_apart ? (int)threadIdx.x >> 5 : 0);
    __syncthreads();
    // An item's first request: rows c0-3 .. c0+G+2, the records and f_n of its first group.  The rows of the
    // first item are requested before the wait: they are the output of the stage kernel two launches
    // back, complete once the closure kernel in between has passed its own wait, which it does before it
    // lets this kernel start.  The records (the closure's output) follow the wait.
    auto first = [&](int4 wi, const InstDev& I, int part) {
        const int c0 = wi.y, cg = min(G, wi.z);
        march_request<T, GEOM, VW, NV, NR_, N2_, N3_>(S, I, wi.w, c0 - 3, R, c0 - 3, c0 + cg + 3, c0, cg, S.rec, c0, c0 + cg, part, A, M);
    };
    // What an item needs of the constants: the geometry of the G cells from c0 + cl on, the wall
    // Maxwellians and the threads' vectors; of the first item also before the wait.
    auto geometry = [&](int4 wi, const InstDev& I, int cl, T* dst) {
        const T* geoT = reinterpret_cast<const T*>(A.geoT) + (long long)(I.cell_off + wi.y) * kGeo;
        for (int e = tid; e < 3 * min(G, wi.z - cl); e += NT) dst[e] = geoT[(long long)(cl + e / 3) * kGeo + 2 + e % 3];
    };
    StageWalk<T, VW, NV> W;
    auto constants = [&](int4 wi, const InstDev& I) {
        geometry(wi, I, 0, S.geo);
        stage_maxwellians<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi.x, A, M);
        stage_walk_init<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, wi.w, A, M);
    };
    int4 wi = make_int4(0, 0, 0, 0);
    InstDev I;
    const bool early = A.use_bulk && it0 < nit;
    if (it0 < nit) {
        wi = A.items[it0];
        I = A.inst[wi.x];
        if (early) first(wi, I, 1);
        constants(wi, I);
    }
    pdl_trigger();
    pdl_wait();  // everything below reads what the previous kernels wrote
    uint32_t phase = 0;
    for (int it = it0; it < nit; it += gridDim.x * teams) {
        if (it != it0) {
            wi = A.items[it];
            I = A.inst[wi.x];
        }
        const int N = I.n_cells, c0 = wi.y, Be = wi.z, sl = wi.w, c1 = c0 + Be;
        first(wi, I, early && it == it0 ? 2 : 3);
        stage_walls<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi.x, I, A, M);
        if (it != it0) constants(wi, I);
        if (!stage_wait<T, GEOM, VW, NV, NR_, N2_, N3_>(S, A, M, phase)) return;
        const T nwL = S.nw[0], nwR = S.nw[1];
        // ring slot of cell r, as an element offset
        auto slot = [&](int r) { return (r - c0 + 3) % R * Ms; };
        auto outer_ghosts = [&]() {
            const int r[4] = {slot(N - 1), slot(N - 2), slot(N - 3), slot(N - 4)};
            stage_ghosts<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, 1, sl, nwR, r, slot(N), slot(N + 1), A, M);
        };
        // the rows beyond the inner wall among c0-3 .. c0+2
        if (c0 < 3) {
            const int r[4] = {slot(0), slot(1), slot(2), slot(3)};
            stage_ghosts<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, 0, sl, nwL, r, slot(-1), c0 < 2 ? slot(-2) : -1, A, M);
        }
        // rows N and N+1 are filled once, by the first group whose stencils reach row N (here when the first
        // face does): rows N-4 .. N-1 are then in the ring, and the rows whose slots they take are behind
        bool outer = c0 + 2 >= N;
        if (outer) outer_ghosts();
        int o[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = k * Ms;
        stage_first_face<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, c0, sl, o, nwL, A, M);
        team_sync<T, GEOM, VW, NV, NR_, N2_, N3_>(A, M);  // the row of cell c0-3 is free
#pragma unroll
        for (int k = 0; k < 6; ++k) o[k] = (k + 1) * Ms;  // rows of cells c0-2 .. c0+3 (R > 6)
        int buf = 0, prev = 0;
        for (int cl = 0; cl < Be; cl += G, buf ^= 1) {
            const int cg = min(G, Be - cl), cn = min(G, Be - cl - G), c = c0 + cl;
            // the next group's rows, records, f_n and geometry, into what the group before this one left
            if (cn > 0) {
                march_request<T, GEOM, VW, NV, NR_, N2_, N3_>(S, I, sl, c0 - 3, R, c + cg + 3, c + cg + cn + 3, c + cg, cn,
                                                              S.rec + (buf ^ 1) * G * rs, c + cg, c + cg + cn, 3, A, M);
                geometry(wi, I, cl + G, S.geo + (buf ^ 1) * 3 * G);
            }
            if (A.mode == 0 && prev > 0)
                stage_sums<T, GEOM, VW, NV, NR_, N2_, N3_>(S.red + (buf ^ 1) * G * nwarps * 16, I, c - prev, prev, sl, A, M);
            if (!outer && c + cg + 2 >= N) {
                outer = true;
                outer_ghosts();
            }
            for (int t = 0; t < cg; ++t) {
                stage_cell<T, GEOM, VW, NV, NR_, N2_, N3_, false, false>(W, S, I, c + t, sl, o, S.rec + (buf * G + t) * rs,
                                                                  S.geo + (buf * G + t) * 3, nullptr, nwR,
                                                                  S.red + (buf * G + t) * nwarps * 16, A, M);
#pragma unroll
                for (int k = 0; k < 5; ++k) o[k] = o[k + 1];
                o[5] = o[4] + Ms == R * Ms ? 0 : o[4] + Ms;
            }
            prev = cg;
            if (cn > 0) {
                if (!stage_wait<T, GEOM, VW, NV, NR_, N2_, N3_>(S, A, M, phase)) return;
            } else {
                team_sync<T, GEOM, VW, NV, NR_, N2_, N3_>(A, M);
            }
        }
        if (A.mode == 0)
            stage_sums<T, GEOM, VW, NV, NR_, N2_, N3_>(S.red + (buf ^ 1) * G * nwarps * 16, I, c1 - prev, prev, sl, A, M);
        team_sync<T, GEOM, VW, NV, NR_, N2_, N3_>(A, M);  // the next item overwrites the wall data and the sums
    }
}

// ---- a whole tile of cells staged at once: the compile-time shapes in FP32 (the rows one after another
// are addressed by immediate offsets; walking the ring, the same kernels issue 12% more instructions and
// take a barrier every two cells: 758 us against 716 us on 128 sweep instances, 84.8 against 80.8 us on the
// 2048-cell sphere), the persistent step kernel, whose closure writes the tile's records into shared
// memory, and the mma.sync form of the K^h contraction, a product over the tile.

// Requests the cells c0-3 .. c0+Be+2 of the item's slice and, when `records`, the tile's records.
// part: as march_request.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void tile_request(const StagePtrs<T>& S, int4 wi, const InstDev& I, bool records, int part,
                                             const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    march_request<T, GEOM, VW, NV, NR_, N2_, N3_>(S, I, wi.w, wi.y - 3, wi.z + 6, wi.y - 3, wi.y + wi.z + 3, wi.y,
                                                  records ? wi.z : 0, S.rec, wi.y, wi.y + wi.z, part, A, M);
}

// Geometry of the tile into shared memory.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void tile_geometry(const StagePtrs<T>& S, int4 wi, const InstDev& I, const StageArgs& A, const MomSet& M) {
    FDLB_STAGE_SIZES;
    const T* g = reinterpret_cast<const T*>(A.geoT) + (long long)(I.cell_off + wi.y) * kGeo;
    for (int c = tid; c < wi.z; c += NT) {
        S.geo[c * 3 + 0] = g[(long long)c * kGeo + 2];
        S.geo[c * 3 + 1] = g[(long long)c * kGeo + 3];
        S.geo[c * 3 + 2] = g[(long long)c * kGeo + 4];
    }
}

// The stage of the tile on the staged rows and records.  nwL, nwR: the wall densities of its instance.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_, bool kCoherent>
__device__ __forceinline__ void tile_compute(const StagePtrs<T>& S, int4 wi, const InstDev& I, T nwL, T nwR, const StageArgs& A,
                                             const MomSet& M) {
    FDLB_STAGE_SIZES;
    const int N = I.n_cells, c0 = wi.y, Be = wi.z, sl = wi.w;
    constexpr bool kMMA = sizeof(T) == 4 && NR_ > 0 && NR_ % 8 == 0 && VW == 4;
    const bool use_mma = kMMA && A.mma;
    StageWalk<T, VW, NV> W;
    stage_walk_init<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, sl, A, M);
    // rows beyond the walls (a tile near a wall needs them whether or not it touches it); the row behind
    // the last staged one is no part of the tile
    auto slot = [&](int r) { return (r - c0 + 3) * Ms; };
    if (c0 < 3) {
        const int r[4] = {slot(0), slot(1), slot(2), slot(3)};
        stage_ghosts<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, 0, sl, nwL, r, slot(-1), c0 < 2 ? slot(-2) : -1, A, M);
    }
    if (c0 + Be + 2 >= N) {
        const int r[4] = {slot(N - 1), slot(N - 2), slot(N - 3), slot(N - 4)};
        stage_ghosts<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, 1, sl, nwR, r, slot(N), N + 1 <= c0 + Be + 2 ? slot(N + 1) : -1, A, M);
    }
    // (K^h f)[i][(k, j)] = sum_a K^h[i][a] f[k][a][j] for the own cells, a GEMM of the nR x nR matrix with
    // the cell's nR x (n2 KS) slice, in split TF32 (K = Kh + Kl, f = fh + fl; Kh fh + Kh fl + Kl fh with FP32
    // accumulation: FP32-level products), n-tiles of 8 columns spread over the warps, results to shared memory.
    if constexpr (kMMA) {
      if (use_mma) {
        constexpr int MT = (NR_ + 15) / 16, KT = NR_ / 8;
        const int krs = kr_stride(nR);
        const int g = lane >> 2, tg = lane & 3;
        uint32_t ah[MT][KT][4], alo[MT][KT][4];
#pragma unroll
        for (int mt = 0; mt < MT; ++mt)
#pragma unroll
            for (int ks = 0; ks < KT; ++ks)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int r = mt * 16 + g + ((q & 1) ? 8 : 0), cidx = ks * 8 + tg + ((q & 2) ? 4 : 0);
                    const float x = r < NR_ ? S.KR[r * krs + cidx] : 0.f;
                    ah[mt][ks][q] = to_tf32(x);
                    alo[mt][ks][q] = to_tf32(x - __uint_as_float(ah[mt][ks][q]));
                }
        const int ncol = n2 * KS, ntc = ncol / 8;
        for (int tt = warp; tt < Be * ntc; tt += nwarps) {
            const int cl = tt / ntc, nt = tt % ntc;
            const int colb = nt * 8 + g;  // this lane's B column (k, j)
            const T* bsrc = S.fs + (long long)(cl + 3) * Ms + ((colb / n2) * nR) * n2 + colb % n2;
            float acc[MT][4];
#pragma unroll
            for (int mt = 0; mt < MT; ++mt) acc[mt][0] = acc[mt][1] = acc[mt][2] = acc[mt][3] = 0.f;
#pragma unroll
            for (int ks = 0; ks < KT; ++ks) {
                const float x0 = bsrc[(ks * 8 + tg) * n2], x1 = bsrc[(ks * 8 + tg + 4) * n2];
                const uint32_t bh0 = to_tf32(x0), bh1 = to_tf32(x1);
                const uint32_t bl0 = to_tf32(x0 - __uint_as_float(bh0)), bl1 = to_tf32(x1 - __uint_as_float(bh1));
#pragma unroll
                for (int mt = 0; mt < MT; ++mt) {
                    mma_tf32(acc[mt], alo[mt][ks], bh0, bh1);
                    mma_tf32(acc[mt], ah[mt][ks], bl0, bl1);
                    mma_tf32(acc[mt], ah[mt][ks], bh0, bh1);
                }
            }
            T* dst = S.skr + (long long)cl * Ms;
#pragma unroll
            for (int mt = 0; mt < MT; ++mt)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int r = mt * 16 + g + ((q & 2) ? 8 : 0), cc = nt * 8 + 2 * tg + (q & 1);
                    if (r < NR_) dst[((cc / n2) * nR + r) * n2 + cc % n2] = acc[mt][q];
                }
        }
        __syncthreads();
      }
    }
    int o[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) o[k] = k * Ms;
    stage_first_face<T, GEOM, VW, NV, NR_, N2_, N3_>(W, S, c0, sl, o, nwL, A, M);
    for (int cl = 0; cl < Be; ++cl) {
        o[0] += Ms;  // the row of cell c-2
        stage_cell<T, GEOM, VW, NV, NR_, N2_, N3_, kCoherent, true>(W, S, I, c0 + cl, sl, o, S.rec + cl * rs, S.geo + cl * 3,
                                                                    use_mma ? S.skr + (long long)cl * Ms : nullptr, nwR,
                                                                    S.red + cl * nwarps * 16, A, M);
    }
    __syncthreads();
    if (A.mode == 0) stage_sums<T, GEOM, VW, NV, NR_, N2_, N3_>(S.red, I, c0, Be, sl, A, M);
    __syncthreads();  // the next item overwrites the staged rows, the records and the sums
}

// The stage over staged tiles, an item to a block or, where there are more, one after another.
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_>
__device__ __forceinline__ void tile_body(const StageArgs& A, const MomSet& M) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ T snw[2];  // wall densities of the item's instance
    StagePtrs<T> S = tile_ptrs<T, GEOM, VW, NV, NR_, N2_, N3_>(smem_raw, A, M);
    S.nw = snw;
    stage_tables<T, GEOM, VW, NV, NR_, N2_, N3_>(S, A, M);
    const int it0 = A.n_items[0] + blockIdx.x, nit = A.n_items[1];
    __syncthreads();
    // (the first tile's rows before the wait, as in march_body)
    const bool early = A.use_bulk && it0 < nit;
    if (early) {
        const int4 wi = A.items[it0];
        tile_request<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi, A.inst[wi.x], true, 1, A, M);
    }
    pdl_trigger();
    pdl_wait();  // everything below reads what the previous kernels wrote
    uint32_t phase = 0;
    for (int it = it0; it < nit; it += gridDim.x) {
        const int4 wi = A.items[it];
        const InstDev I = A.inst[wi.x];
        tile_request<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi, I, true, early && it == it0 ? 2 : 3, A, M);
        // (here, where they overlap the copy: before the wait they cost the tile kernels 4%)
        tile_geometry<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi, I, A, M);
        stage_maxwellians<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi.x, A, M);
        stage_walls<T, GEOM, VW, NV, NR_, N2_, N3_>(S, wi.x, I, A, M);
        if (!stage_wait<T, GEOM, VW, NV, NR_, N2_, N3_>(S, A, M, phase)) return;
        tile_compute<T, GEOM, VW, NV, NR_, N2_, N3_, false>(S, wi, I, snw[0], snw[1], A, M);
    }
}

// The stage kernel; MINB = the blocks per SM the register allocation is bounded for: 1 (up to 512
// threads, 128 registers each; 256 threads where four FP64 momenta per thread need more, 288 for the
// sphere's rows of twelve) or, for blocks of
// at most 256 threads, 3 (at most 85 registers each); for the row kernel (VW = 8, blocks of at most 128
// threads) 5, 3 or 2 (at most 102, 170 or 255 registers each).  The arithmetic and its order are the same
// in all.
template <typename T, int VW, int MINB>
constexpr int stage_max_threads() {
    return VW == 12 ? 288 : VW == 8 ? (MINB == 1 ? 512 : 128) : (sizeof(T) == 8 && VW == 4) || MINB > 1 ? 256 : 512;
}
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_, int MINB>
__global__ void __launch_bounds__(stage_max_threads<T, VW, MINB>(), MINB) stream_kernel(StageArgs A, MomSet M) {
    if constexpr (stage_tiles(sizeof(T), NR_ > 0))
        tile_body<T, GEOM, VW, NV, NR_, N2_, N3_>(A, M);
    else
        march_body<T, GEOM, VW, NV, NR_, N2_, N3_>(A, M);
}

// Launches, or with `blocks_per_sm` plans the launch: reports how many blocks of the shape reside on an SM.
template <typename... Args>
cudaError_t stage_launch(void (*kern)(Args...), const StageArgs& A, const MomSet& M, int grid, int threads, size_t smem,
                         cudaStream_t s, int* blocks_per_sm) {
    if (blocks_per_sm) {
        const cudaError_t e = allow_dynamic_smem((const void*)kern, smem);
        return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, kern, threads, smem);
    }
    return launch_maybe_programmatic(kern, grid, threads, smem, s, A.programmatic, A, M);
}
template <typename T, int GEOM, int VW, int NV, int NR_, int N2_, int N3_, int MINB = 1>
cudaError_t launch_stream_t(const StageArgs& A, const MomSet& M, int grid, int threads, size_t smem, cudaStream_t s, int* bps) {
    if (threads > stage_max_threads<T, VW, MINB>()) return cudaErrorInvalidValue;
    return stage_launch(stream_kernel<T, GEOM, VW, NV, NR_, N2_, N3_, MINB>, A, M, grid, threads, smem, s, bps);
}

// Instantiations: generic shapes (VW 1, 2, 4 for float and double) and the compile-time
// shapes of the cylinder (16 x 8 x 8) and sphere (24 x 12 x 12) workloads.
template <typename T, int G>
cudaError_t launch_stream_dispatch(const StreamCfg& cfg, const StageArgs& A, const MomSet& M, int grid, int threads,
                                   size_t smem, cudaStream_t s, int* bps) {
    constexpr int VS = sizeof(T) == 4 || G == 0 ? 4 : 2;  // vector width of the compile-time shapes
    constexpr int SR = G == 0 ? 16 : 24, S2 = G == 0 ? 8 : 12, S3 = G == 0 ? 8 : 12;
    constexpr int NA = G == 0 ? 1 : 2, NB = G == 0 ? 2 : 4;
    if (cfg.spec) {
        if constexpr (sizeof(T) == 4 && G == 0) {
            // the cylinder's FP32 shape also as one vector of a whole p_2 row (8 momenta) per thread
            if (cfg.vw == 8 && cfg.nv == 1) {
                if (cfg.minb == 5) return launch_stream_t<T, G, 8, 1, SR, S2, S3, 5>(A, M, grid, threads, smem, s, bps);
                if (cfg.minb == 3) return launch_stream_t<T, G, 8, 1, SR, S2, S3, 3>(A, M, grid, threads, smem, s, bps);
                if (cfg.minb == 2) return launch_stream_t<T, G, 8, 1, SR, S2, S3, 2>(A, M, grid, threads, smem, s, bps);
                return launch_stream_t<T, G, 8, 1, SR, S2, S3>(A, M, grid, threads, smem, s, bps);
            }
        }
        if constexpr (sizeof(T) == 4 && G == 1) {
            // the sphere's as one whole p_2 row (12 momenta) per thread
            if (cfg.vw == 12 && cfg.nv == 1) return launch_stream_t<T, G, 12, 1, SR, S2, S3>(A, M, grid, threads, smem, s, bps);
        }
        if (cfg.vw != VS) return cudaErrorInvalidValue;
        if constexpr (sizeof(T) == 4 && G == 0) {
            // the cylinder's FP32 shape also bounded for three blocks of 256 threads per SM
            if (cfg.minb == 3 && cfg.nv == NA && threads <= 256)
                return launch_stream_t<T, G, VS, NA, SR, S2, S3, 3>(A, M, grid, threads, smem, s, bps);
        }
        if (cfg.nv == NA) return launch_stream_t<T, G, VS, NA, SR, S2, S3>(A, M, grid, threads, smem, s, bps);
        if constexpr (sizeof(T) == 4 || G == 1)
            if (cfg.nv == NB) return launch_stream_t<T, G, VS, NB, SR, S2, S3>(A, M, grid, threads, smem, s, bps);
        return cudaErrorInvalidValue;
    }
    // second-axis orders 4 and 8 at compile time: a whole row per thread or half of one
    if (cfg.vw == 4 && M.n2 == 4) {
        if (cfg.nv == 1) return launch_stream_t<T, G, 4, 1, 0, 4, 0>(A, M, grid, threads, smem, s, bps);
        if constexpr (sizeof(T) == 4)
            if (cfg.nv == 2) return launch_stream_t<T, G, 4, 2, 0, 4, 0>(A, M, grid, threads, smem, s, bps);
    }
    if constexpr (sizeof(T) == 4) {
        if (cfg.vw == 8 && cfg.nv == 1 && M.n2 == 8) return launch_stream_t<T, G, 8, 1, 0, 8, 0>(A, M, grid, threads, smem, s, bps);
        if (cfg.vw == 4 && cfg.nv == 2 && M.n2 == 8) return launch_stream_t<T, G, 4, 2, 0, 8, 0>(A, M, grid, threads, smem, s, bps);
    }
    if constexpr (sizeof(T) == 8) {
        if (cfg.vw == 1 && cfg.nv == 1) return launch_stream_t<T, G, 1, 1, 0, 0, 0>(A, M, grid, threads, smem, s, bps);
        if (cfg.vw == 2 && cfg.nv == 1) return launch_stream_t<T, G, 2, 1, 0, 0, 0>(A, M, grid, threads, smem, s, bps);
    }
    if (cfg.vw == 1 && cfg.nv == 4) return launch_stream_t<T, G, 1, 4, 0, 0, 0>(A, M, grid, threads, smem, s, bps);
    if (cfg.vw == 2 && cfg.nv == 4) return launch_stream_t<T, G, 2, 4, 0, 0, 0>(A, M, grid, threads, smem, s, bps);
    if (cfg.vw == 4 && cfg.nv == 1) return launch_stream_t<T, G, 4, 1, 0, 0, 0>(A, M, grid, threads, smem, s, bps);
    if constexpr (sizeof(T) == 4) {
        if (cfg.vw == 4 && cfg.nv == 2) return launch_stream_t<T, G, 4, 2, 0, 0, 0>(A, M, grid, threads, smem, s, bps);
    }
    return cudaErrorInvalidValue;
}

#define FDLB_STREAM_INSTANCE(T, G)                                                                               \
    cudaError_t launch_stream_##T##_##G(const StreamCfg& cfg, const StageArgs& A, const MomSet& M, int grid,    \
                                        int threads, size_t smem, cudaStream_t s, int* blocks_per_sm) {          \
        return launch_stream_dispatch<T, G>(cfg, A, M, grid, threads, smem, s, blocks_per_sm);                   \
    }

}  // namespace fdlb
