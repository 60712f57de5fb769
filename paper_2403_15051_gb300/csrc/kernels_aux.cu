// Auxiliary kernels of the FDLB step (raw sums, closure, residual); the fused stage kernel is
// in stream_kernel.cuh.  See kernels.cuh for the data layout and the launch plan.
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "kernels.cuh"
#include "kernels_decl.h"
#include "closure_item.cuh"
#include "fm_volumes.h"
#include "internal.h"

namespace fdlb {

// ------------------------------------------------------------------------------ moments
// Raw quadrature sums (Eq. mom_quad) of whole cells of a state, a warp per cell: a lane per
// momentum row (k, i) of n2 contiguous values (the rows of a warp are one contiguous span of the
// cell); per row the power sums over p_2 as in the stage kernel's epilogue, the thirteen sums in
// the populations' precision over the lane's rows, then a transposed warp sum.  Written into slice
// 0 of the partial-sum array in FP64 (the other slices cleared), for FP32 populations also as the
// double-float pairs the closure reads, and the slice densities.  Every cell of the state.
constexpr int kMomMaxNodes = 2 * kMaxQR;  // radial nodes

template <typename T>
__global__ void __launch_bounds__(256) moments_kernel(const T* __restrict__ f, double* __restrict__ sums,
                                                      T* __restrict__ dens, float2* __restrict__ sumsw,
                                                      long long total_cells, const double* __restrict__ tab, MomSet M) {
    __shared__ T sp_R[kMomMaxNodes], sp_2[kMaxQ], sp_3[kMaxQ];
    const int lane = threadIdx.x & 31;
    const int nR = M.nR, n2 = M.n2, n3 = M.n3, Np = M.Np;
    for (int e = threadIdx.x; e < nR; e += blockDim.x) sp_R[e] = (T)tab[M.o_pR + e];
    for (int e = threadIdx.x; e < n2; e += blockDim.x) sp_2[e] = (T)tab[M.o_p2 + e];
    for (int e = threadIdx.x; e < n3; e += blockDim.x) sp_3[e] = (T)tab[M.o_p3 + e];
    __syncthreads();
    const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    const int rows = nR * n3;
    for (long long c = w0; c < total_cells; c += nw) {
        const T* fc = f + c * Np;
        T acc[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) acc[q] = T(0);
        for (int r = lane; r < rows; r += 32) {
            const int k = r / nR, i = r % nR;
            const T* row = fc + (long long)r * n2;
            T s0 = T(0), s1 = T(0), s2 = T(0), s3 = T(0);
            for (int j = 0; j < n2; ++j) {
                const T v = row[j], p2v = sp_2[j];
                const T o1 = v * p2v, o2 = o1 * p2v;
                s0 += v;
                s1 += o1;
                s2 += o2;
                s3 += o2 * p2v;
            }
            const T pr = sp_R[i], p3v = sp_3[k];
            const T prs0 = pr * s0, p3s0 = p3v * s0, rr = pr * pr + p3v * p3v;
            if (M.reduced && k == 1) {
                // chi = int p_z^2 f: S2_zz and the p_z^2 p_a part of S3_a
                acc[6] += s0;
                acc[10] += prs0;
                acc[11] += s1;
                continue;
            }
            const T e10 = rr * s0 + s2;
            acc[0] += s0;
            acc[1] += prs0;
            acc[2] += s1;
            acc[3] += p3s0;
            acc[4] += pr * prs0;
            acc[5] += s2;
            acc[6] += p3v * p3s0;
            acc[7] += pr * s1;
            acc[8] += pr * p3s0;
            acc[9] += p3v * s1;
            acc[10] += pr * e10;
            acc[11] += rr * s1 + s3;
            acc[12] += p3v * e10;
        }
        const T tot = warp_sum16_transposed(acc, lane);
        const int q = lane >> 1;
        if (!(lane & 1) && q < kSums) {
            const double sd = (double)tot;
            const long long base = c * M.slices * kSums;
            sums[base + q] = sd;
            for (int sl = 1; sl < M.slices; ++sl) sums[base + sl * kSums + q] = 0.0;
            if (sumsw) {  // the double-float pairs of the FP32 closure
                sumsw[base + q] = make_float2((float)tot, 0.f);
                for (int sl = 1; sl < M.slices; ++sl) sumsw[base + sl * kSums + q] = make_float2(0.f, 0.f);
            }
            if (q == 0) {
                T* dd = dens + c * M.slices;
                dd[0] = tot;
                for (int sl = 1; sl < M.slices; ++sl) dd[sl] = T(0);
            }
        }
    }
}

// ------------------------------------------------------------------------------ closure
// The closure kernel: items of own cells (closure_cells in closure_item.cuh) and wall items
// (kind 1 + side, part): the block sums the outgoing flux of one part of the momenta at one
// wall; the stage kernel forms n_w from the parts (diffuse walls, zero net mass flux).
template <typename T>
__global__ void __launch_bounds__(kClosureThreads) closure_kernel(ClosureArgs A, MomSet M) {
    __shared__ T red[kClosureWarps];
    __shared__ __align__(8) uint64_t cbar;  // completion of the band-row copy
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // staged band rows, then the tables in the populations' precision, then the band-union
    // densities of an item
    T* wst = reinterpret_cast<T*>(smem_raw);
    T* tabs = wst + A.wst_elems;
    const ClosureTabs<T> tb = closure_tables<T>(tabs, A.tabT, M, tid, blockDim.x);
    T* nbuf = tabs + closure_tab_elems(M.nR, M.n2, M.n3);
    if (tid == 0) {
        mbar_init(&cbar, 1);
        fence_mbar_init();
    }
    __syncthreads();
    // A block's first item is looked up and its constants (band extents and rows, geometry) are requested
    // before the wait on the previous kernel; work lists, instances and bands are not written by kernels.
    // The successor (the stage kernel) may start after the wait: it requests the rows of the stage input,
    // written by the kernel this one has just waited for.
    bool waited = false;
    auto wait = [&]() {
        if (!waited) {
            pdl_wait();
            pdl_trigger();
            waited = true;
        }
    };
    const T* fin_all = reinterpret_cast<const T*>(A.f_in);
    T* rec_all = reinterpret_cast<T*>(A.rec);
    T* nwp = reinterpret_cast<T*>(A.nwp);
    uint32_t phase = 0;
    const int nit = A.n_items[1];
    for (int it = A.n_items[0] + blockIdx.x; it < nit; it += gridDim.x) {
        const int4 w = A.items[it];
        const InstDev I = A.inst[w.x];
        if (w.w != 0) {
            // ---- one part of the outgoing flux through a wall
            wait();
            const int side = w.w - 1, part = w.z, P = A.wall_parts;
            const T* wall = fin_all + I.f_off + (side == 0 ? 0LL : (long long)(I.n_cells - 1) * M.Np);
            T acc = wall_flux_partial<T>(wall, side == 0 ? (long long)M.Np : -(long long)M.Np, M, tb, side, part, P, tid);
            acc = warp_sum(acc);
            if (lane == 0) red[warp] = acc;
            __syncthreads();
            if (tid == 0) nwp[((long long)w.x * 2 + side) * P + part] = wall_part_sum(red);
            __syncthreads();
            continue;
        }
        T* recb = rec_all + (long long)(I.cell_off + w.y) * A.rec_stride;
        if (!closure_cells<T>(A, M, tb, I, w.y, w.z, recb, wst, nbuf, &cbar, phase, NoExtra{}, wait, NoHook{})) return;
    }
    wait();
}

// ------------------------------------------------------------------------------ batch closure
// The closure of a batch with a warp for each job and no block barrier.  With many more items than
// co-resident blocks the chain form is bound by how many items are in flight: most of its phases run one
// lane per reach cell while the other warps wait at its barriers, and its FM band rows are read one item
// at a time.  Here closure_band_kernel gives every pair of band rows to a warp (the band sum of Eq. fm,
// then chi and nbar into A.cw) and takes the wall parts; closure_records_kernel gives every item (28 own
// cells, 32 with its reach) to a warp, a lane per cell.  Where the bands are short (kInlineBand columns)
// the records kernel sums them itself and takes the wall parts, and the first launch goes.  All are made
// of the chain's per-cell functions (closure_item.cuh), so the records are the chain's.

// A warp per job of the host-formed list A.pairs: two band rows summed together by clo_band_row2
// with the loads of both in flight, then chi and nbar of the two cells; or one part of the
// outgoing flux through a wall.  A job's description is one 48-byte load, so the weights and
// densities follow it after a single dependent load.
template <typename T>
__global__ void __launch_bounds__(kClosureThreads, sizeof(T) == 4 ? 8 : 4) closure_band_kernel(ClosureArgs A, MomSet M) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const ClosureTabs<T> tb = closure_tables<T>(reinterpret_cast<T*>(smem_raw), A.tabT, M, tid, blockDim.x);
    __syncthreads();
    pdl_wait();  // the densities and populations of the previous kernel
    pdl_trigger();
    const T* fin_all = reinterpret_cast<const T*>(A.f_in);
    const T* band = reinterpret_cast<const T*>(A.band);
    const T* dens = reinterpret_cast<const T*>(A.dens);
    T* nwp = reinterpret_cast<T*>(A.nwp);
    T* cw = reinterpret_cast<T*>(A.cw);
    const int slices = A.slices;
    const int np = A.n_pairs[1];
    const int gw = A.n_pairs[0] + blockIdx.x * kClosureWarps + warp, nw = gridDim.x * kClosureWarps;
    for (int v = gw; v < np; v += nw) {
        const BandPair P = A.pairs[v];
        if (P.kmaxA < 0) {
            const int side = -1 - P.kmaxA, part = P.kmaxB;
            const T x = wall_part_of_warp<T>(fin_all, M, tb, A.inst[P.q], side, part, A.wall_parts, lane);
            if (lane == 0) nwp[((long long)P.q * 2 + side) * A.wall_parts + part] = x;
            continue;
        }
        const T* ndA = dens + P.dA * slices;
        const T* ndB = dens + P.dB * slices;
        auto dA = [&](int k) {
            T x = ndA[(long long)k * slices];
            for (int sl = 1; sl < slices; ++sl) x += ndA[(long long)k * slices + sl];
            return x;
        };
        auto dB = [&](int k) {
            T x = ndB[(long long)k * slices];
            for (int sl = 1; sl < slices; ++sl) x += ndB[(long long)k * slices + sl];
            return x;
        };
        T totA, totB;
        clo_band_row2<T>(band + P.wA, dA, P.kmaxA, band + P.wB, dB, P.kmaxB, lane, totA, totB);
        // lane 0's sums: every lane ends the butterfly with the total, but each in an order of its
        // own, and the chain form takes lane 0's
        if (lane == 0) {
            const InstDev& I = A.inst[P.q];
            const T etaf = inst_param<T>(I.etafac, I.f_etafac);
            const long long gc = P.gc;
            cw[gc * 2] = clo_chi<T>(etaf, totA);
            cw[gc * 2 + 1] = totA;
            if (P.kmaxB > 0) {
                cw[gc * 2 + 2] = clo_chi<T>(etaf, totB);
                cw[gc * 2 + 3] = totB;
            }
        }
    }
}

// What a warp of the records kernel shares among its lanes: an item's reach cells, pair terms and
// expansion coefficients.
template <typename T>
struct WarpReach {
    Wide<T> n[32], Tc[32], u[3][32];
    T nb[32], gp[5][32], nf[32];
    EqCoeffs<T> ecs;
};

// Bound by the latency of one item's chain of phases, with 8 to 16 warps per SM to hide it; every phase
// but the equilibrium vectors has a lane per cell, so its instructions are shared by up to 32 cells (in
// FP64, where an instruction costs the same however few lanes take it, that is the point).  kBand: the
// widest band in units of 32 columns, rounded up to 2 or 4 (0: closure_band_kernel sums the bands).
template <typename T, int kBand>
__global__ void __launch_bounds__(kClosureThreads, sizeof(T) == 4 ? 4 : 2) closure_records_kernel(ClosureArgs A, MomSet M) {
    using W = Wide<T>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, wpb = blockDim.x >> 5;
    WarpReach<T>& R = reinterpret_cast<WarpReach<T>*>(smem_raw)[warp];
    const ClosureTabs<T> tb = closure_tables<T>(reinterpret_cast<T*>(smem_raw + wpb * sizeof(WarpReach<T>)), A.tabT, M, tid, blockDim.x);
    const T* geoT = reinterpret_cast<const T*>(A.geoT);
    const T* band = reinterpret_cast<const T*>(A.band);
    const T* dens = reinterpret_cast<const T*>(A.dens);
    T* cw = reinterpret_cast<T*>(A.cw);
    T* rec_all = reinterpret_cast<T*>(A.rec);
    const int rs = A.rec_stride, slices = A.slices;
    const ReachView<T> RV{R.n, R.Tc, {R.u[0], R.u[1], R.u[2]}, R.nb};
    const int nit = A.n_items[1], nw = gridDim.x * wpb;
    __syncthreads();
    bool waited = false;
    auto wait = [&]() {
        if (!waited) {
            pdl_wait();  // the band results, or the previous stage's sums
            pdl_trigger();
            waited = true;
        }
    };
    for (int it = A.n_items[0] + blockIdx.x * wpb + warp; it < nit; it += nw) {
        const int4 w = A.items[it];
        if (!kBand && w.w != 0) continue;  // wall items: closure_band_kernel
        const InstDev I = A.inst[w.x];
        if (w.w != 0) {
            wait();
            const int side = w.w - 1, part = w.z;
            const T x = wall_part_of_warp<T>(reinterpret_cast<const T*>(A.f_in), M, tb, I, side, part, A.wall_parts, lane);
            if (lane == 0) reinterpret_cast<T*>(A.nwp)[((long long)w.x * 2 + side) * A.wall_parts + part] = x;
            continue;
        }
        const int c0 = w.y, cnt = w.z, N = I.n_cells;
        int h0, h1;
        clo_reach(c0, cnt, N, h0, h1);
        const int nh = h1 - h0, t = h0 + lane - c0;  // this lane's reach cell, and as an own cell
        const long long gc = (long long)I.cell_off + h0 + min(lane, nh - 1);
        const bool own = t >= 0 && t < cnt && lane < nh;
        T* recb = rec_all + ((long long)I.cell_off + c0) * rs;
        T ct[kCellScalars];
        const T etaf = inst_param<T>(I.etafac, I.f_etafac);
        const T geo0 = geoT[gc * kGeo], geo1 = geoT[gc * kGeo + 1];
        int2 bl = make_int2(0, 0);
        if (kBand && !I.chi_local) bl = reinterpret_cast<const int2*>(A.band_lo)[gc];
        wait();
        // ---- n, u, T of the reach cells, nbar (the band kernel's, or summed here, or local)
        W sv[kSums];
        clo_load_sums<T>(A, gc, sv);
        if (kBand && !I.chi_local) {
            constexpr int kRows = kBand == 2 ? 8 : 4;
            for (int r0 = 0; r0 < nh; r0 += kRows) {
                const T *Wr[kRows], *nd[kRows];
                int km[kRows];
                T tot[kRows];
#pragma unroll
                for (int r = 0; r < kRows; ++r) {
                    const int rr = min(r0 + r, nh - 1);
                    const int lo = __shfl_sync(0xffffffffu, bl.x, rr), ext = __shfl_sync(0xffffffffu, bl.y, rr);
                    Wr[r] = band + I.band_off + (long long)(h0 + rr) * I.band_w;
                    nd[r] = dens + ((long long)I.cell_off + lo) * slices;
                    km[r] = r0 + r < nh ? min(ext, N - lo) : 0;
                }
                clo_band_rows<T, kRows, kBand ? kBand : 4>(Wr, nd, km, slices, lane, tot);
                // lane 0's sums (every lane ends the butterfly with the total, each in its own order)
                if (lane == 0)
#pragma unroll
                    for (int r = 0; r < kRows; ++r)
                        if (r0 + r < nh) R.nb[r0 + r] = tot[r];
            }
        }
        W n, u[3], Tc;
        T q[3];
        clo_fields<T>(sv, n, u, Tc, q);
        R.n[lane] = n;
        R.Tc[lane] = Tc;
#pragma unroll
        for (int a = 0; a < 3; ++a) R.u[a][lane] = u[a];
        __syncwarp();
        if (I.chi_local)
            R.nb[lane] = w_hi(n);
        else if (!kBand)
            R.nb[lane] = cw[gc * 2 + 1];
        __syncwarp();
        // ---- the pair terms; of the own cells the expansion coefficients and the transport scalars
        if (lane < nh - 1) {
            T d[5];
            clo_pair_terms<T>(RV, lane, etaf, I.chi_local != 0, d);
#pragma unroll
            for (int v = 0; v < 5; ++v) R.gp[v][lane] = d[v];
        }
        const T cT = w_hi(Tc), cu0 = w_hi(u[0]), cu1 = w_hi(u[1]), cu2 = w_hi(u[2]);
        if (own) {
            const T tm1 = w_hi(w_sub(Tc, w_from_t(T(1))));  // T - 1 without cancellation
            // (a launch runs most of this code once per warp: the loop stays a loop, the kernel small, since fetching
            // its instructions is a good part of a short launch)
#pragma unroll 1
            for (int job = 0; job < 4; ++job) {
                T ev[kMaxE + 1];
                clo_eq_coeffs<T>(job, cT, tm1, cu0, job == 2 ? cu1 : cu2, tb, M, ev);
#pragma unroll
                for (int l = 0; l < kMaxE; ++l) R.ecs.v[job][l][t] = ev[l];
            }
            const T nb = R.nb[lane], chi = clo_chi<T>(etaf, nb);
            if (kBand || I.chi_local) {
                cw[gc * 2] = chi;
                cw[gc * 2 + 1] = nb;
            }
            clo_record_transport<T>(ct, n, cu0, cu1, cu2, cT, chi, q, I);
        }
        __syncwarp();
        if (own) clo_record_gradients<T>(ct, c0 + t, N, h0, R.gp, cu0, cu1, cu2, cT, geo0, geo1, I);
        // ---- the equilibrium vectors and the normalised density (eight lanes per own cell), then the
        // scalars with it
        for (int e = lane; e < (8 * cnt + 31) / 32 * 32; e += 32) {
            const int tt = min(e >> 3, cnt - 1), lt = c0 + tt - h0;
            const bool on = (e >> 3) < cnt;
            const T nf = clo_equilibrium<T>(on, e & 7, recb + (long long)tt * rs, R.n[lt], w_hi(R.Tc[lt]), R.ecs, tt, tb, M);
            if (on && (e & 7) == 0) R.nf[tt] = nf;
        }
        __syncwarp();
        if (own) {
            ct[0] = R.nf[t];
            T* dst = recb + (long long)t * rs;
#pragma unroll
            for (int k = 0; k < kCellScalars; k += 16 / (int)sizeof(T)) {  // 16-byte stores
                if constexpr (sizeof(T) == 4)
                    *reinterpret_cast<float4*>(dst + k) = make_float4(ct[k], ct[k + 1], ct[k + 2], ct[k + 3]);
                else
                    *reinterpret_cast<double2*>(dst + k) = make_double2(ct[k], ct[k + 1]);
            }
        }
        __syncwarp();  // the shared arrays are reused by the next item
    }
    wait();
}

// ------------------------------------------------------------------------------ state change
// Sums over one chunk of an instance's populations of (a - b)^2 and b^2 in FP64 (a the state after
// a step, b before it): chunk k of instance q covers elements [k C, (k + 1) C) of the instance; the
// block's sums go to part[(q * chunks + k) * 2 + {0, 1}] in a fixed tree order.
template <typename T>
__global__ void change_sums_kernel(const T* __restrict__ a, const T* __restrict__ b, const long long* __restrict__ off,
                                   const long long* __restrict__ cnt, int chunks, long long C, double* __restrict__ part) {
    __shared__ double red[2][32];
    const int q = blockIdx.x / chunks, k = blockIdx.x % chunks;
    const long long lo = k * C, hi = min(cnt[q], lo + C);
    double d2 = 0.0, b2 = 0.0;
    for (long long e = lo + threadIdx.x; e < hi; e += blockDim.x) {
        const double x = (double)a[off[q] + e], y = (double)b[off[q] + e];
        d2 += (x - y) * (x - y);
        b2 += y * y;
    }
    d2 = warp_sum(d2);
    b2 = warp_sum(b2);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        red[0][warp] = d2;
        red[1][warp] = b2;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[threadIdx.x][w];
        part[((long long)q * chunks + k) * 2 + threadIdx.x] = s;
    }
}

cudaError_t launch_change_sums(int tsize, const void* a, const void* b, const long long* off, const long long* cnt,
                               int n_inst, int chunks, long long C, double* part, cudaStream_t s) {
    const int grid = n_inst * chunks;
    if (tsize == 4)
        change_sums_kernel<float><<<grid, 256, 0, s>>>((const float*)a, (const float*)b, off, cnt, chunks, C, part);
    else
        change_sums_kernel<double><<<grid, 256, 0, s>>>((const double*)a, (const double*)b, off, cnt, chunks, C, part);
    return cudaGetLastError();
}

// ------------------------------------------------------------------------------ queries
// The FP64 closure record of every cell of the active instances (moments and closure queries,
// not the stage): n, u, T, q, P_12 (Eq. macro_def) from the raw sums in FP64, chi and nbar from
// the closure's side buffer.
template <typename T>
__global__ void ca_kernel(const double* __restrict__ sums, const void* cwv, double* __restrict__ ca, int slices,
                          int total_cells, double* __restrict__ packed) {
    const T* cw = reinterpret_cast<const T*>(cwv);
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < total_cells; c += gridDim.x * blockDim.x) {
        double s[kSums];
        for (int q = 0; q < kSums; ++q) s[q] = 0.0;
        for (int sl = 0; sl < slices; ++sl)
            for (int q = 0; q < kSums; ++q) s[q] += sums[((long long)c * slices + sl) * kSums + q];
        const double n = s[0], in = 1.0 / n;
        const double u0 = s[1] * in, u1 = s[2] * in, u2 = s[3] * in;
        const double tr = s[4] + s[5] + s[6];
        const double uu = u0 * u0 + u1 * u1 + u2 * u2;
        const double Tc = (tr - n * uu) * in * (1.0 / 3.0);
        const double m0 = s[4] * u0 + s[7] * u1 + s[8] * u2;
        const double m1 = s[7] * u0 + s[5] * u1 + s[9] * u2;
        const double m2 = s[8] * u0 + s[9] * u1 + s[6] * u2;
        double* r = ca + (long long)c * kCA;
        r[0] = n;
        r[1] = u0;
        r[2] = u1;
        r[3] = u2;
        r[4] = Tc;
        r[5] = 0.5 * (s[10] - 2.0 * m0 - u0 * tr + 2.0 * n * uu * u0);
        r[6] = 0.5 * (s[11] - 2.0 * m1 - u1 * tr + 2.0 * n * uu * u1);
        r[7] = 0.5 * (s[12] - 2.0 * m2 - u2 * tr + 2.0 * n * uu * u2);
        r[8] = s[7] - n * u0 * u1;  // P_12
        r[9] = (double)cw[2 * (long long)c];
        r[10] = (double)cw[2 * (long long)c + 1];
        r[11] = 0.0;
        if (packed)  // the moments query's rows: the first kNmom columns, contiguous
            for (int e = 0; e < kNmom; ++e) packed[(long long)c * kNmom + e] = r[e];
    }
}

template <typename T>
void launch_ca(const double* sums, const void* cw, double* ca, int slices, int total_cells, cudaStream_t s,
               double* packed) {
    const int g = (total_cells + 255) / 256;
    ca_kernel<T><<<g < 2048 ? (g > 0 ? g : 1) : 2048, 256, 0, s>>>(sums, cw, ca, slices, total_cells, packed);
}

// ------------------------------------------------------------------------------ stream
// ------------------------------------------------------------------------------ residual
// Per instance: the profile moments (n, u_2, T, q_R) of the populations whose raw sums are
// given, the largest change since the saved profile, the largest saved value, the total mass
// sum_c V_c n_c and a non-finite flag; the current profile replaces the saved one.
__global__ void residual_kernel(const double* __restrict__ sums, int slices, const InstDev* __restrict__ inst,
                                const double* __restrict__ geo, double* __restrict__ prev, double* __restrict__ out,
                                int n_inst, int save) {
    __shared__ double red[kMaxRed][10];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int q = blockIdx.x; q < n_inst; q += gridDim.x) {
        const InstDev I = inst[q];
        double loc[10];
        for (int e = 0; e < 10; ++e) loc[e] = 0.0;
        for (int c = threadIdx.x; c < I.n_cells; c += blockDim.x) {
            double s[kSums];
            for (int e = 0; e < kSums; ++e) s[e] = 0.0;
            for (int sl = 0; sl < slices; ++sl)
                for (int e = 0; e < kSums; ++e) s[e] += sums[((long long)(I.cell_off + c) * slices + sl) * kSums + e];
            const double n = s[0], u0 = s[1] / n, u1 = s[2] / n, u2 = s[3] / n;
            const double tr = s[4] + s[5] + s[6], uu = u0 * u0 + u1 * u1 + u2 * u2;
            const double Tc = (tr - n * uu) / (3.0 * n);
            const double m0 = s[4] * u0 + s[7] * u1 + s[8] * u2;
            const double qR = 0.5 * (s[10] - 2.0 * m0 - u0 * tr + 2.0 * n * uu * u0);
            const double cur[4] = {n, u1, Tc, qR};
            double* pv = prev + (long long)(I.cell_off + c) * 4;
            for (int e = 0; e < 4; ++e) {
                double d = fabs(cur[e] - pv[e]);
                if (!(d == d)) d = 1e300;
                loc[e] = fmax(loc[e], d);
                loc[4 + e] = fmax(loc[4 + e], fabs(pv[e]));
                if (save) pv[e] = cur[e];
            }
            loc[8] += geo[(long long)(I.cell_off + c) * kGeo + 5] * n;
            if (!isfinite(n) || !isfinite(Tc) || !isfinite(qR) || !isfinite(u1)) loc[9] = 1.0;
        }
        for (int e = 0; e < 10; ++e) {
            double v = loc[e];
            for (int o = 16; o > 0; o >>= 1) {
                const double w = __shfl_xor_sync(0xffffffffu, v, o);
                v = (e == 8) ? v + w : fmax(v, w);
            }
            if (lane == 0) red[warp][e] = v;
        }
        __syncthreads();
        if (threadIdx.x < 10) {
            double v = threadIdx.x == 8 ? 0.0 : 0.0;
            for (int w = 0; w < nw; ++w) v = (threadIdx.x == 8) ? v + red[w][threadIdx.x] : fmax(v, red[w][threadIdx.x]);
            out[q * 10 + threadIdx.x] = v;
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------------------------ launchers
template <typename T>
void launch_moments(const T* f, double* sums, T* dens, void* sumsw, long long total_cells, int grid, const double* tab,
                    const MomSet& M, cudaStream_t s) {
    moments_kernel<T><<<grid, 256, 0, s>>>(f, sums, dens, reinterpret_cast<float2*>(sumsw), total_cells, tab, M);
}

// Slice densities from restored raw sums.
template <typename T>
__global__ void dens_kernel(const double* __restrict__ sums, T* __restrict__ dens, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dens[i] = (T)sums[i * kSums];
}

// Double-float pairs (hi = fl(s), lo = fl(s - hi)) of FP64 raw sums: the closure's input for
// FP32 populations, where the stage kernel does not write them (set-up, restored checkpoints).
__global__ void sums_pairs_kernel(const double* __restrict__ sums, float2* __restrict__ sw, long long n) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const double v = sums[i];
        const float hi = __double2float_rn(v);
        sw[i] = make_float2(hi, __double2float_rn(v - (double)hi));
    }
}

void launch_sums_pairs(const double* sums, void* sw, long long n, cudaStream_t s) {
    const long long g = (n + 255) / 256;
    sums_pairs_kernel<<<(int)(g < 4096 ? (g > 0 ? g : 1) : 4096), 256, 0, s>>>(sums, reinterpret_cast<float2*>(sw), n);
}

template <typename T>
void launch_dens_from_sums(const double* sums, T* dens, long long n, cudaStream_t s) {
    const long long g = (n + 255) / 256;
    dens_kernel<T><<<(int)(g < 4096 ? (g > 0 ? g : 1) : 4096), 256, 0, s>>>(sums, dens, n);
}

template <typename T>
cudaError_t launch_closure(const ClosureArgs& A, const MomSet& M, int grid, int threads, size_t smem, cudaStream_t s) {
    if (A.wst_elems % 4) return cudaErrorInvalidValue;  // vector loads of the tables behind the band rows
    return launch_maybe_programmatic(closure_kernel<T>, grid, threads, smem, s, A.programmatic, A, M);
}

size_t closure_records_smem(int nR, int n2, int n3, int warps, int tsize) {
    return (size_t)warps * (tsize == 4 ? sizeof(WarpReach<float>) : sizeof(WarpReach<double>)) +
           (size_t)closure_tab_elems(nR, n2, n3) * tsize + 16;
}

template <typename T>
auto closure_records(int inline_band) {
    return inline_band == 2 ? closure_records_kernel<T, 2> : inline_band ? closure_records_kernel<T, 4> : closure_records_kernel<T, 0>;
}

template <typename T>
cudaError_t launch_closure_batch(const ClosureArgs& A, const MomSet& M, const ClosureBatchShape& B, cudaStream_t s) {
    auto rec = closure_records<T>(B.inline_band);
    const size_t smem = closure_records_smem(M.nR, M.n2, M.n3, B.warps, (int)sizeof(T));
    const size_t band_smem = closure_smem_bytes(M.nR, M.n2, M.n3, 0, 0, (int)sizeof(T));
    cudaError_t e = cudaSuccess;
    if (!B.inline_band)
        e = launch_maybe_programmatic(closure_band_kernel<T>, B.grid_band, kClosureThreads, band_smem, s, A.programmatic, A, M);
    if (e == cudaSuccess) e = launch_maybe_programmatic(rec, B.grid, 32 * B.warps, smem, s, A.programmatic, A, M);
    return e;
}

// Launch shape of the batch form for a work list of `items` items and `pairs` band jobs: as many blocks
// as reside; fewer warps per block where the items would otherwise leave SMs without one.
ClosureBatchShape closure_batch_shape(int tsize, int nR, int n2, int n3, int items, int pairs, int inline_band, int n_sm) {
    ClosureBatchShape B{};
    B.inline_band = inline_band;
    B.warps = kClosureWarps;
    while (B.warps > 1 && items < 2 * B.warps * n_sm) B.warps /= 2;
    const size_t smem = closure_records_smem(nR, n2, n3, B.warps, tsize);
    auto resident = [](const void* k, int threads, size_t sm) {
        int n = 0;
        if (allow_dynamic_smem(k, sm) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, sm) != cudaSuccess) {
            cudaGetLastError();
            return 4;
        }
        return n > 0 ? n : 1;
    };
    const void* rec = tsize == 4 ? (const void*)closure_records<float>(inline_band) : (const void*)closure_records<double>(inline_band);
    const void* bk = tsize == 4 ? (const void*)closure_band_kernel<float> : (const void*)closure_band_kernel<double>;
    auto clamp = [](long long need, long long most) { return (int)(need < 1 ? 1 : need < most ? need : most); };
    B.grid = clamp((items + B.warps - 1) / B.warps, (long long)n_sm * resident(rec, 32 * B.warps, smem));
    B.grid_band = clamp((pairs + kClosureWarps - 1) / kClosureWarps,
                        (long long)n_sm * resident(bk, kClosureThreads, closure_smem_bytes(nR, n2, n3, 0, 0, tsize)));
    return B;
}

cudaError_t plan_closure(int tsize, size_t smem) {
    return allow_dynamic_smem(tsize == 4 ? (const void*)closure_kernel<float> : (const void*)closure_kernel<double>, smem);
}

int closure_blocks_per_sm(int tsize, size_t smem) {
    int n = 0;
    const cudaError_t e = tsize == 4 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, closure_kernel<float>, kClosureThreads, smem)
                                     : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, closure_kernel<double>, kClosureThreads, smem);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 8;
    }
    return n > 0 ? n : 1;
}

// ------------------------------------------------------------------------------ FM weights
// The Fischer-Methfessel band of one instance (Eq. fm, App. A), in FP64, stored in the
// populations' precision: a block per cell, the volumes U_i(R_f[j]) of the cell's ball inside the
// faces of its band into shared memory, then W_ij = norm (U_i(R_f[j+1]) - U_i(R_f[j])) over the
// stored extent (zero beyond the domain), the rest of the row zero.  Rc: cell centres (stride
// rc_stride), Rf: the N + 1 faces, blo: (first column, stored extent) per cell.
template <typename T>
__global__ void fm_band_kernel(const double* __restrict__ Rc, int rc_stride, const double* __restrict__ Rf, int N,
                               int sphere, double sigma, int width, const int2* __restrict__ blo, T* __restrict__ W,
                               FmRule rule) {
    extern __shared__ double U[];  // width + 1 values
    const double norm = 3.0 / (4.0 * kFmPi * sigma * sigma * sigma);
    for (int i = blockIdx.x; i < N; i += gridDim.x) {
        const int lo = blo[i].x, cnt = blo[i].y;
        const double d = Rc[(long long)i * rc_stride];
        for (int t = threadIdx.x; t <= cnt; t += blockDim.x) {
            const int j = min(lo + t, N);
            U[t] = fm_volume_inside(sphere, sigma, d, Rf[j], rule);
        }
        __syncthreads();
        for (int t = threadIdx.x; t < width; t += blockDim.x) {
            const double w = (t < cnt && lo + t < N) ? norm * (U[t + 1] - U[t]) : 0.0;
            W[(long long)i * width + t] = (T)w;
        }
        __syncthreads();
    }
}

cudaError_t launch_fm_band(int tsize, const double* Rc, int rc_stride, const double* Rf, int N, int sphere, double sigma,
                           int width, const int2* blo, void* W, const FmRule& rule, int grid, cudaStream_t s) {
    const size_t smem = (size_t)(width + 1) * sizeof(double);
    if (tsize == 4) {
        if (const cudaError_t e = allow_dynamic_smem((const void*)fm_band_kernel<float>, smem)) return e;
        fm_band_kernel<float><<<grid, 128, smem, s>>>(Rc, rc_stride, Rf, N, sphere, sigma, width, blo, (float*)W, rule);
    } else {
        if (const cudaError_t e = allow_dynamic_smem((const void*)fm_band_kernel<double>, smem)) return e;
        fm_band_kernel<double><<<grid, 128, smem, s>>>(Rc, rc_stride, Rf, N, sphere, sigma, width, blo, (double*)W, rule);
    }
    return cudaPeekAtLastError();
}

size_t closure_smem(int nR, int n2, int n3, int max_union, int wst_elems, int tsize) {
    return closure_smem_bytes(nR, n2, n3, max_union, wst_elems, tsize);
}

void launch_residual(const double* sums, int slices, const InstDev* inst, const double* geo, double* prev, double* out,
                     int n_inst, int save, cudaStream_t s) {
    residual_kernel<<<n_inst < 1024 ? n_inst : 1024, 256, 0, s>>>(sums, slices, inst, geo, prev, out, n_inst, save);
}

// Populations of one precision copied into the other (rounding to nearest for FP64 -> FP32).
template <typename A, typename B>
__global__ void convert_kernel(const A* __restrict__ src, B* __restrict__ dst, long long n, double scale) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        dst[i] = (B)((double)src[i] * scale);
}

void launch_convert(const void* src, int src_fp32, void* dst, int dst_fp32, long long n, cudaStream_t s, double scale) {
    const long long g = (n + 255) / 256;
    const int grid = (int)(g < 8192 ? (g > 0 ? g : 1) : 8192);
    if (src_fp32 && !dst_fp32)
        convert_kernel<float, double><<<grid, 256, 0, s>>>((const float*)src, (double*)dst, n, scale);
    else if (!src_fp32 && dst_fp32)
        convert_kernel<double, float><<<grid, 256, 0, s>>>((const double*)src, (float*)dst, n, scale);
    else if (src_fp32)
        convert_kernel<float, float><<<grid, 256, 0, s>>>((const float*)src, (float*)dst, n, scale);
    else
        convert_kernel<double, double><<<grid, 256, 0, s>>>((const double*)src, (double*)dst, n, scale);
}

template void launch_ca<float>(const double*, const void*, double*, int, int, cudaStream_t, double*);
template void launch_ca<double>(const double*, const void*, double*, int, int, cudaStream_t, double*);
template void launch_dens_from_sums<float>(const double*, float*, long long, cudaStream_t);
template void launch_dens_from_sums<double>(const double*, double*, long long, cudaStream_t);
template void launch_moments<float>(const float*, double*, float*, void*, long long, int, const double*, const MomSet&,
                                    cudaStream_t);
template void launch_moments<double>(const double*, double*, double*, void*, long long, int, const double*,
                                     const MomSet&, cudaStream_t);
template cudaError_t launch_closure<float>(const ClosureArgs&, const MomSet&, int, int, size_t, cudaStream_t);
template cudaError_t launch_closure<double>(const ClosureArgs&, const MomSet&, int, int, size_t, cudaStream_t);
template cudaError_t launch_closure_batch<float>(const ClosureArgs&, const MomSet&, const ClosureBatchShape&, cudaStream_t);
template cudaError_t launch_closure_batch<double>(const ClosureArgs&, const MomSet&, const ClosureBatchShape&, cudaStream_t);

}  // namespace fdlb
