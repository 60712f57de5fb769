// Device helpers shared by the kernel translation units: PTX wrappers for the bulk-copy
// engine and mbarriers, the WENO5 reconstruction, the Carnahan-Starling contact value and
// warp reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace fdlb {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
// One-dimensional bulk copy global -> shared by the TMA engine; completion is counted in
// bytes on `bar`.  Both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}
// Asks the bulk-copy engine to bring `bytes` at `src` into L2 (a hint: no completion, no effect on
// results).  Address 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t phase) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(phase)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Bounded wait: gives up after 1 s of global time (a copy completes in microseconds), or after
// 2^22 tries (each suspends for a hardware-chosen interval) whichever comes first.  Returns false
// if the phase never completed.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* bar, uint32_t phase) {
    if (mbar_try_wait(bar, phase)) return true;
    const unsigned long long t0 = global_ns();
    for (int it = 1; it < (1 << 22); ++it) {
        if (mbar_try_wait(bar, phase)) return true;
        if ((it & 63) == 0 && global_ns() - t0 > 1000000000ull) return false;
    }
    return false;
}

// Programmatic dependent launch.  A kernel launched with programmatic stream serialization may
// start while its predecessor in the stream is still running: it does only work that reads
// nothing the predecessor writes (constant tables into shared memory), then pdl_wait(), which
// returns once the predecessor grid has completed and its memory is visible.  pdl_trigger() lets
// the successor be scheduled as soon as every block of this grid has started.  Both are no-ops
// for a kernel launched the ordinary way.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// TF32 tensor-core helpers: round to TF32 (ties away), and the warp-wide m16n8k8 product with
// FP32 accumulation.  Fragment ownership (g = lane / 4, t = lane % 4): A (16 x 8, row major)
// a0 (g, t), a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4); B (8 x 8) b0 (t, g), b1 (t + 4, g);
// C, D (16 x 8) c0 (g, 2t), c1 (g, 2t + 1), c2 (g + 8, 2t), c3 (g + 8, 2t + 1).
__device__ __forceinline__ uint32_t to_tf32(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <typename T>
__device__ __forceinline__ T ldg_t(const T* p) {
    return __ldg(p);
}

// A product that is rounded by itself: never contracted into a following addition, so code that must
// give the same bits from every kernel it is inlined into says with fma() and mul_rn() what is fused.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

__device__ __forceinline__ float ratio_fast(float a, float b) { return __fdividef(a, b); }
__device__ __forceinline__ double ratio_fast(double a, double b) { return a / b; }

// ---- pairs of lanes: two momenta of a vector per instruction.  FP32 pairs use the packed FP32x2
// operations of the sm_100 family (__ffma2_rn, __fadd2_rn, __fmul2_rn: one issue slot for two
// FP32 operations, each lane rounded like the scalar operation); FP64 pairs are two scalar
// operations.  Every operation is written out (nothing is left to the compiler's contraction),
// so a lane's result is the same whichever pair it travels in.
template <typename T>
struct PairT;
template <>
struct PairT<float> {
    using type = float2;
};
template <>
struct PairT<double> {
    using type = double2;
};
template <typename T>
using Pair = typename PairT<T>::type;

__device__ __forceinline__ float2 p_make(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ double2 p_make(double a, double b) { return make_double2(a, b); }
__device__ __forceinline__ float2 p_splat(float a) { return make_float2(a, a); }
__device__ __forceinline__ double2 p_splat(double a) { return make_double2(a, a); }
__device__ __forceinline__ float2 p_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 p_fma(double2 a, double2 b, double2 c) {
    return make_double2(__fma_rn(a.x, b.x, c.x), __fma_rn(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ double2 p_add(double2 a, double2 b) { return make_double2(__dadd_rn(a.x, b.x), __dadd_rn(a.y, b.y)); }
__device__ __forceinline__ float2 p_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ double2 p_mul(double2 a, double2 b) { return make_double2(__dmul_rn(a.x, b.x), __dmul_rn(a.y, b.y)); }
// a - b: b times -1 is exact, so the fused form rounds once, like a subtraction
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ double2 p_sub(double2 a, double2 b) { return make_double2(__dsub_rn(a.x, b.x), __dsub_rn(a.y, b.y)); }
__device__ __forceinline__ float2 p_min(float2 a, float2 b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }
// Approximate FP32 reciprocal (the PTX rcp.approx instruction: at most one unit in the last place
// off, subnormals flushed to zero).
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
// a / b lane by lane, as the product with the approximate reciprocal (the operands here are normal
// numbers well inside the range).
__device__ __forceinline__ float2 p_ratio(float2 a, float2 b) {
    return __fmul2_rn(a, make_float2(rcp_approx(b.x), rcp_approx(b.y)));
}

// Fifth-order WENO reconstruction (Jiang & Shu 1996; epsilon 1e-6, power 2) of the face value on
// the window w0..w4 in ascending cell order, for either upwind direction: sigma = +1 gives the value at
// the right face of w2's cell, from the left; sigma = -1 the value at its left face, from the right.
// The three smoothness indicators belong to the left, centre and right stencils whatever the direction,
// and every candidate value is (D_k + 12 w2 -+ 3 sigma t_k) / 2 with D_k the stencil's second
// difference and t_k the first-difference part of its indicator, so the value is
// w2 + sum_k a_k X_k / (12 sum_k a_k), X_k = D_k +- 3 sigma t_k.  The linear weights follow the
// direction: (dL, dC, dR) = (0.1, 0.6, 0.3) or (0.3, 0.6, 0.1); s3 = 3 sigma.  Indicators are
// taken four times over (e4 + 13/3 D^2 + t^2, e4 = 4 eps): the normalised weights are unchanged.
// The reconstruction is homogeneous of degree one in the window once eps scales with its square:
// the value for c w0..c w4 with c^2 e4 is c times the value for w0..w4 with e4.  The window's
// first difference enters negated (w0 - w1), and so does the centre stencil's first-difference
// part (-tC = d1 + d2), which the indicators square and the candidate values take with the
// opposite sign: no negation is ever formed.
//
// FP32: a pair of momenta, one packed operation per step.  The nonlinear weights d_k / E_k^2 are
// scaled by the square of the smallest indicator, which leaves the normalised weights unchanged and
// keeps every intermediate in [0, 1] (no overflow for large populations).  ns3 = -3 sigma.
__device__ __forceinline__ float2 weno5_pair(float2 w0, float2 w1, float2 w2, float2 w3, float2 w4, float2 s3, float2 ns3,
                                             float2 dL, float2 dR, float2 e4) {
    using P = float2;
    const P nd0 = p_sub(w0, w1), d1 = p_sub(w2, w1), d2 = p_sub(w3, w2), d3 = p_sub(w4, w3);
    const P D1 = p_add(d1, nd0), D2 = p_sub(d2, d1), D3 = p_sub(d3, d2);
    const P tL = p_fma(p_splat(3.f), d1, nd0);    // 3 d1 - d0
    const P ntC = p_add(d1, d2);                    // -tC
    const P tR = p_fma(p_splat(-3.f), d2, d3);     // d3 - 3 d2
    const P c = p_splat((float)(13.0 / 3.0));
    const P EL = p_fma(tL, tL, p_fma(p_mul(c, D1), D1, e4));
    const P EC = p_fma(ntC, ntC, p_fma(p_mul(c, D2), D2, e4));
    const P ER = p_fma(tR, tR, p_fma(p_mul(c, D3), D3, e4));
    const P m = p_min(EL, p_min(EC, ER));
    const P sL = p_ratio(m, EL), sC = p_ratio(m, EC), sR = p_ratio(m, ER);
    const P aL = p_mul(dL, p_mul(sL, sL)), aC = p_mul(p_splat(0.6f), p_mul(sC, sC)), aR = p_mul(dR, p_mul(sR, sR));
    const P XL = p_fma(s3, tL, D1), XC = p_fma(s3, ntC, D2), XR = p_fma(ns3, tR, D3);
    const P num = p_fma(aR, XR, p_fma(aC, XC, p_mul(aL, XL)));
    const P den = p_mul(p_splat(12.f), p_add(p_add(aL, aC), aR));
    return p_add(w2, p_ratio(num, den));
}

// FP64: the FP64 unit takes a warp instruction every 16 cycles, so its operations are what a stage
// costs, and a division is a chain of them.  The weights are taken without a quotient, d_k times the square
// of the product of the other two indicators, with the indicators' exponents lowered by the smallest one's
// (an integer operation on the high words, exact) and held below 2^200, so the products stay within the range.
// A stencil that much rougher than the smoothest has a weight below 2^-400 and is given none: held at 2^200 it
// would still count where its candidate differs by more than 2^347.  One division remains of four.
constexpr int kF64Rough = 200 << 20;
__device__ __forceinline__ int f64_above(double E, int base) { return __double2hiint(E) - base; }  // (>= 0: base is the least)
__device__ __forceinline__ double f64_lowered(double E, int above) {
    return __hiloint2double(min(above, kF64Rough) + (1023 << 20), __double2loint(E));
}
__device__ __forceinline__ double weno5_f64(double w0, double w1, double w2, double w3, double w4, double s3, double dL,
                                            double dR, double e4) {
    const double nd0 = __dsub_rn(w0, w1), d1 = __dsub_rn(w2, w1), d2 = __dsub_rn(w3, w2), d3 = __dsub_rn(w4, w3);
    const double D1 = __dadd_rn(d1, nd0), D2 = __dsub_rn(d2, d1), D3 = __dsub_rn(d3, d2);
    const double tL = __fma_rn(3.0, d1, nd0), ntC = __dadd_rn(d1, d2), tR = __fma_rn(-3.0, d2, d3);
    const double c = 13.0 / 3.0;
    double EL = __fma_rn(tL, tL, __fma_rn(__dmul_rn(c, D1), D1, e4));
    double EC = __fma_rn(ntC, ntC, __fma_rn(__dmul_rn(c, D2), D2, e4));
    double ER = __fma_rn(tR, tR, __fma_rn(__dmul_rn(c, D3), D3, e4));
    // (positive doubles order like their high words; a window that is not finite keeps the value not
    // finite through the candidates)
    const int hm = min(__double2hiint(EL), min(__double2hiint(EC), __double2hiint(ER)));
    const int base = hm & 0x7ff00000, xL = f64_above(EL, base), xC = f64_above(EC, base), xR = f64_above(ER, base);
    EL = f64_lowered(EL, xL);
    EC = f64_lowered(EC, xC);
    ER = f64_lowered(ER, xR);
    const double pL = __dmul_rn(EC, ER), pC = __dmul_rn(EL, ER), pR = __dmul_rn(EL, EC);
    // (a candidate that is not finite gives a product with a weight of zero that is not a number)
    const double aL = xL > kF64Rough ? 0.0 : __dmul_rn(dL, __dmul_rn(pL, pL));
    const double aC = xC > kF64Rough ? 0.0 : __dmul_rn(0.6, __dmul_rn(pC, pC));
    const double aR = xR > kF64Rough ? 0.0 : __dmul_rn(dR, __dmul_rn(pR, pR));
    const double XL = __fma_rn(s3, tL, D1), XC = __fma_rn(s3, ntC, D2), XR = __fma_rn(-s3, tR, D3);
    const double num = __fma_rn(aR, XR, __fma_rn(aC, XC, __dmul_rn(aL, XL)));
    return __fma_rn(num / __dadd_rn(__dadd_rn(aL, aC), aR), 1.0 / 12.0, w2);
}
__device__ __forceinline__ double2 weno5_pair(double2 w0, double2 w1, double2 w2, double2 w3, double2 w4, double2 s3,
                                              double2, double2 dL, double2 dR, double2 e4) {
    return make_double2(weno5_f64(w0.x, w1.x, w2.x, w3.x, w4.x, s3.x, dL.x, dR.x, e4.x),
                        weno5_f64(w0.y, w1.y, w2.y, w3.y, w4.y, s3.y, dL.y, dR.y, e4.y));
}
// One momentum (the wall fluxes).
__device__ __forceinline__ double weno5_one(double w0, double w1, double w2, double w3, double w4, double s3, double dL,
                                            double dR, double e4) {
    return weno5_f64(w0, w1, w2, w3, w4, s3, dL, dR, e4);
}
__device__ __forceinline__ float weno5_one(float w0, float w1, float w2, float w3, float w4, float s3, float dL, float dR,
                                           float e4) {
    return weno5_pair(p_splat(w0), p_splat(w1), p_splat(w2), p_splat(w3), p_splat(w4), p_splat(s3), p_splat(-s3), p_splat(dL),
                      p_splat(dR), p_splat(e4)).x;
}

// ---- wide accumulators: plain FP64 for FP64 populations; for FP32 populations a double-float
// (hi + lo, about 44 significant bits) on the FP32 pipe, because FP64 arithmetic on GB300 costs
// 64 cycles per dependent operation and about 440 per division.  The error-free transformations
// are Knuth's TwoSum and the fused-multiply-add TwoProduct (Dekker 1971; the double-double
// algorithms of Hida, Li and Bailey 2001, restated for float pairs).
template <typename T>
struct Wide;
template <>
struct Wide<double> {
    double v;
};
template <>
struct Wide<float> {
    float hi, lo;
};

__device__ __forceinline__ Wide<double> w_from(double s, double*) { return {s}; }
__device__ __forceinline__ Wide<float> w_from(double s, float*) {
    const float hi = __double2float_rn(s);
    return {hi, __double2float_rn(s - (double)hi)};
}
__device__ __forceinline__ Wide<double> w_from_t(double x) { return {x}; }
__device__ __forceinline__ Wide<float> w_from_t(float x) { return {x, 0.f}; }
__device__ __forceinline__ double w_hi(Wide<double> a) { return a.v; }
__device__ __forceinline__ float w_hi(Wide<float> a) { return a.hi; }
__device__ __forceinline__ Wide<double> w_add(Wide<double> a, Wide<double> b) { return {a.v + b.v}; }
__device__ __forceinline__ Wide<double> w_sub(Wide<double> a, Wide<double> b) { return {a.v - b.v}; }
__device__ __forceinline__ Wide<double> w_mul(Wide<double> a, Wide<double> b) { return {__dmul_rn(a.v, b.v)}; }
__device__ __forceinline__ Wide<double> w_div(Wide<double> a, Wide<double> b) { return {a.v / b.v}; }
__device__ __forceinline__ Wide<double> w_scale(Wide<double> a, double c) { return {__dmul_rn(a.v, c)}; }

__device__ __forceinline__ Wide<float> w_norm(float s, float e) {  // |s| >= |e|
    const float hi = s + e;
    return {hi, e - (hi - s)};
}
__device__ __forceinline__ Wide<float> w_add(Wide<float> a, Wide<float> b) {
    const float s = a.hi + b.hi, v = s - a.hi;
    float e = (a.hi - (s - v)) + (b.hi - v);
    e += a.lo + b.lo;
    return w_norm(s, e);
}
__device__ __forceinline__ Wide<float> w_sub(Wide<float> a, Wide<float> b) { return w_add(a, {-b.hi, -b.lo}); }
__device__ __forceinline__ Wide<float> w_mul(Wide<float> a, Wide<float> b) {
    const float p = __fmul_rn(a.hi, b.hi);
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return w_norm(p, e);
}
__device__ __forceinline__ Wide<float> w_scale(Wide<float> a, float c) {
    const float p = __fmul_rn(a.hi, c);
    const float e = fmaf(a.lo, c, fmaf(a.hi, c, -p));
    return w_norm(p, e);
}
// a / b: a first quotient, the remainder a - q1 b in double-float, a correction.  The two
// quotients need only single-precision accuracy (the remainder is exact to the double-float
// level), so they are the fast ones.
__device__ __forceinline__ Wide<float> w_div(Wide<float> a, Wide<float> b) {
    const float q1 = __fdividef(a.hi, b.hi);
    const Wide<float> r = w_sub(a, w_scale(b, q1));
    return w_norm(q1, __fdividef(r.hi, b.hi));
}
__device__ __forceinline__ Wide<double> w_shfl_xor(Wide<double> a, int o) { return {__shfl_xor_sync(0xffffffffu, a.v, o)}; }
__device__ __forceinline__ Wide<float> w_shfl_xor(Wide<float> a, int o) {
    return {__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

template <typename T>
__device__ __forceinline__ T chi_cs_t(T eta) {
    const T om = T(1) - eta;
    return (T(2) - eta) / (T(2) * om * om * om);
}

__device__ __forceinline__ double chi_cs(double eta) {
    const double om = 1.0 - eta;
    return (2.0 - eta) / (2.0 * om * om * om);
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums of 16 values over the 32 lanes of a warp, transposed: at every level of the butterfly a
// lane keeps half of its values and sends the other half, so the warp needs 16 shuffles instead
// of 16 x 5.  Lane L returns the sum of value (L >> 1).  Fixed order: deterministic.
template <typename T>
__device__ __forceinline__ T warp_sum16_transposed(const T (&v)[16], int lane) {
    T w8[8], w4[4], w2[2];
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        const T send = b4 ? v[t] : v[t + 8], keep = b4 ? v[t + 8] : v[t];
        w8[t] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        const T send = b3 ? w8[t] : w8[t + 4], keep = b3 ? w8[t + 4] : w8[t];
        w4[t] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
        const T send = b2 ? w4[t] : w4[t + 2], keep = b2 ? w4[t + 2] : w4[t];
        w2[t] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    const T send = b1 ? w2[0] : w2[1], keep = b1 ? w2[1] : w2[0];
    const T w1 = keep + __shfl_xor_sync(0xffffffffu, send, 2);
    return w1 + __shfl_xor_sync(0xffffffffu, w1, 1);
}

}  // namespace fdlb
