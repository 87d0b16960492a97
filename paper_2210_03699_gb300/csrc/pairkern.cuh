// Dense pair-sum core shared by the single-system operator (pairsum.cu) and
// the multi-slot engine (engine.cu): kernel constants, bulk-copy/mbarrier
// helpers, float-float arithmetic, the three pair policies and one work item
// of the tiled pair sum.  Internal to the library.
#pragma once

#include "common.cuh"

namespace ctr {
namespace pk {

constexpr int kThreads = 256;
constexpr uint32_t kWaitLimit = 1u << 22;   // default polls of a bounded mbarrier wait
constexpr int kExpHi = 64;      // e^{-k}, k = 0..63
constexpr int kExpLo = 1024;    // e^{-k/1024}, k = 0..1023
constexpr int kExp2 = 1024;     // FP64 tables: 2^{-k/1024} (double), then its relative rounding error (float)
constexpr int kExp2F2 = kExp2 + kExp2 / 2;   // their size in float2

// Flags of an excluded pair (Exclusions): the source is left out of the target's row, the target of the source's
enum : int { kOutTarget = 1, kOutSource = 2 };

struct PairConsts {
    float c1f, c2f, kappaf, kl2f;    // eps_E/eps_I, eps_I/eps_E, kappa, -kappa log2(e)
    double c1, c2, kappa;
    float2 c1d, c2d, kappad;         // float-float copies
    double k2;                       // kappa log2(e), rounded; k2f: in FP32; k2d: -ln 2 times its rounding error
    float k2f, k2d;
    double c1kap;                    // (eps_E/eps_I) kappa
    const float2* exp_tab;           // exponential tables of the arithmetic (float-float or FP64), global
    // the FP32 values duplicated into both halves of a 64-bit word (f32x2 operands)
    unsigned long long one2, mone2, three2, mthree2, c1x2, nc1x2, c2x2, kap2, kl2x2;
    unsigned long long c1kap2;       // (eps_E/eps_I) kappa
    uint32_t wait_limit;             // polls of a source-tile wait before the block gives up
    uint32_t pad_;
};

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
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
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
// Bounded wait: false after `limit` polls (each poll may suspend briefly).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit = kWaitLimit) {
    for (uint32_t it = 0; it < limit; ++it)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

__device__ __forceinline__ float rsqrt_sfu(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_sfu(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ------------------------------------------------------------------ f32x2 arithmetic
// Two FP32 values in one 64-bit register pair, one IEEE round-to-nearest operation per half
// (add/sub/mul/fma.rn.f32x2): half the issue slots of two scalar instructions.
using u64 = unsigned long long;
__device__ __forceinline__ u64 pk2(float a, float b) {
    u64 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void up2(u64 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
// -v as -0 - v: folded into the operand of the instruction that uses it (measured: no slot of its own)
__device__ __forceinline__ u64 neg2(u64 v) { return sub2(0x8000000080000000ull, v); }
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {   // a * b + c
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ u64 rsqrt2(u64 v) {
    float a, b;
    up2(v, a, b);
    return pk2(rsqrt_sfu(a), rsqrt_sfu(b));
}
__device__ __forceinline__ u64 ex2_2(u64 v) {
    float a, b;
    up2(v, a, b);
    return pk2(ex2_sfu(a), ex2_sfu(b));
}

// ------------------------------------------------------------------ float-float arithmetic
// A value is hi + lo with |lo| <= ulp(hi)/2.  Error-free transformations use
// explicitly rounded intrinsics so that nothing is fused or reassociated.
struct F2 {
    float hi, lo;
};
__device__ __forceinline__ F2 f2(float2 v) { return F2{v.x, v.y}; }
__device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return F2{s, e};
}
__device__ __forceinline__ F2 fast_two_sum(float a, float b) {   // |a| >= |b|, or a == 0
    const float s = __fadd_rn(a, b);
    return F2{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ F2 two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return F2{p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ F2 neg(F2 a) { return F2{-a.hi, -a.lo}; }
__device__ __forceinline__ F2 add(F2 a, F2 b) {
    const F2 s = two_sum(a.hi, b.hi);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo)));
}
__device__ __forceinline__ F2 sub(F2 a, F2 b) { return add(a, neg(b)); }
__device__ __forceinline__ F2 mul(F2 a, F2 b) {
    const F2 p = two_prod(a.hi, b.hi);
    return fast_two_sum(p.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo)));
}
// Lazy forms for the symmetric pair terms.  A lazy value is hi + lo with |lo|
// a few ulp(hi) instead of at most ulp(hi)/2: it carries the same value to the
// same accuracy, and a product of two lazy values loses only the dropped
// lo * lo term (relative 2^-44 or less).  Results that meet a cancellation
// (differences, 1 - E, 3 - E q) go through the normalised add, whose two_sum
// is exact for any inputs.
__device__ __forceinline__ F2 mull(F2 a, F2 b) {
    const F2 p = two_prod(a.hi, b.hi);
    return F2{p.hi, __fmaf_rn(a.hi, b.lo, __fmaf_rn(a.lo, b.hi, p.lo))};
}
// acc += x without renormalising acc: exact two_sum of the high parts, plain sum of the low parts
__device__ __forceinline__ void acc_add(F2& acc, F2 x) {
    const F2 s = two_sum(acc.hi, x.hi);
    acc.hi = s.hi;
    acc.lo = __fadd_rn(acc.lo, __fadd_rn(s.lo, x.lo));
}
// Sums and differences without the final renormalisation: exact two_sum of the high parts, plain sum of
// the low parts.
__device__ __forceinline__ F2 addl(F2 a, F2 b) {
    const F2 s = two_sum(a.hi, b.hi);
    return F2{s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ F2 subl(F2 a, F2 b) { return addl(a, neg(b)); }
// 1 - a for 0 <= a <= 1 (1 - a.hi and its rounding error are exact), and for any a
__device__ __forceinline__ F2 one_minus(F2 a) {
    const float s = __fsub_rn(1.0f, a.hi);
    return F2{s, __fsub_rn(__fsub_rn(__fsub_rn(1.0f, s), a.hi), a.lo)};
}
__device__ __forceinline__ F2 one_minus_any(F2 a) {
    const F2 s = two_sum(1.0f, -a.hi);
    return F2{s.hi, __fsub_rn(s.lo, a.lo)};
}
// acc += a b: the product's leading part by an exact two_sum, everything else into the low part
__device__ __forceinline__ void acc_mul(F2& acc, F2 a, F2 b) { acc_add(acc, mull(a, b)); }
// a0 b0 + a1 b1 + a2 b2, unnormalised: the low part is within a few 2^-24 of the largest product, so what a
// later lazy product drops stays below 2^-46 of the factors' own scale even where the sum cancels
__device__ __forceinline__ F2 dot3l(F2 a0, F2 a1, F2 a2, F2 b0, F2 b1, F2 b2) {
    const F2 p0 = two_prod(a0.hi, b0.hi), p1 = two_prod(a1.hi, b1.hi), p2 = two_prod(a2.hi, b2.hi);
    const F2 s = two_sum(p0.hi, p1.hi);
    const F2 t = two_sum(s.hi, p2.hi);
    float e = __fadd_rn(__fadd_rn(p0.lo, p1.lo), __fadd_rn(p2.lo, __fadd_rn(s.lo, t.lo)));
    e = __fmaf_rn(a0.hi, b0.lo, __fmaf_rn(a0.lo, b0.hi, e));
    e = __fmaf_rn(a1.hi, b1.lo, __fmaf_rn(a1.lo, b1.hi, e));
    e = __fmaf_rn(a2.hi, b2.lo, __fmaf_rn(a2.lo, b2.hi, e));
    return F2{t.hi, e};
}
// a0^2 + a1^2 + a2^2, unnormalised (the two halves of each cross product are equal)
__device__ __forceinline__ F2 sq3l(F2 a0, F2 a1, F2 a2) {
    const F2 p0 = two_prod(a0.hi, a0.hi), p1 = two_prod(a1.hi, a1.hi), p2 = two_prod(a2.hi, a2.hi);
    const F2 s = two_sum(p0.hi, p1.hi);
    const F2 t = two_sum(s.hi, p2.hi);
    const float x = __fmaf_rn(a2.hi, a2.lo, __fmaf_rn(a1.hi, a1.lo, __fmul_rn(a0.hi, a0.lo)));
    const float e = __fadd_rn(__fadd_rn(p0.lo, p1.lo), __fadd_rn(p2.lo, __fadd_rn(s.lo, t.lo)));
    return F2{t.hi, __fmaf_rn(2.0f, x, e)};
}
// 1/sqrt(x), normalised: SFU seed y (rel. err < 2^-22), its residual e = 1 - x y^2 (1 - x.hi w is exact, the
// rest follows in FP32), y + y e (1/2 + 3/8 e): truncation below 2^-64
__device__ __forceinline__ F2 rsqrt_ff(F2 x) {
    const float y = rsqrt_sfu(x.hi);
    const F2 w = two_prod(y, y);
    const float t = __fmul_rn(x.hi, w.hi);
    const float l = __fmaf_rn(x.lo, w.hi, __fmaf_rn(x.hi, w.lo, __fmaf_rn(x.hi, w.hi, -t)));
    const float e = __fsub_rn(__fsub_rn(1.0f, t), l);
    return fast_two_sum(y, __fmul_rn(__fmul_rn(__fmul_rn(0.5f, y), e), __fmaf_rn(0.75f, e, 1.0f)));
}
// e^{-x}, x >= 0: x = k/1024 + a + x.lo (k nearest to 1024 x.hi, a exact), e^{-x} = e^{-(k>>10)} e^{-(k&1023)/1024} e^{-f},
// e^{-f} = 1 - a - x.lo + q with q = f^2 (1/2 - f/6 + f^2/24), f = a + x.lo, |f| <= 1/2048 (truncation < 3e-19).
// x is capped at 63.9, where e^{-x} < 2e-28: the cap keeps the table index in range for any input
// (fminf returns the number when the other operand is a NaN).  The last factor is normalised: its low part holds q
// and x.lo, and the product drops low times low, which otherwise is most of the error (rms of E, unnormalised
// against normalised: 4.2e-15 : 3.8e-15 for x < 0.04, 7.6e-15 : 5.2e-15 below 8, 4.6e-14 : 1.9e-14 below 60).
// Lazy result.
__device__ __forceinline__ F2 exp_neg_ffl(F2 x, const float2* tab) {
    const float xh = fminf(x.hi, 63.9f);
    const float xl = x.hi > 63.9f ? 0.f : x.lo;
    const float t = __fmaf_rn(xh, 1024.f, 12582912.f);   // 1.5 * 2^23: round(x * 1024) in the mantissa
    const int k = __float_as_int(t) - 0x4B400000;
    const float a = __fmaf_rn(__fsub_rn(t, 12582912.f), -1.0f / 1024.f, xh);
    const float f = __fadd_rn(a, xl);
    const float poly = __fmaf_rn(__fmaf_rn(f, 1.0f / 24.0f, -1.0f / 6.0f), f, 0.5f);
    const float q = __fmul_rn(__fmul_rn(f, f), poly);
    const float s = __fsub_rn(1.0f, a);
    const float l = __fadd_rn(__fsub_rn(__fsub_rn(__fsub_rn(1.0f, s), a), xl), q);
    return mull(mull(f2(tab[k >> 10]), f2(tab[kExpHi + (k & (kExpLo - 1))])), fast_two_sum(s, l));
}

// ------------------------------------------------------------------ FP64 arithmetic
// The FP64 pipe (1.9 operations a clock and SM, conversions included, against about 110 on the FP32 pipe)
// bounds the FP64 kernels, so what need not run on it does not: seeds come from the SFU, indices and
// high-order terms from FP32, conversions are bit operations.
// FP64 bits of a positive normal FP32 value (0 becomes 2^-127, nothing at the places this is used)
__device__ __forceinline__ double widen_pos(float v) {
    const uint32_t b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}
__device__ __forceinline__ double widen(float v) {
    const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
    return __hiloint2double((int)((b & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(b << 29));
}
// the leading 24 bits of a positive FP64 value, kept within the FP32 range
__device__ __forceinline__ float narrow_pos(double v) {
    const int hi = min(max(__double2hiint(v), 0x38100000), 0x47e00000);
    return __uint_as_float(__funnelshift_l((uint32_t)__double2loint(v), (uint32_t)(hi - 0x38000000), 3));
}
// 1/sqrt(x): SFU seed y of 20 bits (its square is exact in FP64), residual e = 1 - x y^2, and the binomial series
// of (1 - e)^(-1/2) to its second power: y (1 + e/2 + 3/8 e^2); five operations.  rms error 0.42 x 2^-53, largest
// 1.0 x 2^-53.
__device__ __forceinline__ double rsqrt_d(double x) {
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    const double e = fma(-x, y * y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
// 2^-990 <= x < 2^990: where rsqrt_d holds (its seed and the seed's square are normal)
__device__ __forceinline__ bool rsqrt_d_range(double x) {
    return (uint32_t)__double2hiint(x) - 0x02100000u < 0x7bc00000u;
}
// e^{-kappa r} by table (Tang, "Table-driven implementation of the exponential function in IEEE floating-point
// arithmetic", ACM TOMS 15(2), 1989): 2^-i T_j 2^-f with kappa r log2(e) = i + j/1024 + f, the index from FP32, f by
// one fused operation, 2^-f - 1 = f (-ln2 + f (ln2^2/2 - f g)) by its Taylor series with g = ln2^3/6 - f ln2^4/24 in
// FP32 (f^3 g < 2^-37), corrected by the relative rounding errors of T_j and of kappa log2(e) (q's constant term);
// five FP64 operations.  Error in units of 2^-53: rms 0.42 and at most 1.03 up to kappa r = 30; the index comes from
// 24 bits of r, so f grows with kappa r, and with it g's error: at most 1.9 up to 350, 3.8 up to 680 (rms 0.60).
__device__ __forceinline__ double exp_neg_d(double r, const PairConsts& k, const float2* tab) {
    const double* T = reinterpret_cast<const double*>(tab);
    const float* tau = reinterpret_cast<const float*>(T + kExp2);
    const float rf = narrow_pos(r);
    const float y = __fmul_rn(k.k2f, rf);
    const float t = __fmaf_rn(fminf(y, 1000.f), 1024.f, 12582912.f);
    const int i = __float_as_int(t) - 0x4B400000;
    const float c = __fmul_rn(__fsub_rn(t, 12582912.f), 1.0f / 1024.f);
    const double f = fma(k.k2, r, -widen_pos(c));
    const float g = __fmaf_rn(-0.00961812910762848f, __fmaf_rn(k.k2f, rf, -c), 0.05550410866482158f);
    const double h = fma(f, fma(-f, widen_pos(g), 0.2402265069591007), -0.6931471805599453);
    const double q = fma(f, h, widen(__fmaf_rn(k.k2d, rf, tau[i & (kExp2 - 1)])));
    const double Tj = T[i & (kExp2 - 1)];
    const double s = __hiloint2double(__double2hiint(Tj) - ((i >> 10) << 20), __double2loint(Tj));
    return y < 1000.f ? fma(s, q, s) : 0.0;   // below 2^-1000: nothing
}

// ------------------------------------------------------------------ exact node accumulators
// The dense sum's partial results (an item's target sums, a symmetric tile's source sums, a far item's
// sums) are added into per-node accumulators in whatever order the blocks run.  To keep the result
// independent of that order, each contribution v (FP64) is turned into the integer round(|v| 2^kFxFrac)
// and added exactly: the integer's 32-bit chunks go to 64-bit words by atomic addition (fewer than 2^31
// contributions per word cannot carry out of it), positive and negative contributions to separate sets
// of kFxChunks words, so a contribution touches at most the three words its 53 significant bits span.
// Reading a node's sum propagates the carries, subtracts the two sets and rounds once to FP64.
// Range: |v| < 2^(32 kFxChunks - kFxFrac) = 2^72; below 2^-kFxFrac a contribution is rounded to a
// multiple of 2^-kFxFrac = 7.5e-37.  A non-finite or out-of-range contribution marks the node
// (its last word), and the node then reads as NaN, as an FP64 sum of such a term would.
// Layout: word k of sign set g (0 positive, 1 negative) of sum c (0, 1) of node position p at
// acc[((2 c + g) kFxChunks + k) * stride + p], the mark at acc[4 kFxChunks * stride + p]:
// kFxWords 64-bit words per node.
constexpr int kFxChunks = 6;
constexpr int kFxFrac = 120;
constexpr int kFxWords = 4 * kFxChunks + 1;

__device__ __forceinline__ void fx_add(unsigned long long* __restrict__ acc, int64_t stride, int c, double v) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
    const int ex = (int)((bits >> 52) & 0x7ff);
    if (ex == 0x7ff) {   // not finite
        atomicOr(acc + (int64_t)(4 * kFxChunks) * stride, 1ull);
        return;
    }
    unsigned long long m = bits & ((1ull << 52) - 1);
    if (ex != 0) m |= 1ull << 52;
    if (m == 0) return;
    int sh = (ex != 0 ? ex - 1075 : -1074) + kFxFrac;   // |v| 2^kFxFrac = m 2^sh
    if (sh < 0) {                                       // below the resolution: round to nearest
        if (sh < -60) return;
        m = (m + (1ull << (-sh - 1))) >> (-sh);
        sh = 0;
        if (m == 0) return;
    }
    if (sh + 53 > 32 * kFxChunks) {   // out of range
        atomicOr(acc + (int64_t)(4 * kFxChunks) * stride, 1ull);
        return;
    }
    unsigned long long* base = acc + (int64_t)((2 * c + (int)(bits >> 63)) * kFxChunks) * stride;
    // m 2^sh spans the 32-bit chunks k0 .. k0 + 2 (m < 2^53)
    const int k0 = sh >> 5, r = sh & 31;
    const unsigned long long lo = m << r;                       // bits 0..63 of m 2^r
    const unsigned long long hi = r ? (m >> (64 - r)) : 0ull;   // bits 64.. (m 2^r < 2^85)
    const unsigned long long ch[3] = {lo & 0xffffffffull, lo >> 32, hi};
#pragma unroll
    for (int q = 0; q < 3; ++q)
        if (ch[q] != 0 && k0 + q < kFxChunks) atomicAdd(base + (int64_t)(k0 + q) * stride, ch[q]);
}

// One sum (c) of the node at acc (stride as in fx_add), rounded to FP64: carries of both sign sets,
// positive minus negative, one rounding.  The node's words of that sum are cleared when `clear`.
__device__ __forceinline__ double fx_read_one(unsigned long long* __restrict__ acc, int64_t stride, int c,
                                              bool clear) {
    unsigned long long wp[kFxChunks], wn[kFxChunks];   // every load in flight before the first use
    unsigned long long* ap = acc + (int64_t)(2 * c) * kFxChunks * stride;
    unsigned long long* an = ap + (int64_t)kFxChunks * stride;
#pragma unroll
    for (int k = 0; k < kFxChunks; ++k) {
        wp[k] = ap[(int64_t)k * stride];
        wn[k] = an[(int64_t)k * stride];
    }
    if (clear) {
#pragma unroll
        for (int k = 0; k < kFxChunks; ++k) ap[(int64_t)k * stride] = an[(int64_t)k * stride] = 0ull;
    }
    uint32_t D[kFxChunks + 1];
    unsigned long long cp = 0, cn = 0;
    long long borrow = 0;
#pragma unroll
    for (int k = 0; k <= kFxChunks; ++k) {
        unsigned long long tp = cp, tn = cn;
        if (k < kFxChunks) {
            tp += wp[k];
            tn += wn[k];
        }
        cp = tp >> 32;
        cn = tn >> 32;
        const long long t = (long long)(tp & 0xffffffffull) - (long long)(tn & 0xffffffffull) - borrow;
        D[k] = (uint32_t)t;
        borrow = t < 0 ? 1 : 0;
    }
    const bool neg = borrow != 0;
    if (neg) {   // two's complement of the chunk string
        unsigned long long carry = 1;
#pragma unroll
        for (int k = 0; k <= kFxChunks; ++k) {
            const unsigned long long t = (unsigned long long)(uint32_t)~D[k] + carry;
            D[k] = (uint32_t)t;
            carry = t >> 32;
        }
    }
    double v = 0.0;
#pragma unroll
    for (int k = kFxChunks; k >= 0; --k) v = fma(v, 4294967296.0, (double)D[k]);
    v = ldexp(v, -kFxFrac);
    return neg ? -v : v;
}

// ------------------------------------------------------------------ finishing a row
// What the finishing kernels need besides the accumulated sum: the correction rows (CSR, weights omega11,
// omega21, omega22, omega12 of E entries each).
struct FinishRows {
    const int32_t* ptr;
    const int32_t* node;
    const double* w;
    const double* W;
    int64_t M, E;
    double h2, h3;
};

// Component c (0: omega11, omega12; 1: omega21, omega22) of row i applied to x, without the diagonal:
// accumulated sum (read and cleared) + correction.  NaN when a contribution was marked (`bad`).
__device__ __forceinline__ double finish_row(const FinishRows& f, unsigned long long* __restrict__ acc,
                                             int64_t pos, int64_t i, int c, const double* __restrict__ x, bool bad) {
    const int64_t M = f.M, E = f.E;
    const int e0 = f.ptr[i], e1 = f.ptr[i + 1];
    const double* wa = f.w + (c == 0 ? 0 : E);
    const double* wb = f.w + (c == 0 ? 3 : 2) * E;
    const double hb = c == 0 ? f.h3 : f.h2;
    const double s = fx_read_one(acc + pos, M, c, true);
    double v = 0.0;
    for (int e = e0; e < e1; e += 4) {   // four entries (a row has about four) with their gathers in flight
        int m[4];
        double a[4], b[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int q = min(e + k, e1 - 1);
            m[k] = f.node[q];
            a[k] = wa[q];
            b[k] = wb[q];
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const double t = f.W[m[k]] * (f.h2 * a[k] * x[m[k]] - hb * b[k] * x[M + m[k]]);
            if (e + k < e1) v += t;
        }
    }
    return bad ? __longlong_as_double(0x7ff8000000000000ll) : s + v;
}

// The rows of a finishing kernel: a block of kFinishThreads takes kFinishRows rows, the two components of a
// row in different warps (half the serial chain of one thread per row, and twice the threads for the small
// systems, where the chain's latency is the whole kernel: 15 -> 9 us at 3 214 nodes, 74 -> 40 us at 178 575).
// put(i, c, value) receives the results.
constexpr int kFinishThreads = 256, kFinishRows = kFinishThreads / 2;
template <typename Put>
__device__ __forceinline__ void finish_rows(const FinishRows& f, unsigned long long* __restrict__ acc,
                                            const int32_t* __restrict__ tinv, const double* __restrict__ x,
                                            const Put& put) {
    const int c = threadIdx.x / kFinishRows, at = threadIdx.x % kFinishRows;
    for (int64_t base = (int64_t)blockIdx.x * kFinishRows; base < f.M; base += (int64_t)gridDim.x * kFinishRows) {
        const int64_t i = base + at;
        bool bad = false;
        unsigned long long* mark = nullptr;
        if (i < f.M) {
            const int64_t pos = tinv ? (int64_t)tinv[i] : i;
            mark = acc + (int64_t)(4 * kFxChunks) * f.M + pos;
            bad = *mark != 0ull;
            put(i, c, finish_row(f, acc, pos, i, c, x, bad));
        }
        __syncthreads();   // both components have read the mark
        if (bad && c == 0) *mark = 0ull;
    }
}


// ------------------------------------------------------------------ pair policies
// Fp32: 4 pi K terms, d = x - y, s = 1/r^3, E = e^{-kappa r}, E1 = E (1 + kappa r):
//   4pi K11 = (d.n_y) s (1 - (eps_E/eps_I) E1)
//   4pi K12 = (1 - E)/r
//   4pi K22 = -(d.n_x) s (1 - (eps_I/eps_E) E1)
//   4pi K21 = s [ (1 - E1) n_x.n_y - (3 - E (3 + 3 kappa r + kappa^2 r^2)) (d.n_x)(d.n_y)/r^2 ]
// and acc1 += a K11 - b K12, acc2 += a K21 - b K22.
struct Fp32Policy {
    using Src = float4;
    static constexpr int kMinBlocks = 2;   // resident blocks per SM the registers are limited for
    static constexpr int kVec = 2;    // Src per node
    static constexpr int kTile = 256; // nodes per tile (8 KB)
    static constexpr int kTab = 0;
    static constexpr bool kRenorm = false;   // running sums need no renormalisation
    static constexpr bool kStepTranspose = false;
    static constexpr int kSymStep = 32;   // symmetric chunk fully unrolled
    struct Tgt {
        float px, py, pz, qx, qy, qz, wa, wb;
    };
    struct Acc {
        float a1, a2;
    };
    using JAcc = Acc;
    using JAccR = Acc;                  // source-side sums while a source meets the thread's targets
    static constexpr int kPack = 1;     // targets per thread slot
    __device__ static JAcc jfinal(const JAccR& a) { return a; }   // source-side (transposed) sums of a symmetric tile
    __device__ static Tgt load(const Src* src, int t) {
        const float4 a = src[2 * t], b = src[2 * t + 1];
        return Tgt{a.x, a.y, a.z, b.x, b.y, b.z, a.w, b.w};
    }
    __device__ static void clear_w(Tgt& t) { t.wa = t.wb = 0.f; }
    __device__ static void zero(Acc& c) { c.a1 = c.a2 = 0.f; }
    __device__ static void fold(const Acc& c, double& s1, double& s2) {
        s1 += (double)c.a1;
        s2 += (double)c.a2;
    }
    __device__ static JAcc jadd(const JAcc& x, const JAcc& y) { return JAcc{x.a1 + y.a1, x.a2 + y.a2}; }
    __device__ static JAcc jshfl_xor(const JAcc& x, int m) {
        return JAcc{__shfl_xor_sync(0xffffffffu, x.a1, m), __shfl_xor_sync(0xffffffffu, x.a2, m)};
    }
    template <bool kMask>
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2*, Acc& acc, const bool* exv) {
        const bool ex = exv[0];
        float4 pa = S[0], nb = S[1];
        if (kMask && ex) {   // excluded correction pair: a zero-weight source at distance 1
            pa = make_float4(T.px + 1.f, T.py, T.pz, 0.f);
            nb.w = 0.f;
        }
        const float dx = T.px - pa.x, dy = T.py - pa.y, dz = T.pz - pa.z;
        const float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
        const float rinv = rsqrt_sfu(r2);
        const float r = r2 * rinv;
        const float E = ex2_sfu(k.kl2f * r);
        const float kr = k.kappaf * r;
        const float E1 = fmaf(E, kr, E);
        const float dny = fmaf(dz, nb.z, fmaf(dy, nb.y, dx * nb.x));
        const float dnx = fmaf(dz, T.qz, fmaf(dy, T.qy, dx * T.qx));
        const float nn = fmaf(T.qz, nb.z, fmaf(T.qy, nb.y, T.qx * nb.x));
        const float rinv2 = rinv * rinv;
        const float s = rinv2 * rinv;
        const float as = pa.w * s, bs = nb.w * s;
        const float t1 = fmaf(-k.c1f, E1, 1.f);
        acc.a1 = fmaf(as, dny * t1, acc.a1);
        const float om = fmaf(-rinv, E, rinv);
        acc.a1 = fmaf(-nb.w, om, acc.a1);
        const float t2 = fmaf(-k.c2f, E1, 1.f);
        acc.a2 = fmaf(bs, dnx * t2, acc.a2);
        const float u = 1.f - E1;
        const float q = fmaf(kr, kr + 3.f, 3.f);
        const float t3 = fmaf(-E, q, 3.f);
        const float B = t3 * dnx * dny * rinv2;
        acc.a2 = fmaf(as, fmaf(u, nn, -B), acc.a2);
    }
};

// Packed FP32: the Fp32 terms for two targets at once (lanes of f32x2 operations).  A thread slot
// holds targets a, b (lanes x, y); a source node is stored with every value duplicated,
// {(x,x),(y,y)} {(z,z),(a,a)} {(nx,nx),(ny,ny)} {(nz,nz),(-b,-b)} (64 B), so a broadcast
// shared-memory load gives ready operands.  The signs sit in the stored weights:
//   s t1 = s - c1 s E1, s t2n = c2 s E1 - s, om = (1 - E)/r, u = 1 - E1,
//   t3n = E q - 3, Bn = t3n (d.n_x)(d.n_y)/r^2, X = u n_x.n_y + Bn,
//   target rows: a1 += a (d.n_y) s t1 + (-b) om,   a2 += (-b)(d.n_x) s t2n + a s X;
//   source rows: a1 += (-a_t)(d.n_x) s t1 + (-b_t) om,
//                -a2 += (-b_t)(d.n_y) s t2n + (-a_t) s X   (negated; jfinal restores the sign).
struct Fp32x2Policy {
    using Src = ulonglong2;
    static constexpr int kMinBlocks = 2;   // resident blocks per SM the registers are limited for
    static constexpr int kVec = 4;      // Src per node (64 B)
    static constexpr int kTile = 256;   // nodes per tile (16 KB)
    static constexpr int kTab = 0;
    static constexpr bool kRenorm = false;   // running sums need no renormalisation
    static constexpr bool kStepTranspose = false;
    static constexpr int kSymStep = 32;
    static constexpr int kNearStep = 4;   // sources per transposed step of a near symmetric item
    static constexpr int kPack = 2;
    struct Tgt {
        u64 px, py, pz, qx, qy, qz, nwa, nwb;
    };
    struct Acc {
        u64 a1, a2;
    };
    struct JAcc {
        float a1, a2;
    };
    using JAccR = Acc;
    __device__ static JAcc jfinal(const JAccR& j) {
        float x0, x1, y0, y1;
        up2(j.a1, x0, x1);
        up2(j.a2, y0, y1);
        return JAcc{x0 + x1, -(y0 + y1)};
    }
    __device__ static Tgt load_pack(const Src* src, int M, const int* ti) {
        float v[2][8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = min(ti[h], M - 1);
            const ulonglong2 a = src[4 * t], b = src[4 * t + 1], c = src[4 * t + 2], d = src[4 * t + 3];
            float dummy;
            up2(a.x, v[h][0], dummy);
            up2(a.y, v[h][1], dummy);
            up2(b.x, v[h][2], dummy);
            up2(b.y, v[h][6], dummy);   // a
            up2(c.x, v[h][3], dummy);
            up2(c.y, v[h][4], dummy);
            up2(d.x, v[h][5], dummy);
            up2(d.y, v[h][7], dummy);   // -b
            v[h][6] = -v[h][6];                        // -a
            if (ti[h] >= M) v[h][6] = v[h][7] = 0.f;   // a padding target adds nothing to the sources
        }
        return Tgt{pk2(v[0][0], v[1][0]), pk2(v[0][1], v[1][1]), pk2(v[0][2], v[1][2]), pk2(v[0][3], v[1][3]),
                   pk2(v[0][4], v[1][4]), pk2(v[0][5], v[1][5]), pk2(v[0][6], v[1][6]), pk2(v[0][7], v[1][7])};
    }
    __device__ static void zero(Acc& c) { c.a1 = c.a2 = 0ull; }
    __device__ static void zero(JAcc& c) { c.a1 = c.a2 = 0.f; }
    __device__ static void fold_pack(const Acc& c, double* s1, double* s2) {
        float x0, x1, y0, y1;
        up2(c.a1, x0, x1);
        up2(c.a2, y0, y1);
        s1[0] += (double)x0;
        s1[1] += (double)x1;
        s2[0] += (double)y0;
        s2[1] += (double)y1;
    }
    __device__ static void fold(const JAcc& c, double& s1, double& s2) {
        s1 += (double)c.a1;
        s2 += (double)c.a2;
    }
    __device__ static JAcc jadd(const JAcc& x, const JAcc& y) { return JAcc{x.a1 + y.a1, x.a2 + y.a2}; }
    __device__ static JAcc jshfl_xor(const JAcc& x, int m) {
        return JAcc{__shfl_xor_sync(0xffffffffu, x.a1, m), __shfl_xor_sync(0xffffffffu, x.a2, m)};
    }
    struct Node {
        u64 x, y, z, nx, ny, nz, a, nb;
    };
    __device__ static Node node(const Src* S) {
        const ulonglong2 v0 = S[0], v1 = S[1], v2 = S[2], v3 = S[3];
        return Node{v0.x, v0.y, v1.x, v2.x, v2.y, v3.x, v1.y, v3.y};
    }
    // The halves of `other` where excluded, else of `mine`.
    __device__ static u64 pick(const bool* ex, u64 mine, u64 other) {
        float m0, m1, o0, o1;
        up2(mine, m0, m1);
        up2(other, o0, o1);
        return pk2(ex[0] ? o0 : m0, ex[1] ? o1 : m1);
    }
    // Excluded pairs (per half): a zero-weight source at distance 1 of the target.
    __device__ static void exclude(const Tgt& T, Node& q, const bool* ex, u64 one2) {
        q.x = pick(ex, q.x, add2(T.px, one2));
        q.y = pick(ex, q.y, T.py);
        q.z = pick(ex, q.z, T.pz);
        q.a = pick(ex, q.a, 0ull);
        q.nb = pick(ex, q.nb, 0ull);
    }
    // The terms shared by both orientations for the two targets of T and source q.
    struct Common {
        u64 dnx, dny, om, st1, st2n, sX;
    };
    __device__ static Common common(const Tgt& T, const Node& q, const PairConsts& k) {
        const u64 dx = sub2(T.px, q.x), dy = sub2(T.py, q.y), dz = sub2(T.pz, q.z);
        const u64 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        const u64 rinv = rsqrt2(r2);
        const u64 r = mul2(r2, rinv);
        const u64 E = ex2_2(mul2(k.kl2x2, r));
        const u64 kr = mul2(k.kap2, r);
        const u64 E1 = fma2(E, kr, E);
        Common c;
        c.dny = fma2(dz, q.nz, fma2(dy, q.ny, mul2(dx, q.nx)));
        c.dnx = fma2(dz, T.qz, fma2(dy, T.qy, mul2(dx, T.qx)));
        const u64 nn = fma2(T.qz, q.nz, fma2(T.qy, q.ny, mul2(T.qx, q.nx)));
        const u64 rinv2 = mul2(rinv, rinv);
        const u64 s = mul2(rinv2, rinv);
        const u64 v = mul2(s, E1);
        c.st1 = fma2(k.nc1x2, v, s);
        c.st2n = fma2(k.c2x2, v, neg2(s));
        c.om = fma2(neg2(rinv), E, rinv);
        const u64 u = sub2(k.one2, E1);
        const u64 p = fma2(kr, add2(kr, k.three2), k.three2);
        const u64 t3n = fma2(E, p, k.mthree2);
        const u64 Bn = mul2(mul2(mul2(t3n, c.dnx), c.dny), rinv2);
        c.sX = mul2(s, fma2(u, nn, Bn));
        return c;
    }
    __device__ static void target_terms(const Common& c, u64 Sa, u64 Snb, Acc& acc) {
        acc.a1 = fma2(mul2(Sa, c.dny), c.st1, acc.a1);
        acc.a1 = fma2(Snb, c.om, acc.a1);
        acc.a2 = fma2(mul2(Snb, c.dnx), c.st2n, acc.a2);
        acc.a2 = fma2(Sa, c.sX, acc.a2);
    }
    template <bool kMask>
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2*, Acc& acc,
                                const bool* ex) {
        Node q = node(S);
        if (kMask && (ex[0] || ex[1])) exclude(T, q, ex, k.one2);
        target_terms(common(T, q, k), q.a, q.nb, acc);
    }
    // Both orientations: the factors s t1, s t2n, s X and (1 - E)/r are formed once (40 operations per one-sided
    // evaluation, 47 per symmetric one; of the 47, 19 are multiply-adds with three distinct register operands,
    // which run at 84 lanes a clock and SM against 127 for the others (probe/probe.cu; scalar ones at 85): the mix
    // allows 82% of the pipe, the kernel keeps it busy for 78% of its active cycles).
    // kMask: flags per half (Exclusions); a pair left out of both rows is moved to distance 1 (no NaN).
    template <bool kFirst, bool kMask = false>
    __device__ static void pair_sym(const Tgt& T, const Src* S, const PairConsts& k, const float2*, Acc& acc,
                                    JAccR& ja, const int* ex = nullptr) {
        Node q = node(S);
        u64 nwa = T.nwa, nwb = T.nwb;
        if constexpr (kMask) {
            if (ex[0] | ex[1]) {
                const bool both[2] = {ex[0] == 3, ex[1] == 3};
                const bool out_t[2] = {(ex[0] & kOutTarget) != 0, (ex[1] & kOutTarget) != 0};
                const bool out_s[2] = {(ex[0] & kOutSource) != 0, (ex[1] & kOutSource) != 0};
                q.x = pick(both, q.x, add2(T.px, k.one2));
                q.y = pick(both, q.y, T.py);
                q.z = pick(both, q.z, T.pz);
                q.a = pick(out_t, q.a, 0ull);
                q.nb = pick(out_t, q.nb, 0ull);
                nwa = pick(out_s, nwa, 0ull);
                nwb = pick(out_s, nwb, 0ull);
            }
        }
        const Common c = common(T, q, k);
        target_terms(c, q.a, q.nb, acc);
        if constexpr (kFirst) {
            ja.a1 = mul2(mul2(nwa, c.dnx), c.st1);
            ja.a2 = mul2(mul2(nwb, c.dny), c.st2n);   // ja.a2 holds -a2 until jfinal
        } else {
            ja.a1 = fma2(mul2(nwa, c.dnx), c.st1, ja.a1);
            ja.a2 = fma2(mul2(nwb, c.dny), c.st2n, ja.a2);
        }
        ja.a1 = fma2(nwb, c.om, ja.a1);
        ja.a2 = fma2(nwa, c.sX, ja.a2);
    }
};

struct Fp64Policy {
    using Src = double4;
    static constexpr int kMinBlocks = 2;   // resident blocks per SM the registers are limited for
    static constexpr int kVec = 2;
    static constexpr int kTile = 128;   // 8 KB
    static constexpr int kTab = kExp2F2;
    static constexpr bool kRenorm = false;   // running sums need no renormalisation
    static constexpr bool kStepTranspose = false;
    static constexpr int kSymStep = 4;
    static constexpr int kNearStep = 2;
    struct Tgt {
        double px, py, pz, qx, qy, qz, wa, wb;
    };
    struct Acc {
        double a1, a2;
    };
    using JAcc = Acc;
    using JAccR = Acc;                  // source-side sums while a source meets the thread's targets
    static constexpr int kPack = 1;     // targets per thread slot
    __device__ static JAcc jfinal(const JAccR& a) { return a; }
    __device__ static Tgt load(const Src* src, int t) {
        const double4 a = src[2 * t], b = src[2 * t + 1];
        return Tgt{a.x, a.y, a.z, b.x, b.y, b.z, a.w, b.w};
    }
    __device__ static void clear_w(Tgt& t) { t.wa = t.wb = 0.0; }
    __device__ static void zero(Acc& c) { c.a1 = c.a2 = 0.0; }
    __device__ static void fold(const Acc& c, double& s1, double& s2) {
        s1 += c.a1;
        s2 += c.a2;
    }
    __device__ static JAcc jadd(const JAcc& x, const JAcc& y) { return JAcc{x.a1 + y.a1, x.a2 + y.a2}; }
    __device__ static JAcc jshfl_xor(const JAcc& x, int m) {
        return JAcc{__shfl_xor_sync(0xffffffffu, x.a1, m), __shfl_xor_sync(0xffffffffu, x.a2, m)};
    }
    // The factors the two orientations share: d . n_x, d . n_y, s t1, s t2, s X and (1 - E)/r (u, w, c as in
    // Df64Policy): 55 FP64 operations per symmetric evaluation, 50 per one-sided one (before rsqrt_d, exp_neg_d and
    // the shared factors the profiler counted 69 per symmetric one).  Per application 9.7 -> 7.8 ms at 11 203 nodes, 133 -> 107 ms at 44 597, 90% of
    // the FP64 pipe's measured rate; every term's error as before.
    struct Common {
        double dnx, dny, st1, st2, sX, om;
    };
    __device__ static Common common(const Tgt& T, const double4& pa, const double4& nb, const PairConsts& k,
                                    const float2* tab) {
        const double dx = T.px - pa.x, dy = T.py - pa.y, dz = T.pz - pa.z;
        const double r2 = fma(dz, dz, fma(dy, dy, dx * dx));
        const double rinv = rsqrt_d(r2);
        const double r = r2 * rinv;
        const double E = exp_neg_d(r, k, tab);
        const double kr = k.kappa * r;
        const double E1 = fma(E, kr, E);
        Common c;
        c.dny = fma(dz, nb.z, fma(dy, nb.y, dx * nb.x));
        c.dnx = fma(dz, T.qz, fma(dy, T.qy, dx * T.qx));
        const double nn = fma(T.qz, nb.z, fma(T.qy, nb.y, T.qx * nb.x));
        const double rinv2 = rinv * rinv;
        const double s = rinv2 * rinv;
        const double v = s * E1;
        const double cc = c.dnx * c.dny * rinv2;
        const double X = fma(E * kr * kr, cc, (1.0 - E1) * fma(-3.0, cc, nn));
        c.om = fma(-rinv, E, rinv);
        c.st1 = fma(-k.c1, v, s);
        c.st2 = fma(-k.c2, v, s);
        c.sX = s * X;
        return c;
    }
    __device__ static void target_terms(const Common& c, double a, double b, Acc& acc) {
        acc.a1 = fma(a, c.dny * c.st1, acc.a1);
        acc.a1 = fma(-b, c.om, acc.a1);
        acc.a2 = fma(b, c.dnx * c.st2, acc.a2);
        acc.a2 = fma(a, c.sX, acc.a2);
    }
    // kMask: flags (Exclusions); a pair left out of both rows is moved to distance 1 (no NaN).
    template <bool kFirst, bool kMask = false>
    __device__ static void pair_sym(const Tgt& T, const Src* S, const PairConsts& k, const float2* tab, Acc& acc,
                                    JAcc& ja, const int* ex = nullptr) {
        double4 pa = S[0], nb = S[1];
        double wa = T.wa, wb = T.wb;
        if constexpr (kMask) {
            if (*ex == 3) exclude(T, pa, nb);
            if (*ex & kOutTarget) pa.w = nb.w = 0.0;
            if (*ex & kOutSource) wa = wb = 0.0;
        }
        const Common c = common(T, pa, nb, k, tab);
        target_terms(c, pa.w, nb.w, acc);
        const double x1 = c.dnx * c.st1, y2 = c.dny * c.st2;
        if constexpr (kFirst) {
            ja.a1 = -wa * x1;
            ja.a2 = -wb * y2;
        } else {
            ja.a1 = fma(-wa, x1, ja.a1);
            ja.a2 = fma(-wb, y2, ja.a2);
        }
        ja.a1 = fma(-wb, c.om, ja.a1);
        ja.a2 = fma(wa, c.sX, ja.a2);
    }
    __device__ static void exclude(const Tgt& T, double4& pa, double4& nb) {
        pa = make_double4(T.px + 1.0, T.py, T.pz, 0.0);
        nb.w = 0.0;
    }
    template <bool kMask>
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2* tab, Acc& acc,
                                const bool* exv) {
        double4 pa = S[0], nb = S[1];
        if (kMask && exv[0]) exclude(T, pa, nb);
        target_terms(common(T, pa, nb, k, tab), pa.w, nb.w, acc);
    }
};

// Source node = 4 float4: {P.hi, a.hi} {P.lo, a.lo} {n.hi, b.hi} {n.lo, b.lo}.
// Bound: the FP32 pipe (no FP64 in the pair loops).  Products and sums are lazy; renormalised are only the
// node differences, 1/r, E and 1 - E1 (and the running sums once per step), which is what keeps every term's error at or below that of fully
// normalised arithmetic (a pair's K11, K12, K21 against 64 bits, 2e5 pairs of an ellipsoid 0.3 to 8 apart:
// rms 6.3e-14, 5.1e-14, 2.0e-12 of the uncancelled term; normalised throughout: 7.1e-14, 5.5e-14, 2.1e-12).
// With u = 1 - E1, w = E kappa r, c = (d . n_x)(d . n_y)/r^2 the bracket of K21 is
// u (n_x . n_y - 3 c) + w kappa r c, which needs neither 3 + 3 kappa r + kappa^2 r^2 nor 3 - E (..).
// About 423 FP32 operations per symmetric evaluation (500 before): 217 ms instead of 255 ms per application
// at 178 575 nodes, 13.9 instead of 16.5 ms at 44 597.  Shape: 24 warps per SM (80 registers) and fully
// unrolled steps of 4 sources, transposed step by step; longer unrolled code misses the instruction cache
// (steps of 8: 265 ms), steps of 2 measured 221 ms, 16 warps 213 against 209 ms (before the running sums were
// renormalised), two targets per f32x2 operation 227 ms: the FMA pipe, not issue, is the limit, and a packed
// multiplication is contracted with the packed addition that follows it, which breaks error-free sums.
struct Df64Policy {
    using Src = float4;
    static constexpr int kVec = 4;
    static constexpr int kTile = 128;   // 8 KB
    static constexpr int kMinBlocks = 3;
    static constexpr int kTab = kExpHi + kExpLo;   // exponential tables in shared memory (float2)
    static constexpr bool kRenorm = true;
    static constexpr bool kStepTranspose = true;   // each step's sources are transposed on their own
    static constexpr int kSymStep = 4;
    static constexpr int kNearStep = 2;
    struct Tgt {
        F2 px, py, pz, qx, qy, qz, wa, wb;
    };
    struct Acc {
        F2 a1, a2;
    };
    using JAcc = Acc;
    using JAccR = Acc;                  // source-side sums while a source meets the thread's targets
    static constexpr int kPack = 1;     // targets per thread slot
    __device__ static JAcc jfinal(const JAccR& a) { return a; }
    __device__ static Tgt load(const Src* src, int t) {
        const float4 a = src[4 * t], b = src[4 * t + 1], c = src[4 * t + 2], d = src[4 * t + 3];
        return Tgt{F2{a.x, b.x}, F2{a.y, b.y}, F2{a.z, b.z}, F2{c.x, d.x}, F2{c.y, d.y}, F2{c.z, d.z},
                   F2{a.w, b.w}, F2{c.w, d.w}};
    }
    __device__ static void clear_w(Tgt& t) { t.wa = t.wb = F2{0.f, 0.f}; }
    __device__ static void zero(Acc& c) { c.a1 = c.a2 = F2{0.f, 0.f}; }
    __device__ static void fold(const Acc& c, double& s1, double& s2) {
        s1 += (double)c.a1.hi + (double)c.a1.lo;
        s2 += (double)c.a2.hi + (double)c.a2.lo;
    }
    // the low parts of a running sum grow with every lazy addition: renormalised once per step
    __device__ static void renorm(Acc& c) {
        c.a1 = fast_two_sum(c.a1.hi, c.a1.lo);
        c.a2 = fast_two_sum(c.a2.hi, c.a2.lo);
    }
    // unnormalised sums (exact two_sum of the high parts); the caller folds the result to FP64
    __device__ static JAcc jadd(const JAcc& x, const JAcc& y) {
        JAcc r = x;
        acc_add(r.a1, y.a1);
        acc_add(r.a2, y.a2);
        return r;
    }
    __device__ static JAcc jshfl_xor(const JAcc& x, int m) {
        return JAcc{F2{__shfl_xor_sync(0xffffffffu, x.a1.hi, m), __shfl_xor_sync(0xffffffffu, x.a1.lo, m)},
                    F2{__shfl_xor_sync(0xffffffffu, x.a2.hi, m), __shfl_xor_sync(0xffffffffu, x.a2.lo, m)}};
    }
    struct Node {
        F2 x, y, z, nx, ny, nz, a, b;
    };
    __device__ static Node node(const Src* S) {
        const float4 p = S[0], pl = S[1], n = S[2], nl = S[3];
        return Node{F2{p.x, pl.x}, F2{p.y, pl.y}, F2{p.z, pl.z}, F2{n.x, nl.x},
                    F2{n.y, nl.y}, F2{n.z, nl.z}, F2{p.w, pl.w}, F2{n.w, nl.w}};
    }
    // The factors the two orientations share: d . n_x, d . n_y, s t1, s t2, s X and (1 - E)/r.
    struct Common {
        F2 dnx, dny, st1, st2, sX, om;
    };
    __device__ static Common common(const Tgt& T, const Node& q, const PairConsts& k, const float2* tab) {
        const F2 dx = sub(T.px, q.x), dy = sub(T.py, q.y), dz = sub(T.pz, q.z);
        const F2 r2 = sq3l(dx, dy, dz);
        const F2 rinv = rsqrt_ff(r2);
        const F2 kr = mull(f2(k.kappad), mull(r2, rinv));
        F2 E = exp_neg_ffl(kr, tab);
        E = fast_two_sum(E.hi, E.lo);
        const F2 w = mull(E, kr);
        const F2 E1 = addl(E, w);
        Common c;
        c.om = mull(rinv, one_minus(E));
        c.dny = dot3l(dx, dy, dz, q.nx, q.ny, q.nz);
        c.dnx = dot3l(dx, dy, dz, T.qx, T.qy, T.qz);
        const F2 nn = dot3l(T.qx, T.qy, T.qz, q.nx, q.ny, q.nz);
        const F2 rinv2 = mull(rinv, rinv);
        const F2 s = mull(rinv2, rinv);
        const F2 cc = mull(mull(c.dnx, c.dny), rinv2);
        const F2 c3 = two_prod(3.0f, cc.hi);
        const F2 m = subl(nn, F2{c3.hi, __fmaf_rn(3.0f, cc.lo, c3.lo)});
        F2 u = one_minus(E1);
        u = fast_two_sum(u.hi, u.lo);
        const F2 X = addl(mull(u, m), mull(mull(w, kr), cc));
        c.st1 = mull(s, one_minus_any(mull(E1, f2(k.c1d))));
        c.st2 = mull(s, one_minus_any(mull(E1, f2(k.c2d))));
        c.sX = mull(s, X);
        return c;
    }
    __device__ static void target_terms(const Common& c, F2 A, F2 B, Acc& acc) {
        acc_mul(acc.a1, A, mull(c.dny, c.st1));
        acc_mul(acc.a1, neg(B), c.om);
        acc_mul(acc.a2, B, mull(c.dnx, c.st2));
        acc_mul(acc.a2, A, c.sX);
    }
    template <bool kMask>
    __device__ static void pair(const Tgt& T, const Src* S, const PairConsts& k, const float2* tab, Acc& acc,
                                const bool* exv) {
        Node q = node(S);
        if (kMask && exv[0]) exclude(T, q);
        target_terms(common(T, q, k, tab), q.a, q.b, acc);
    }
    __device__ static void exclude(const Tgt& T, Node& q) {   // a zero-weight source at distance 1
        q.x = F2{T.px.hi + 1.f, T.px.lo};
        q.y = T.py;
        q.z = T.pz;
        q.a = q.b = F2{0.f, 0.f};
    }
    // kMask: flags (Exclusions); a pair left out of both rows is moved to distance 1 (no NaN).
    template <bool kFirst, bool kMask = false>
    __device__ static void pair_sym(const Tgt& T, const Src* S, const PairConsts& k, const float2* tab, Acc& acc,
                                    JAcc& ja, const int* ex = nullptr) {
        Node q = node(S);
        F2 wa = T.wa, wb = T.wb;
        if constexpr (kMask) {
            if (*ex == 3) exclude(T, q);
            if (*ex & kOutTarget) q.a = q.b = F2{0.f, 0.f};
            if (*ex & kOutSource) wa = wb = F2{0.f, 0.f};
        }
        const Common c = common(T, q, k, tab);
        target_terms(c, q.a, q.b, acc);
        const F2 x1 = mull(c.dnx, c.st1), y2 = mull(c.dny, c.st2);
        if constexpr (kFirst) {
            ja.a1 = neg(mull(wa, x1));
            ja.a2 = neg(mull(wb, y2));
        } else {
            acc_mul(ja.a1, neg(wa), x1);
            acc_mul(ja.a2, neg(wb), y2);
        }
        acc_mul(ja.a1, neg(wb), c.om);
        acc_mul(ja.a2, wa, c.sX);
    }
};

// Generic target handling for policies with kPack targets per thread slot: slot r of a thread holds
// targets tblock * BS + (r * kPack + h) * kThreads + tid, h < kPack.
template <typename Policy>
__device__ __forceinline__ typename Policy::Tgt load_targets(const typename Policy::Src* src, int M, const int* ti) {
    if constexpr (Policy::kPack == 1) {
        typename Policy::Tgt t = Policy::load(src, min(ti[0], M - 1));
        if (ti[0] >= M) Policy::clear_w(t);   // a padding target adds nothing to the sources
        return t;
    } else {
        return Policy::load_pack(src, M, ti);
    }
}
template <typename Policy>
__device__ __forceinline__ void fold_targets(const typename Policy::Acc& a, double* s1, double* s2) {
    if constexpr (Policy::kPack == 1) Policy::fold(a, s1[0], s2[0]);
    else Policy::fold_pack(a, s1, s2);
}

// Where a work item's sums go.  RegionOut: the sums of node i to out[c * cstride + (i - t0)], c = 0, 1
// (one region per item, added later in a fixed order); FxOut: added into the node's exact accumulators.
struct RegionOut {
    double* out;
    int64_t cstride, t0;
    __device__ __forceinline__ void put(int64_t i, double s1, double s2) const {
        out[i - t0] = s1;
        out[cstride + i - t0] = s2;
    }
};
struct FxOut {
    unsigned long long* acc;
    int64_t stride;
    __device__ __forceinline__ void put(int64_t i, double s1, double s2) const {
        fx_add(acc + i, stride, 0, s1);
        fx_add(acc + i, stride, 1, s2);
    }
};

// What the items leave out, by target position i, ascending.
//   own: the correction nodes N(i), own_list[own_begin[i] .. own_begin[i + 1]): the one-sided items' masks.
//   closed: every node j with j in N(i) or i in N(j), as 4 j + flags (kOutTarget: j is left out of row i,
//   kOutSource: i is left out of row j), list[begin[i] .. end[i]): the near symmetric items' masks.
// (Positions: node ids, or tree positions in a treecode handle.)
struct Exclusions {
    const int32_t* own_begin;
    const int32_t* own_list;
    const int32_t* begin;
    const int32_t* end;
    const int32_t* list;
};

// The first two entries of the ascending list[b .. e) that are >= j (INT_MAX where there is none) and the
// first one's position; eight entries (few lists are longer) are read at a time, their latencies overlapping.
__device__ __forceinline__ void first_excluded(const int32_t* __restrict__ list, int b, int e, int j, int& pos,
                                               int& next, int& after) {
    pos = b;
    next = after = INT_MAX;
    while (pos < e) {
        int v[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) v[k] = pos + k < e ? list[pos + k] : INT_MAX;
        int below = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) below += v[k] < j;
#pragma unroll
        for (int k = 7; k >= 0; --k) {
            if (v[k] >= j) {
                after = v[k + 1];
                next = v[k];
            }
        }
        pos += below;
        if (below < 8) break;
    }
}

// One one-sided work item of the dense pair sum: target block `tblock`
// (kThreads * R targets) against sources [j_begin, j_end), with the correction
// pairs masked; the sums of target i go to `out` (RegionOut or FxOut).
// Shared memory (ring, tables, barriers) is set up by the caller; `gt` counts
// the tiles this block has consumed so far (it fixes the mbarrier phase parity
// across items).  Returns false when a bounded wait expired (the error word is
// set; the caller must return).
template <typename Policy, int R, int U = 2, typename Out = FxOut>
__device__ __forceinline__ bool pair_item(const typename Policy::Src* __restrict__ src, int M,
                                          const Exclusions& cl, int tblock, int j_begin, int j_end, const Out& out,
                                          const PairConsts& kc,
                                          int* __restrict__ err, typename Policy::Src* ring, const float2* tab,
                                          uint64_t* bar, uint32_t& gt) {
    using Src = typename Policy::Src;
    constexpr int TILE = Policy::kTile;
    constexpr int VEC = Policy::kVec;
    constexpr int P = Policy::kPack;
    constexpr int RP = R * P;
    const int tid = threadIdx.x;
    const int ntiles = (j_end > j_begin) ? (j_end - j_begin + TILE - 1) / TILE : 0;

    typename Policy::Tgt tg[R];
    double s1[RP], s2[RP];
    int ti[RP], epos[RP], eend[RP], enext[RP], eafter[RP];   // the entry after the next one is read ahead
#pragma unroll
    for (int a = 0; a < RP; ++a) {
        ti[a] = tblock * (kThreads * RP) + a * kThreads + tid;
        const int t = min(ti[a], M - 1);
        s1[a] = 0.0;
        s2[a] = 0.0;
        eend[a] = cl.own_begin[t + 1];
        first_excluded(cl.own_list, cl.own_begin[t], eend[a], j_begin, epos[a], enext[a], eafter[a]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) tg[r] = load_targets<Policy>(src, M, &ti[r * P]);
    auto issue = [&](int k) {
        const uint32_t g = gt + (uint32_t)k;
        const int j0 = j_begin + k * TILE;
        const int n = min(TILE, j_end - j0);
        const uint32_t bytes = (uint32_t)(n * VEC * sizeof(Src));
        Src* dst = ring + (g & 1) * TILE * VEC;
        fence_proxy_async();
        mbar_expect_tx(&bar[g & 1], bytes);
        bulk_load(dst, src + (size_t)VEC * j0, bytes, &bar[g & 1]);
    };
    if (tid == 0 && ntiles > 0) issue(0);

    for (int k = 0; k < ntiles; ++k) {
        const uint32_t g = gt + (uint32_t)k;
        if (tid == 0 && k + 1 < ntiles) issue(k + 1);
        const bool ok = mbar_wait(&bar[g & 1], (g >> 1) & 1, kc.wait_limit);
        if (__syncthreads_or(!ok)) {
            // give up: flag it, let the copies that may still be in flight (this tile's and the
            // next one's) land in this block's shared memory, return
            if (tid == 0) {
                atomicOr(err, kErrWait);
                (void)mbar_wait(&bar[g & 1], (g >> 1) & 1);
                if (k + 1 < ntiles) (void)mbar_wait(&bar[(g + 1) & 1], ((g + 1) >> 1) & 1);
            }
            return false;
        }
        const Src* tile = ring + (g & 1) * TILE * VEC;
        const int j0 = j_begin + k * TILE;
        const int n = min(TILE, j_end - j0);
        bool need = false;
#pragma unroll
        for (int a = 0; a < RP; ++a) need |= (enext[a] < j0 + n);
        typename Policy::Acc acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) Policy::zero(acc[r]);
        if (!__any_sync(0xffffffffu, need)) {
            const bool none[P] = {};
#pragma unroll U
            for (int q = 0; q < n; ++q) {
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    Policy::template pair<false>(tg[r], tile + q * VEC, kc, tab, acc[r], none);
                    if constexpr (Policy::kRenorm) Policy::renorm(acc[r]);
                }
            }
        } else {
            for (int q = 0; q < n; ++q) {
                const int j = j0 + q;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    bool ex[P];
#pragma unroll
                    for (int h = 0; h < P; ++h) {
                        const int a = r * P + h;
                        ex[h] = (j == enext[a]);
                        if (ex[h]) {
                            ++epos[a];
                            enext[a] = eafter[a];
                            eafter[a] = (epos[a] + 1 < eend[a]) ? cl.own_list[epos[a] + 1] : INT_MAX;
                        }
                    }
                    Policy::template pair<true>(tg[r], tile + q * VEC, kc, tab, acc[r], ex);
                    if constexpr (Policy::kRenorm) Policy::renorm(acc[r]);
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) fold_targets<Policy>(acc[r], &s1[r * P], &s2[r * P]);
        __syncthreads();   // the buffer of this tile is free for the tile after next
    }
    gt += (uint32_t)ntiles;
#pragma unroll
    for (int a = 0; a < RP; ++a)
        if (ti[a] < M) out.put(ti[a], s1[a], s2[a]);
    return true;
}

// In-warp transpose-and-sum of V per-lane values v[0..V) (V a power of two <= 32):
// afterwards every lane holds, in v[0], the sum over all 32 lanes of entry
// lane >> (5 - log2 V).  Each exchange stage halves the entries a lane keeps
// (it sends the half its partner keeps); the remaining stages are a plain
// butterfly.  The summation tree is the hypercube order 16, 8, 4, 2, 1 for any V.
template <typename Policy, int V>
__device__ __forceinline__ void transpose_sum(typename Policy::JAcc (&v)[V], int lane) {
    using J = typename Policy::JAcc;
    int cnt = V;
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1) {
        if (cnt > 1) {
            const bool upper = (lane & m) != 0;
            const int h = cnt / 2;
#pragma unroll
            for (int i = 0; i < V / 2; ++i) {
                if (i < h) {
                    const J send = upper ? v[i] : v[i + h];
                    const J keep = upper ? v[i + h] : v[i];
                    v[i] = Policy::jadd(keep, Policy::jshfl_xor(send, m));
                }
            }
            cnt = h;
        } else {
            v[0] = Policy::jadd(v[0], Policy::jshfl_xor(v[0], m));
        }
    }
}

// One symmetric work item: target block `tblock` against sources
// [j_begin, j_end), no correction pair among them (the schedule guarantees it).
// Every pair is evaluated once for both orientations (Policy::pair_sym).  The
// target sums (at the item's end) and the source sums (per tile) are added
// into the nodes' exact accumulators (`out`).  Sources are read by
// broadcast as in the one-sided item; a thread accumulates the source-side
// terms of a chunk of V sources over its R targets, the warp transposes and
// sums them (transpose_sum), and the kWarps warp sums of a tile are added in
// warp order in shared memory (jred: kWarps * TILE entries).  The chunk loop
// is unrolled S sources at a time (S = V: fully); with S < V the chunk's
// accumulators shift by S registers per step (or, Policy::kStepTranspose, each
// step's sums are transposed on their own), which keeps the code of long pair
// arithmetics within the instruction cache.
template <typename Policy, int R, int V, int U, int S = V>
__device__ __forceinline__ bool pair_item_sym(const typename Policy::Src* __restrict__ src, int M, int tblock,
                                              int j_begin, int j_end, const FxOut& out, const PairConsts& kc,
                                              int* __restrict__ err, typename Policy::Src* ring,
                                              typename Policy::JAcc* jred, const float2* tab, uint64_t* bar,
                                              uint32_t& gt) {
    using Src = typename Policy::Src;
    using J = typename Policy::JAcc;
    constexpr int TILE = Policy::kTile;
    constexpr int VEC = Policy::kVec;
    constexpr int P = Policy::kPack;
    constexpr int RP = R * P;
    constexpr int BS = kThreads * RP;
    constexpr int kWarps = kThreads / 32;
    constexpr int kShift = (V == 32) ? 0 : (V == 16) ? 1 : (V == 8) ? 2 : (V == 4) ? 3 : (V == 2) ? 4 : 5;
    static_assert(TILE % V == 0 && TILE <= kThreads, "tile layout");
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int len = j_end - j_begin;
    const int ntiles = (len + TILE - 1) / TILE;

    typename Policy::Tgt tg[R];
    double s1[RP], s2[RP];
    int ti[RP];
#pragma unroll
    for (int a = 0; a < RP; ++a) {
        ti[a] = tblock * BS + a * kThreads + tid;
        s1[a] = 0.0;
        s2[a] = 0.0;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) tg[r] = load_targets<Policy>(src, M, &ti[r * P]);
    auto issue = [&](int k) {
        const uint32_t g = gt + (uint32_t)k;
        const int j0 = j_begin + k * TILE;
        const int n = min(TILE, j_end - j0);
        const uint32_t bytes = (uint32_t)(n * VEC * sizeof(Src));
        Src* dst = ring + (g & 1) * TILE * VEC;
        fence_proxy_async();
        mbar_expect_tx(&bar[g & 1], bytes);
        bulk_load(dst, src + (size_t)VEC * j0, bytes, &bar[g & 1]);
    };
    if (tid == 0 && ntiles > 0) issue(0);

    for (int k = 0; k < ntiles; ++k) {
        const uint32_t g = gt + (uint32_t)k;
        if (tid == 0 && k + 1 < ntiles) issue(k + 1);
        const bool ok = mbar_wait(&bar[g & 1], (g >> 1) & 1, kc.wait_limit);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {   // as in pair_item: flag, drain both copies in flight, return
                atomicOr(err, kErrWait);
                (void)mbar_wait(&bar[g & 1], (g >> 1) & 1);
                if (k + 1 < ntiles) (void)mbar_wait(&bar[(g + 1) & 1], ((g + 1) >> 1) & 1);
            }
            return false;
        }
        const Src* tile = ring + (g & 1) * TILE * VEC;
        const int j0 = j_begin + k * TILE;
        const int n = min(TILE, j_end - j0);
        typename Policy::Acc acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) Policy::zero(acc[r]);
#pragma unroll U
        for (int c0 = 0; c0 < n; c0 += V) {
            if constexpr (Policy::kStepTranspose) {
                // S sources per step, transposed and summed at once: registers for S sums only
#pragma unroll 1
                for (int q0 = 0; q0 < V && c0 + q0 < n; q0 += S) {
                    J cur[S];
                    auto source = [&](int t) {
                        typename Policy::JAccR jr;
                        const Src* q = tile + (c0 + q0 + t) * VEC;
                        Policy::template pair_sym<true>(tg[0], q, kc, tab, acc[0], jr);
#pragma unroll
                        for (int r = 1; r < R; ++r)
                            Policy::template pair_sym<false>(tg[r], q, kc, tab, acc[r], jr);
                        cur[t] = Policy::jfinal(jr);
                    };
                    if (c0 + q0 + S <= n) {
#pragma unroll
                        for (int t = 0; t < S; ++t) source(t);
                    } else {   // ragged end of the item: warp-uniform skip
#pragma unroll
                        for (int t = 0; t < S; ++t) {
                            Policy::zero(cur[t]);
                            if (c0 + q0 + t < n) source(t);
                        }
                    }
#pragma unroll
                    for (int r = 0; r < R; ++r) Policy::renorm(acc[r]);
                    transpose_sum<Policy, S>(cur, lane);
                    const int qs = c0 + q0 + lane / (32 / S);
                    if (lane % (32 / S) == 0 && qs < n) jred[warp * TILE + qs] = cur[0];
                }
                continue;
            }
            J ja[V];
#pragma unroll
            for (int q = 0; q < V; ++q) Policy::zero(ja[q]);
            if constexpr (S == V) {
                if (c0 + V <= n) {
#pragma unroll
                    for (int q = 0; q < V; ++q) {
                        typename Policy::JAccR jr;
                        Policy::template pair_sym<true>(tg[0], tile + (c0 + q) * VEC, kc, tab, acc[0], jr);
#pragma unroll
                        for (int r = 1; r < R; ++r)
                            Policy::template pair_sym<false>(tg[r], tile + (c0 + q) * VEC, kc, tab, acc[r], jr);
                        ja[q] = Policy::jfinal(jr);
                    }
                } else {   // ragged end of the item: warp-uniform skip
#pragma unroll
                    for (int q = 0; q < V; ++q) {
                        if (c0 + q < n) {
                            typename Policy::JAccR jr;
                            Policy::template pair_sym<true>(tg[0], tile + (c0 + q) * VEC, kc, tab, acc[0], jr);
#pragma unroll
                            for (int r = 1; r < R; ++r)
                                Policy::template pair_sym<false>(tg[r], tile + (c0 + q) * VEC, kc, tab, acc[r], jr);
                            ja[q] = Policy::jfinal(jr);
                        }
                    }
                }
            } else {
                // S sources per step; afterwards ja[k] holds source V - S (k / S + 1) + k % S of the chunk
#pragma unroll 1
                for (int q0 = 0; q0 < V; q0 += S) {
                    J cur[S];
#pragma unroll
                    for (int t = 0; t < S; ++t) {
                        Policy::zero(cur[t]);
                        const int q = c0 + q0 + t;
                        if (q < n) {   // warp-uniform
                            typename Policy::JAccR jr;
                            Policy::template pair_sym<true>(tg[0], tile + q * VEC, kc, tab, acc[0], jr);
#pragma unroll
                            for (int r = 1; r < R; ++r)
                                Policy::template pair_sym<false>(tg[r], tile + q * VEC, kc, tab, acc[r], jr);
                            cur[t] = Policy::jfinal(jr);
                        }
                    }
#pragma unroll
                    for (int k = V - 1; k >= S; --k) ja[k] = ja[k - S];
#pragma unroll
                    for (int t = 0; t < S; ++t) ja[t] = cur[t];
                }
            }
            transpose_sum<Policy, V>(ja, lane);
            const int e = lane >> kShift;
            const int qs = V - S * (e / S + 1) + e % S;
            if ((lane & ((1 << kShift) - 1)) == 0 && c0 + qs < n) jred[warp * TILE + c0 + qs] = ja[0];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) fold_targets<Policy>(acc[r], &s1[r * P], &s2[r * P]);
        __syncthreads();   // all warp sums of this tile are in jred
        if (tid < n) {
            J t = jred[tid];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) t = Policy::jadd(t, jred[w * TILE + tid]);
            double d1 = 0.0, d2 = 0.0;
            Policy::fold(t, d1, d2);
            out.put(j0 + tid, d1, d2);
        }
        __syncthreads();   // jred and the buffer of this tile are free again
    }
    gt += (uint32_t)ntiles;
#pragma unroll
    for (int a = 0; a < RP; ++a)
        if (ti[a] < M) out.put(ti[a], s1[a], s2[a]);
    return true;
}

// One symmetric work item with correction pairs among its pairs: as pair_item_sym, but an excluded pair adds
// nothing to the row(s) that leave it out.  A target is compared with its next excluded node at every source;
// kNearStep sources are transposed at a time, which keeps the code short (a few per cent of the pairs of a
// large system come here, most of a small one's).
template <typename Policy, int R>
__device__ __forceinline__ bool pair_item_near(const typename Policy::Src* __restrict__ src, int M, const Exclusions& cl,
                                               int tblock, int j_begin, int j_end, const FxOut& out,
                                               const PairConsts& kc, int* __restrict__ err, typename Policy::Src* ring,
                                               typename Policy::JAcc* jred, const float2* tab, uint64_t* bar,
                                               uint32_t& gt) {
    using Src = typename Policy::Src;
    using J = typename Policy::JAcc;
    constexpr int TILE = Policy::kTile;
    constexpr int VEC = Policy::kVec;
    constexpr int P = Policy::kPack;
    constexpr int RP = R * P;
    constexpr int BS = kThreads * RP;
    constexpr int kWarps = kThreads / 32;
    constexpr int S = Policy::kNearStep;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ntiles = (j_end - j_begin + TILE - 1) / TILE;

    typename Policy::Tgt tg[R];
    double s1[RP], s2[RP];
    int ti[RP], epos[RP], eend[RP], enext[RP], eafter[RP];
#pragma unroll
    for (int a = 0; a < RP; ++a) {
        ti[a] = tblock * BS + a * kThreads + tid;
        s1[a] = 0.0;
        s2[a] = 0.0;
        const int t = min(ti[a], M - 1);
        eend[a] = cl.end[t];
        first_excluded(cl.list, cl.begin[t], eend[a], 4 * j_begin, epos[a], enext[a], eafter[a]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) tg[r] = load_targets<Policy>(src, M, &ti[r * P]);
    auto issue = [&](int k) {
        const uint32_t g = gt + (uint32_t)k;
        const int j0 = j_begin + k * TILE;
        const int n = min(TILE, j_end - j0);
        const uint32_t bytes = (uint32_t)(n * VEC * sizeof(Src));
        Src* dst = ring + (g & 1) * TILE * VEC;
        fence_proxy_async();
        mbar_expect_tx(&bar[g & 1], bytes);
        bulk_load(dst, src + (size_t)VEC * j0, bytes, &bar[g & 1]);
    };
    if (tid == 0 && ntiles > 0) issue(0);

    for (int k = 0; k < ntiles; ++k) {
        const uint32_t g = gt + (uint32_t)k;
        if (tid == 0 && k + 1 < ntiles) issue(k + 1);
        const bool ok = mbar_wait(&bar[g & 1], (g >> 1) & 1, kc.wait_limit);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {   // as in pair_item: flag, drain both copies in flight, return
                atomicOr(err, kErrWait);
                (void)mbar_wait(&bar[g & 1], (g >> 1) & 1);
                if (k + 1 < ntiles) (void)mbar_wait(&bar[(g + 1) & 1], ((g + 1) >> 1) & 1);
            }
            return false;
        }
        const Src* tile = ring + (g & 1) * TILE * VEC;
        const int j0 = j_begin + k * TILE;
        const int n = min(TILE, j_end - j0);
        typename Policy::Acc acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) Policy::zero(acc[r]);
#pragma unroll 1
        for (int c0 = 0; c0 < n; c0 += S) {
            J cur[S];
#pragma unroll
            for (int t = 0; t < S; ++t) {
                Policy::zero(cur[t]);
                const int q = c0 + t;
                if (q < n) {   // warp-uniform
                    typename Policy::JAccR jr;
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        int ex[P];
#pragma unroll
                        for (int h = 0; h < P; ++h) {
                            const int a = r * P + h;
                            ex[h] = 0;
                            if (j0 + q == enext[a] >> 2) {
                                ex[h] = enext[a] & 3;
                                ++epos[a];
                                enext[a] = eafter[a];
                                eafter[a] = (epos[a] + 1 < eend[a]) ? cl.list[epos[a] + 1] : INT_MAX;
                            }
                        }
                        if (r == 0) Policy::template pair_sym<true, true>(tg[r], tile + q * VEC, kc, tab, acc[r], jr, ex);
                        else Policy::template pair_sym<false, true>(tg[r], tile + q * VEC, kc, tab, acc[r], jr, ex);
                    }
                    cur[t] = Policy::jfinal(jr);
                }
            }
            if constexpr (Policy::kRenorm) {
#pragma unroll
                for (int r = 0; r < R; ++r) Policy::renorm(acc[r]);
            }
            transpose_sum<Policy, S>(cur, lane);
            const int qs = c0 + lane / (32 / S);
            if (lane % (32 / S) == 0 && qs < n) jred[warp * TILE + qs] = cur[0];
        }
#pragma unroll
        for (int r = 0; r < R; ++r) fold_targets<Policy>(acc[r], &s1[r * P], &s2[r * P]);
        __syncthreads();   // all warp sums of this tile are in jred
        if (tid < n) {
            J t = jred[tid];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) t = Policy::jadd(t, jred[w * TILE + tid]);
            double d1 = 0.0, d2 = 0.0;
            Policy::fold(t, d1, d2);
            out.put(j0 + tid, d1, d2);
        }
        __syncthreads();   // jred and the buffer of this tile are free again
    }
    gt += (uint32_t)ntiles;
#pragma unroll
    for (int a = 0; a < RP; ++a)
        if (ti[a] < M) out.put(ti[a], s1[a], s2[a]);
    return true;
}

// Runs one item of a schedule (dispatch on its kind); its sums go into the nodes' exact accumulators
// (acc, M words per accumulator word, fx_add).
template <typename Policy, int R, int V, int U>
__device__ __forceinline__ bool run_item(const PairItem& it, const typename Policy::Src* __restrict__ src, int M,
                                         const Exclusions& cl, unsigned long long* __restrict__ acc,
                                         const PairConsts& kc, int* __restrict__ err, typename Policy::Src* ring,
                                         typename Policy::JAcc* jred, const float2* tab, uint64_t* bar,
                                         uint32_t& gt) {
    constexpr int S = Policy::kSymStep < V ? Policy::kSymStep : V;
    const FxOut out{acc, (int64_t)M};
    if (it.sym == kItemNear)
        return pair_item_near<Policy, R>(src, M, cl, it.I, it.j_begin, it.j_end, out, kc, err, ring, jred, tab, bar, gt);
    if (it.sym == kItemSym)
        return pair_item_sym<Policy, R, V, U, S>(src, M, it.I, it.j_begin, it.j_end, out, kc, err, ring, jred, tab,
                                                 bar, gt);
    return pair_item<Policy, R, U>(src, M, cl, it.I, it.j_begin, it.j_end, out, kc, err, ring, tab, bar, gt);
}

// Shared-memory bytes of a pair block: the two-stage source ring, the warp
// sums of a symmetric tile and, for the float-float and FP64 policies, the exponential
// tables (in that order; each part a multiple of 16 bytes).
template <typename Policy>
constexpr size_t pair_ring_bytes() {
    return 2 * Policy::kTile * Policy::kVec * sizeof(typename Policy::Src);
}
template <typename Policy>
constexpr size_t pair_jred_bytes() {
    return (size_t)(kThreads / 32) * Policy::kTile * sizeof(typename Policy::JAcc);
}
template <typename Policy>
constexpr size_t pair_smem_bytes() {
    return pair_ring_bytes<Policy>() + pair_jred_bytes<Policy>() +
           Policy::kTab * sizeof(float2);
}
// The dynamic shared memory of a pair block, carved in the order above.
template <typename Policy>
struct PairSmem {
    typename Policy::Src* ring;
    typename Policy::JAcc* jred;
    float2* tab;
    __device__ explicit PairSmem(unsigned char* raw)
        : ring(reinterpret_cast<typename Policy::Src*>(raw)),
          jred(reinterpret_cast<typename Policy::JAcc*>(raw + pair_ring_bytes<Policy>())),
          tab(reinterpret_cast<float2*>(raw + pair_ring_bytes<Policy>() + pair_jred_bytes<Policy>())) {}
};

// Launch shapes of the schedules: thread slots (x the policy's kPack targets) and sources per
// transposed chunk.  R and the tile fix the target blocks and the per-tile sums, hence the summation
// order: they are a property of a system's schedule (set when the system is set up), the same
// wherever the system runs.  The float-float and FP64 shapes are fixed; kR32 is the default FP32 one.
constexpr int kR32 = 2, kRdf = 1, kR64 = 1;   // thread slots (FP32: 2 packed pairs = 4 targets)
constexpr int kChunkDf = 8, kChunk64 = 8;

// The packed FP32 policy with another source tile (sources per shared-memory stage).
template <int TILE>
struct Fp32x2T : Fp32x2Policy {
    static constexpr int kTile = TILE;
};

// FP32 schedule-kernel variants, one of which each system's FP32 schedule uses: thread slots R (R x 2
// targets per thread: 512 or 1024 per block), source tile, sources per transposed chunk V and unroll
// U of the chunk loop.  Variant 0 is the default shape (the treecode's near items always use it).
struct Var32 {
    int R, tile, V, U;
};
constexpr int kNumVar32 = 6;
constexpr Var32 kVar32[kNumVar32] = {{2, 256, 8, 1}, {2, 256, 8, 2}, {1, 256, 8, 2},
                                     {2, 128, 8, 2}, {1, 128, 8, 2}, {2, 256, 4, 2}};

// f.template run<Policy, R, V, U>() for FP32 variant v (a functor with a member template `run`)
template <typename F>
inline int with_var32(int v, const F& f) {
    switch (v) {
        case 1: return f.template run<Fp32x2T<256>, 2, 8, 2>();
        case 2: return f.template run<Fp32x2T<256>, 1, 8, 2>();
        case 3: return f.template run<Fp32x2T<128>, 2, 8, 2>();
        case 4: return f.template run<Fp32x2T<128>, 1, 8, 2>();
        case 5: return f.template run<Fp32x2T<256>, 2, 4, 2>();
        default: return f.template run<Fp32x2T<256>, 2, 8, 1>();
    }
}

// Per-block setup shared by every pair kernel: exponential tables and the two mbarriers.
template <typename Policy>
__device__ __forceinline__ void pair_block_init(const float2* exp_tab, float2* tab, uint64_t* bar) {
    for (int q = threadIdx.x; q < Policy::kTab; q += kThreads) tab[q] = exp_tab[q];
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        fence_mbar_init();
    }
    __syncthreads();
}

inline float2 split_ff(double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
}
__device__ __forceinline__ float2 split_ff_dev(double v) {
    const float hi = __double2float_rn(v);
    return make_float2(hi, __double2float_rn(v - (double)hi));
}

}  // namespace pk

// Exponential tables of pair arithmetic pol on a device: 1 the float-float e^{-k} (k < 64) and e^{-k/1024}
// (k < 1024), 2 the FP64 2^{-k/1024} and their relative rounding errors (k < 1024), 0 none (NULL)
int exp_table(int device, int pol, const float2** out);
// What a handle's pair items leave out
pk::Exclusions exclusions_of(const ctr_ibim* s);
// The finishing kernels' view of a handle's rows
pk::FinishRows finish_rows_of(const ctr_ibim* s);
// Splits of the source range for equal-work items filling whole waves of `slots` resident blocks
// (one-sided grid launch of the fixed-scratch entry point)
PairPlan make_plan(int64_t M, int R, int tile, int slots);
// Resident blocks of the schedule kernels of the three arithmetics: [0] FP32 (default variant),
// [1] float-float, [2] FP64
int schedule_slots(int sms, int slots[3]);
// The FP32 variant of the most recent tuning in this process (-1 before any)
int last_fp32_variant();
// Runs a handle's schedule of one arithmetic (policy index 0 FP32, 1 float-float, 2 FP64) on its stream
int launch_schedule(ctr_ibim* s, int pol, const void* src, const pk::PairConsts& kc);
// Fill the f32x2 copies of a PairConsts from its FP32 fields
void set_packed_consts(pk::PairConsts& kc);
// Pair constants of a handle (kernel-ratio terms, kappa) and the tables of pair arithmetic pol
int pair_consts(ctr_ibim* s, int pol, pk::PairConsts* out);
// Polls of the pair kernels' bounded waits for launches prepared from now on (ctr_set_wait_limit)
uint32_t wait_limit();

}  // namespace ctr
