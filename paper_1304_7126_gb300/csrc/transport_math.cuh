// Scalar pieces of the transport: reciprocals and square roots with two or three
// FP64 instructions, and the wave speeds of Eq. (hll) in 64-bit fixed point.
#pragma once

#include <cuda_runtime.h>

#include "dfmath.cuh"
#include "rt_internal.h"

namespace rtgb {
namespace {

__device__ __forceinline__ float trcp(float d) { return __fdividef(1.0f, d); }

// ---- FP64 pieces on the integer and FP32 pipes ----
__device__ __forceinline__ long long tbits(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ double tdbl(long long b) { return __longlong_as_double(b); }
__device__ __forceinline__ double tabs_(double x) { return tdbl(tbits(x) & 0x7fffffffffffffffLL); }

// 1/b and 1/sqrt(x) of positive doubles of any normal size: the argument
// scaled to [1, 2) or [1, 4) by its exponent, an FP32 approximation corrected
// in float pairs (2^-45), one FP64 Newton step (two and three instructions,
// within an ulp); zero, subnormal, extreme, infinite and NaN arguments take
// CUDA's functions.
static __device__ __noinline__ double rcp_any(double b) { return 1.0 / b; }
static __device__ __noinline__ double rsqrt_any(double x) { return rsqrt(x); }

__device__ __forceinline__ double trcp(double b)
{
    const int e = (int)(tbits(b) >> 52);   // (sign included: negative arguments are out of range)
    if (e < 8 || e > 2038) return rcp_any(b);
    const long long sh = (long long)(e - 1023) << 52;
    const double t = tdbl(tbits(b) - sh);
    const double r0 = dfm::rcp_seed(t);
    const double r = __fma_rn(__fma_rn(-t, r0, 1.0), r0, r0);
    return tdbl(tbits(r) - sh);
}

__device__ __forceinline__ float rsqrt_approx(float a)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

__device__ __forceinline__ double trsqrt(double x)
{
    const int e = (int)(tbits(x) >> 52);
    if (e < 8 || e > 2038) return rsqrt_any(x);
    const int ee = (e - 1023) & ~1;
    const double t = tdbl(tbits(x) - ((long long)ee << 52));
    const dfm::F2 s = dfm::split_near(t);
    const float y = rsqrt_approx(s.hi);
    const dfm::F2 p = dfm::two_prod(y, y);
    const float d = __fmaf_rn(-s.lo, p.hi, __fmaf_rn(-s.hi, p.lo, __fmaf_rn(-s.hi, p.hi, 1.0f)));   // 1 - t y^2
    const double r0 = dfm::combine(y, __fmul_rn(y, __fmul_rn(d, __fmaf_rn(0.375f, d, 0.5f))));
    const double r = __fma_rn(tdbl(tbits(r0) - (1LL << 52)), __fma_rn(-__dmul_rn(t, r0), r0, 1.0), r0);
    return tdbl(tbits(r) - ((long long)(ee / 2) << 52));
}

// sqrt(t) of t in [1, 4], two FP64 instructions
__device__ __forceinline__ double tsqrt14(double t)
{
    const dfm::F2 s = dfm::split_near(t);
    const float y = rsqrt_approx(s.hi), g = __fmul_rn(s.hi, y), hy = 0.5f * y;
    const float d = __fadd_rn(__fmaf_rn(-g, g, s.hi), s.lo);
    const double s0 = dfm::combine(g, __fmul_rn(d, hy));
    return __fma_rn(__fma_rn(-s0, s0, t), dfm::widen(hy), s0);
}

// |x| <= 1 as fixed point, value 2^62 (at most 2^63 whatever x is), and a
// non-negative fixed-point value as the nearest double
__device__ __forceinline__ unsigned long long to_fix(double x)
{
    const unsigned long long b = (unsigned long long)tbits(x) & 0x7fffffffffffffffULL;
    int sh = 1023 - (int)(b >> 52);
    sh = sh < 0 ? 0 : (sh > 63 ? 63 : sh);
    return (((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10) >> sh;
}
__device__ __forceinline__ double from_fix(unsigned long long v)
{
    if (v == 0) return 0.0;
    const int lz = __clzll((long long)v);
    const unsigned long long m = v << lz;
    return tdbl((long long)(((unsigned long long)(1023 - lz) << 52) + (m >> 11) + ((m >> 10) & 1ULL)));
}
// d w / 2^64, rounded down
__device__ __forceinline__ long long fix_mul(long long d, unsigned long long w)
{
    return (long long)(__umul64hi((unsigned long long)d, w) - (d < 0 ? w : 0ULL));
}

// Wave speeds of a cell along a direction of cosine mu from the bilinear
// table, in fixed point throughout: f and mu are on its grid's scale by their
// leading bits, the weights by the rest (rounding 2^-60).  k, wf: the row of
// f and its weight.  Indices are clamped to the table whatever the state.
__device__ __forceinline__ void hll_lookup_fix(const long long *__restrict__ tab, int k, unsigned long long wf,
                                               double mu, long long &lo, long long &hi)
{
    const unsigned long long a = to_fix(mu);
    unsigned long long v = (1ULL << 62) + (tbits(mu) < 0 ? 0ULL - a : a);   // (mu + 1) 2^62, mod 2^64
    const unsigned long long end = tbits(mu) < 0 ? 0ULL : 0x7fffffffffffffffULL;
    v = (v >> 63) ? end : v;                                       // |mu| >= 1
    const int j = (int)(v >> 55);                                  // 0..255
    const unsigned long long wm = v << 9;
    const longlong2 *t = reinterpret_cast<const longlong2 *>(tab) + k * kHllNMU + j;
    const longlong2 A = __ldg(t), B = __ldg(t + 1), C = __ldg(t + kHllNMU), D = __ldg(t + kHllNMU + 1);
    const long long lo0 = A.x + fix_mul(B.x - A.x, wm), lo1 = C.x + fix_mul(D.x - C.x, wm);
    const long long hi0 = A.y + fix_mul(B.y - A.y, wm), hi1 = C.y + fix_mul(D.y - C.y, wm);
    lo = lo0 + fix_mul(lo1 - lo0, wf);
    hi = hi0 + fix_mul(hi1 - hi0, wf);
}

}  // namespace
}  // namespace rtgb
