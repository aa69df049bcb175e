// Double-float ("F2") exp, log, log1p, square root and reciprocal for the
// rate transcendentals, on the FP32 pipe.
//
// On GB300 a warp issues one FP64 instruction per ~64 cycles whatever the
// dependences between them (one FP64 FMA chain and two independent chains
// per warp both run at 64 cycles per FMA), while a dependent FP32 FMA takes
// ~4.6 cycles; float <-> double conversions also run on the FP64 pipe.  A
// thermochemistry attempt is therefore bounded by its count of FP64
// instructions, and the transcendentals of the rate fits were about half
// of them.  Here every value is an unevaluated sum hi + lo of two floats
// (48 significant bits, the double-float arithmetic of Dekker, Numer. Math.
// 18 (1971) 224, with the error-free sum of Knuth and the FMA product);
// doubles enter and leave through integer bit operations, and each result
// costs one FP64 addition (hi + lo, exact).  exp and log follow P. T. P.
// Tang's table-driven reductions (ACM TOMS 15 (1989) 144 and 16 (1990)
// 378) with 64 and 128 table points; the tables and split constants come
// from gen_dfmath_tables.py.
//
// Accuracy (relative to the exact function of the double input, checked
// against CUDA's FP64 exp, log and log1p by tests/test_gpu_fmath.py):
//   exp(x)    (3 |x| + 16) 2^-48 (the 48-bit argument dominates for |x| > 8)
//   log(x)    2^-46 max(1, |ln x|) absolute
//   log1p(w)  2^-45
//   1/a, sqrt(a) of a pair: 2^-44
// i.e. 1e-14 to 1e-12 relative for the rate coefficients, far inside the
// 1e-10 parity the FP64 path is held to.  Inputs outside the ranges the
// rate fits produce (a double beyond 2^-60 .. 2^60 in magnitude) go to
// CUDA's FP64 functions (log1p of w < 2^-60 is w itself).
#pragma once

#include <cuda_runtime.h>

#include "dfmath_tables.h"

namespace rtgb {
namespace dfm {

struct F2 {
    float hi, lo;   // value hi + lo, |lo| <= ulp(hi) / 2
};

// ---- error-free transformations (rounded intrinsics: never contracted) ----
__device__ __forceinline__ F2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}

__device__ __forceinline__ F2 fast_two_sum(float a, float b)   // |a| >= |b| or a == 0
{
    const float s = __fadd_rn(a, b);
    return {s, __fsub_rn(b, __fsub_rn(s, a))};
}

__device__ __forceinline__ F2 two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}

// ---- double-float arithmetic ----
__device__ __forceinline__ F2 add(F2 a, F2 b)
{
    F2 s = two_sum(a.hi, b.hi);
    const F2 t = two_sum(a.lo, b.lo);
    s = fast_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
    return fast_two_sum(s.hi, __fadd_rn(s.lo, t.lo));
}

// Products and sums without the final normalisation: the low part stays
// within a few ulps of the high one, which the next operation takes as well
// (errors of 2^-46 of the operands' magnitude, what the arguments and terms
// they are used on carry anyway).  4, 8 and 5 instructions, mul() has 7 and
// add() 20; a pair is normalised (norm) where it is stored or converted.
// addu is commutative, adding a zero pair or multiplying by one returns the
// operand unchanged.
__device__ __forceinline__ F2 norm(F2 a) { return fast_two_sum(a.hi, a.lo); }

__device__ __forceinline__ F2 addu(F2 a, F2 b)
{
    const F2 s = two_sum(a.hi, b.hi);
    return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}

// |a.hi| >= |b.hi| or a.hi == 0
__device__ __forceinline__ F2 addf(F2 a, F2 b)
{
    const F2 s = fast_two_sum(a.hi, b.hi);
    return {s.hi, __fadd_rn(s.lo, __fadd_rn(a.lo, b.lo))};
}

__device__ __forceinline__ F2 mulu(F2 a, F2 b)
{
    const F2 p = two_prod(a.hi, b.hi);
    return {p.hi, __fmaf_rn(a.lo, b.hi, __fmaf_rn(a.hi, b.lo, p.lo))};
}

__device__ __forceinline__ F2 add(F2 a, float b)
{
    const F2 s = two_sum(a.hi, b);
    return fast_two_sum(s.hi, __fadd_rn(s.lo, a.lo));
}

__device__ __forceinline__ F2 neg(F2 a) { return {-a.hi, -a.lo}; }

__device__ __forceinline__ F2 mul(F2 a, F2 b)
{
    F2 p = two_prod(a.hi, b.hi);
    p.lo = __fmaf_rn(a.hi, b.lo, p.lo);
    p.lo = __fmaf_rn(a.lo, b.hi, p.lo);
    return fast_two_sum(p.hi, p.lo);
}

__device__ __forceinline__ F2 mul(F2 a, float b)
{
    F2 p = two_prod(a.hi, b);
    p.lo = __fmaf_rn(a.lo, b, p.lo);
    return fast_two_sum(p.hi, p.lo);
}

// 2^n as a float, n in [-126, 127]
__device__ __forceinline__ float pow2f(int n) { return __uint_as_float((unsigned)(n + 127) << 23); }

// ---- doubles in and out through integer operations ----
// |x| in [2^-60, 2^60) (or 0): the double split into a float pair (hi: the
// top 24 bits, lo: the next 29 rounded to 24), relative error <= 2^-48; the
// range keeps the low floats of the results below (reciprocals, square
// roots, logarithms) clear of float subnormals.
__device__ __forceinline__ bool splittable(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffULL;
    return b == 0ULL || (b >= 0x3c30000000000000ULL && b < 0x43b0000000000000ULL);
}

__device__ __forceinline__ F2 split(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sign = (unsigned)(b >> 63) << 31;
    const int e = (int)((b >> 52) & 0x7ff);
    if (e == 0) return {0.0f, 0.0f};
    if (e == 0x7ff) return {__uint_as_float(sign | 0x7f800000u | ((b & 0xfffffffffffffULL) ? 0x400000u : 0u)), 0.0f};
    const float hi = __uint_as_float(sign | ((unsigned)(e - 896) << 23) | (unsigned)((b >> 29) & 0x7fffff));
    const float lo = __uint2float_rn((unsigned)(b & 0x1fffffffULL)) * pow2f(e - 1075);
    return {hi, sign ? -lo : lo};
}

// any double as a pair (outside the range above through FP64 conversions)
__device__ __forceinline__ F2 split_any(double x)
{
    if (splittable(x)) return split(x);
    const float hi = __double2float_rn(x);
    return {hi, __double2float_rn(x - (double)hi)};
}

// the double of a float (exact; subnormal floats, which the pairs here never
// hold in a significant place, count as zero)
__device__ __forceinline__ double widen(float f)
{
    const unsigned u = __float_as_uint(f);
    const unsigned e = (u >> 23) & 0xff;
    if (e == 0) return 0.0;
    const unsigned long long bits = ((unsigned long long)(u >> 31) << 63) |
                                    ((unsigned long long)(e + 896) << 52) |
                                    ((unsigned long long)(u & 0x7fffff) << 29);
    return __longlong_as_double((long long)bits);
}

__device__ __forceinline__ double to_double(F2 a) { return widen(a.hi) + widen(a.lo); }

// (hi + lo) 2^m as a double without the FP64 pipe: lo, at most 1.5 2^-23 of
// hi and rounded to 2^-52 of hi's binade, is added to the bits of hi.  hi a
// positive float of 2^-75 and more, the result a normal double.
__device__ __forceinline__ double combine(float hi, float lo, int m = 0)
{
    const unsigned u = __float_as_uint(hi);
    int L = __float2int_rn(__fmul_rn(lo, __uint_as_float((306u << 23) - (u & 0x7f800000u))));
    if ((u & 0x7fffffu) == 0 && L < 0) L *= 2;   // below hi the binade's steps are half as long
    const unsigned top = (u >> 3) + 0x38000000u + ((unsigned)m << 20);
    return __longlong_as_double((long long)(((unsigned long long)top << 32) | (unsigned long long)(u << 29)) + L);
}

// any pair times 2^m, |m| below 2000 (a zero or tiny high part through the
// FP64 pipe; results below the normal doubles are 0)
__device__ __forceinline__ double to_double_i(F2 a, int m = 0)
{
    const float h = fabsf(a.hi);
    const bool neg = a.hi < 0.0f;
    if (!(h > 0x1p-70f && h < 0x1p120f)) return ldexp((double)a.hi + (double)a.lo, m);
    const int e = (int)(__float_as_uint(h) >> 23) - 127 + m;
    if (e < -1020) return 0.0;
    const long long r = __double_as_longlong(combine(h, neg ? -a.lo : a.lo, m));
    return __longlong_as_double(neg ? r | (1LL << 63) : r);   // (a negation may take the FP64 pipe)
}

// Two ways to deal with arguments outside an operation's range.  Exact: a
// branch to the general form there.  Fast: no branch; `odd` is set and the
// value is of no use, and the caller repeats the whole computation the exact
// way (the team kernel's attempts, a single basic block that the compiler
// can interleave).  In range both give the same bits.
struct Exact {
    static constexpr bool fast = false;
};
struct Fast {
    static constexpr bool fast = true;
    bool odd = false, reject = false;
};

template <class CTL>
__device__ __forceinline__ double to_double_c(F2 a, int m, CTL &ctl)
{
    if constexpr (!CTL::fast) {
        return to_double_i(a, m);
    } else {
        const float h = fabsf(a.hi);
        const bool neg = a.hi < 0.0f, in = h > 0x1p-70f && h < 0x1p120f;
        ctl.odd |= !in && a.hi != 0.0f;   // (a NaN compares unequal)
        const int e = (int)(__float_as_uint(h) >> 23) - 127 + m;
        const long long r = __double_as_longlong(combine(in ? h : 1.0f, neg ? -a.lo : a.lo, m));
        return __longlong_as_double(!in || e < -1020 ? 0LL : neg ? r | (1LL << 63) : r);
    }
}

// ---- reciprocal and quotient of doubles ----
// The IEEE quotient takes some nine FP64 instructions, and a warp issues one
// per 64 cycles.  Here the reciprocal of the divisor comes from float pairs
// (an approximate FP32 reciprocal and one Newton step in pairs, 2^-45), and
// one FP64 residual step corrects the quotient, whose error before rounding
// is then below 2^-88: the nearest double but for one quotient in 2^35.
// 1/b needs two FP64 instructions, a/b three.  |b| outside 2^-70 .. 2^70,
// zero, infinite or NaN takes the IEEE quotient.
__device__ __forceinline__ float rcp_approx(float a)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}

// a double of 2^-74 .. 2^127 in magnitude as the nearest float and the rest
__device__ __forceinline__ F2 split_near(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const unsigned u = __funnelshift_l(lw, hw, 3) - 0xC0000000u;   // exponent rebiased by 896, mantissa cut to 23 bits
    const float hi = __uint_as_float(u + ((lw >> 28) & 1u));
    const float lo = __int2float_rn((int)(lw << 3) >> 3) * __uint_as_float((u & 0x7f800000u) - (52u << 23));
    return {hi, lo};
}

__device__ __forceinline__ bool div_range(double b)
{
    const unsigned h = (unsigned)((unsigned long long)__double_as_longlong(b) >> 32) & 0x7fffffffu;
    return h - (953u << 20) < (140u << 20);
}

__device__ __forceinline__ double rcp_seed(double b)   // div_range(b)
{
    const F2 s = split_near(__longlong_as_double(__double_as_longlong(b) & 0x7fffffffffffffffLL));
    const float r0 = rcp_approx(s.hi);
    const float e = __fmaf_rn(-s.lo, r0, __fmaf_rn(-s.hi, r0, 1.0f));
    return __longlong_as_double(__double_as_longlong(combine(r0, __fmul_rn(r0, e))) |
                                (__double_as_longlong(b) & (1LL << 63)));
}

static __device__ __noinline__ double ieee_div(double a, double b) { return a / b; }

__device__ __forceinline__ double fast_rcp(double b)
{
    if (!div_range(b)) return ieee_div(1.0, b);
    const double r = rcp_seed(b);
    return __fma_rn(__fma_rn(-b, r, 1.0), r, r);
}

__device__ __forceinline__ double fast_div(double a, double b)
{
    if (!div_range(b)) return ieee_div(a, b);
    const double r = rcp_seed(b);
    const double q = __dmul_rn(a, r);
    return __fma_rn(__fma_rn(-q, b, a), r, q);
}

template <class CTL>
__device__ __forceinline__ double rcp_c(double b, CTL &ctl)
{
    if constexpr (!CTL::fast) {
        return fast_rcp(b);
    } else {
        ctl.odd |= !div_range(b);
        const double r = rcp_seed(b);
        return __fma_rn(__fma_rn(-b, r, 1.0), r, r);
    }
}
template <class CTL>
__device__ __forceinline__ double div_c(double a, double b, CTL &ctl)
{
    if constexpr (!CTL::fast) {
        return fast_div(a, b);
    } else {
        ctl.odd |= !div_range(b);
        const double r = rcp_seed(b);
        const double q = __dmul_rn(a, r);
        return __fma_rn(__fma_rn(-q, b, a), r, q);
    }
}

// a double as the nearest float on the integer pipe: 0 below the normal
// floats, NaN above them (and for infinities and NaN)
__device__ __forceinline__ float near_float(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hw = (unsigned)(b >> 32), lw = (unsigned)b;
    const unsigned e = hw & 0x7ff00000u;
    unsigned u = __funnelshift_l(lw, hw, 3) - 0xC0000000u + ((lw >> 28) & 1u);
    if (e < (897u << 20)) u = 0;
    if (e > (1149u << 20)) u = 0x7fc00000u;
    return __uint_as_float(u | (hw & 0x80000000u));
}

// 1 / a and sqrt(a) of a positive pair: one Newton step in pair arithmetic
// from the correctly rounded FP32 value (relative error <= 2^-24, squared by
// the step)
__device__ __forceinline__ F2 rcp(F2 a)
{
    const float r0 = __frcp_rn(a.hi);
    const F2 e = two_prod(a.hi, r0);
    const float err = __fsub_rn(__fsub_rn(1.0f, e.hi), __fmaf_rn(a.lo, r0, e.lo));
    return fast_two_sum(r0, r0 * err);
}

// 1/a refined by a second Newton step (2^-47)
__device__ __forceinline__ F2 rcp2(F2 a)
{
    const F2 r = rcp(a);
    const F2 p = two_prod(a.hi, r.hi);
    const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, p.hi), p.lo),
                              __fmaf_rn(a.hi, r.lo, __fmul_rn(a.lo, r.hi)));
    return fast_two_sum(r.hi, __fmaf_rn(r.hi, e, r.lo));
}

__device__ __forceinline__ F2 sqrt2(F2 a)
{
    const float s0 = __fsqrt_rn(a.hi);
    const F2 p = two_prod(s0, s0);
    const float d = __fadd_rn(__fsub_rn(__fsub_rn(a.hi, p.hi), p.lo), a.lo);
    return fast_two_sum(s0, d * rsqrtf(a.hi) * 0.5f);
}

// ---- elementary functions ----
// exp2d, log2f2 and log1pd are called out of line: inlined at every call
// site of every thermochemistry kernel they made ptxas run for tens of
// minutes.

// e^x of a pair as y 2^m, y an unnormalised pair in [0.99, 2.02); |x| below 1420
__device__ __forceinline__ void exp_pair(F2 x, F2 &y, int &m)
{
    const float kf = rintf(__fmul_rn(x.hi, kDfInvL));
    const int k = (int)kf;
    // r = x - k ln2/64: k L1 exact, x.hi - k L1 exact (Sterbenz), k L2 split
    // exactly; x.lo, the low part of k L2 and k L3 (all below 2^-24 |x|)
    // summed in FP32
    const F2 p2 = two_prod(kf, kDfL2);
    const F2 s = two_sum(__fmaf_rn(-kf, kDfL1, x.hi), -p2.hi);
    const F2 r = fast_two_sum(s.hi, __fadd_rn(s.lo, __fsub_rn(x.lo, __fmaf_rn(kf, kDfL3, p2.lo))));
    // e^r - 1 = r + [r^2/2 + r^3 (1/6 + r/24 + r^2/120)], |r| <= ln2/128; the
    // bracket (< 1.6e-5) as a pair from r.hi^2 exactly plus FP32 terms
    const float rh = r.hi;
    const F2 h2 = two_prod(rh, rh);
    const float c = __fmaf_rn(rh, r.lo,
                              rh * h2.hi * __fmaf_rn(rh, __fmaf_rn(rh, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f));
    const F2 q = fast_two_sum(0.5f * h2.hi, __fmaf_rn(0.5f, h2.lo, c));
    const F2 p = addf(r, q);
    const float2 t = __ldg(&kDfExp2Tab[k & 63]);
    const F2 T{t.x, t.y};
    y = addf(T, mulu(T, p));   // 2^(j/64) e^r
    m = k >> 6;               // floor(k / 64)
}

// e^x of a pair; a double result (subnormal, 0 and infinity as CUDA's exp)
__device__ __forceinline__ double exp2d_inl(F2 x)
{
    if (!(x.hi > -745.2f)) return (x.hi != x.hi) ? (double)x.hi : 0.0;
    if (x.hi > 709.78f) return __longlong_as_double(0x7ff0000000000000LL);
    F2 y;
    int m;
    exp_pair(x, y, m);
    y = norm(y);
    if (m > -1020 && m < 1020) return combine(y.hi, y.lo, m);
    return ldexp(to_double(y), m);
}

static __device__ __noinline__ double exp2d(F2 x) { return exp2d_inl(x); }

// ln(v / 2^shift) of a positive normal pair
__device__ __forceinline__ F2 log2f2_inl(F2 v, int shift)
{
    const unsigned bits = __float_as_uint(v.hi);
    const int e = (int)(bits >> 23) - 127;
    const int j = (int)(((bits & 0x7fffff) + (1u << 15)) >> 16);   // F = 1 + j/128 nearest the mantissa
    const float Fs = __uint_as_float((unsigned)(e + 127) << 23) * (1.0f + (float)j * (1.0f / 128.0f));
    // f = v - F 2^e: exact (Sterbenz), then scaled exactly to v / 2^e - F
    const F2 fs = two_sum(__fsub_rn(v.hi, Fs), v.lo);
    const float sc = pow2f(-e);
    const F2 f{fs.hi * sc, fs.lo * sc};
    const float4 L = __ldg(&kDfLogTab[j]);
    const F2 u = mul(f, F2{L.z, L.w});   // u = f / F, |u| <= 1/256
    // ln(1 + u) = u - u^2/2 + u^3 (1/3 - u/4 + u^2/5 - u^3/6), the cubic and
    // higher terms (below 2^-25) in FP32
    const float uh = u.hi;
    const F2 u2 = mulu(u, u);
    const float u3 = __fmul_rn(uh, u2.hi);
    const float c = __fmaf_rn(u3, 1.0f / 3.0f, u3 * uh * __fmaf_rn(uh, __fmaf_rn(uh, -1.0f / 6.0f, 0.2f), -0.25f));
    F2 q = fast_two_sum(uh, -0.5f * u2.hi);
    q.lo = __fadd_rn(q.lo, __fadd_rn(__fmaf_rn(-0.5f, u2.lo, u.lo), c));
    // e ln2 + ln F + q; e A exact.  The two small terms first, so that only
    // two roundings are of the size of the sum's low part.
    const float ef = (float)(e - shift);
    const F2 p = two_prod(ef, kDfLn2B);
    const F2 s = fast_two_sum(ef * kDfLn2A, L.x);
    const F2 m = two_sum(p.hi, q.hi);
    const F2 r = two_sum(s.hi, m.hi);
    const float lo = __fadd_rn(m.lo, __fadd_rn(__fadd_rn(__fmaf_rn(ef, kDfLn2C, p.lo), L.y), q.lo));
    return fast_two_sum(r.hi, __fadd_rn(__fadd_rn(s.lo, r.lo), lo));
}

static __device__ __noinline__ F2 log2f2(F2 v, int shift) { return log2f2_inl(v, shift); }

// ln x of a double
__device__ __forceinline__ F2 logd(double x)
{
    if (x > 0.0 && splittable(x)) return log2f2(split(x), 0);
    const double r = log(x);
    return split(r);   // out of range: CUDA's log, split (|ln x| < 746)
}

// ln of a pair above 1 with every sum in full pair precision (relative error
// 2^-46 also where the result is small), for log1pd
__device__ __forceinline__ F2 log2f2_rel(F2 v)
{
    const unsigned bits = __float_as_uint(v.hi);
    const int e = (int)(bits >> 23) - 127;
    const int j = (int)(((bits & 0x7fffff) + (1u << 15)) >> 16);
    const float Fs = __uint_as_float((unsigned)(e + 127) << 23) * (1.0f + (float)j * (1.0f / 128.0f));
    const F2 fs = two_sum(__fsub_rn(v.hi, Fs), v.lo);
    const float sc = pow2f(-e);
    const float4 L = __ldg(&kDfLogTab[j]);
    const F2 u = mul(F2{fs.hi * sc, fs.lo * sc}, F2{L.z, L.w});
    const F2 u2 = mul(u, u);
    const F2 u3 = mul(u2, u.hi);
    const float uh = u.hi;
    F2 q = add(u, F2{-0.5f * u2.hi, -0.5f * u2.lo});
    q = add(q, mul(u3, F2{kDfThirdHi, kDfThirdLo}));
    q = add(q, u3.hi * uh * __fmaf_rn(uh, __fmaf_rn(uh, -1.0f / 6.0f, 0.2f), -0.25f));
    const float ef = (float)e;
    F2 s = two_prod(ef, kDfLn2B);
    s = add(F2{ef * kDfLn2A, 0.0f}, s);
    s = add(s, ef * kDfLn2C);
    s = add(s, F2{L.x, L.y});
    return add(s, q);
}

// ln(1 + w) of a double w >= 0
static __device__ __noinline__ F2 log1pd(double w)
{
    if (!(w >= 0.0) || w >= 1.152921504606847e18) return split(log1p(w));   // NaN, w >= 2^60
    if (!splittable(w)) return {__double2float_rn(w), 0.0f};                     // w < 2^-60: ln(1 + w) = w
    const F2 W = split(w);
    if (W.hi < 0.03125f) {
        // 2 atanh(z), z = w / (2 + w) <= 1/65: 2 (z + z^3/3 + z^5/5 + z^7/7)
        const F2 rd = rcp(add(W, 2.0f));   // 1 / (2 + w)
        const F2 z = mul(W, rd);
        const F2 z2 = mul(z, z);
        const float zh = z2.hi;
        F2 s = mul(z2, F2{kDfThirdHi, kDfThirdLo});
        s = add(s, zh * zh * __fmaf_rn(zh, 1.0f / 7.0f, 0.2f));
        const F2 y = add(z, mul(z, s));
        return {2.0f * y.hi, 2.0f * y.lo};
    }
    // v = 1 + w exactly as a pair plus a remainder c below its last bit
    const F2 s = two_sum(1.0f, W.hi);
    const F2 t = two_sum(s.lo, W.lo);
    const F2 v = fast_two_sum(s.hi, t.hi);
    const F2 lv = log2f2_rel(v);
    return add(lv, __fdividef(t.lo, v.hi));   // + c / v
}

static __device__ __noinline__ F2 softplus_far(F2 z, F2 &sig)
{
    const double w = exp2d(z);
    sig = split_any(w < 1e300 ? w / (1.0 + w) : 1.0);
    return log1pd(w);
}

// ln(1 + e^z) of a pair z, with its derivative 1/(1 + e^-z) as a pair.
// On [-16, 16): the interpolating polynomials of kDfSoftplusTab (degree 7
// in t = z - middle of a 1/32-wide interval, |t| <= 1/64); the terms of
// degree 3 and up (in the derivative beyond 3 c3 t^2) are small enough to be
// summed in FP32, the rest in pairs (absolute error
// ~1e-14 at |z| ~ 16, that of the pair coefficients).  80 instructions; 250
// with 1/4-wide intervals and degree 9.  Outside (temperatures far beyond
// the fits' range) from e^z and log1p.
template <class CTL>
__device__ __forceinline__ F2 softplus2(F2 z, F2 &sig, CTL &ctl)
{
    const bool in = z.hi >= (float)kDfSpLo && z.hi < -(float)kDfSpLo;
    if constexpr (CTL::fast) ctl.odd |= !in;
    if (CTL::fast || in) {
        int k = (int)__fmul_rn(__fadd_rn(z.hi, -(float)kDfSpLo), (float)kDfSpPer);
        k = k < kDfSpN - 1 ? k : kDfSpN - 1;
        if (CTL::fast) k = k < 0 ? 0 : k;
        const float mid = (float)kDfSpLo + ((float)k + 0.5f) / (float)kDfSpPer;   // exact
        const F2 t0 = two_sum(z.hi, -mid);
        const F2 t = fast_two_sum(t0.hi, __fadd_rn(t0.lo, z.lo));
        const float th = t.hi;
        const float4 *c = reinterpret_cast<const float4 *>(kDfSoftplusTab[k]);
        const float4 c01 = __ldg(c), c23 = __ldg(c + 1), c45 = __ldg(c + 2), c67 = __ldg(c + 3);
        const F2 c0{c01.x, c01.y}, c1{c01.z, c01.w};
        const float r = __fmaf_rn(th, __fmaf_rn(th, __fmaf_rn(th, c67.x, c45.z), c45.x), c23.z);   // c3 + .. + c6 t^3
        F2 P = fast_two_sum(c23.x, __fmul_rn(th, r));
        P.lo = __fadd_rn(P.lo, c23.y);
        P = addf(c1, mulu(P, t));
        P = addf(c0, mulu(P, t));
        const float d = __fmaf_rn(th, __fmaf_rn(th, __fmaf_rn(th, 7.0f * c67.z, 6.0f * c67.x), 5.0f * c45.z),
                                  4.0f * c45.x);
        const F2 c3 = two_prod(3.0f, c23.z);
        F2 D = fast_two_sum(c3.hi, __fmul_rn(th, d));
        D.lo = __fadd_rn(D.lo, __fmaf_rn(3.0f, c23.w, c3.lo));
        D = addf(F2{2.0f * c23.x, 2.0f * c23.y}, mulu(D, t));
        sig = norm(addf(c1, mulu(D, t)));
        return norm(P);
    }
    return softplus_far(z, sig);
}
__device__ __forceinline__ F2 softplus2(F2 z, F2 &sig)
{
    Exact e;
    return softplus2(z, sig, e);
}

}  // namespace dfm
}  // namespace rtgb
