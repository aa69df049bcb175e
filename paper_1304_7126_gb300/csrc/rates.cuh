// Device rate-coefficient fits of the paper's appendix on interaction rate
// coefficients (collisional ionisation: Cen 1992; recombination and
// recombination cooling: Hui & Gnedin 1997; collisional excitation: Cen
// 1992; bremsstrahlung; Compton: Haiman et al. 1996; dielectronic: Black
// 1981), each with its analytic temperature derivative, in float pairs (48 bits)
// up to the FP64 update.
//
// Every rate coefficient and every cooling term is one function of T of
// the form
//     f(T) = Cc exp(c0 + c1 ln T + c2 / T - c3 softplus(c4 ln T + c5)),
// softplus(z) = ln(1 + e^z) (see RateFn below).  The lanes of a team of two,
// four or eight that share a cell take a function each; one thread evaluates
// the ones it needs in turn.  The argument, its exponential (dfm::exp_pair) and
// the product with the factor (Cm, with the reference's share of the argument)
// are formed in the double-float arithmetic of dfmath.cuh, on the FP32 pipe;
// both paths run the same expressions and so give identical bits.
//
// What bounds them: the FP64 pipe, of which a warp gets one instruction per
// 64 cycles (so the count of FP64 instructions sets both the length of a lone
// cell's chain of attempts and the throughput of the kernels).
// The functions, their T-derivatives and the cooling sums therefore stay
// float pairs until they enter the FP64 update, and enter it through integer
// operations (dfm::combine) instead of an FP64 addition each.
#pragma once

#include <cuda_runtime.h>

#include "dual.cuh"
#include "dfmath.cuh"

namespace rtgb {

// Quotients and reciprocals of the thermochemistry (dfmath.cuh: three and
// two FP64 instructions).
// dual numbers: the derivative (a' - q b')/b takes the refined reciprocal that
// the quotient's seed gives with one more instruction
template <class CTL>
__device__ __forceinline__ Dual cdiv(const Dual &a, const Dual &b, CTL &ctl)
{
    const bool in = dfm::div_range(b.v);
    if constexpr (CTL::fast) {
        ctl.odd |= !in;
    } else if (!in) {
        const double q = dfm::ieee_div(a.v, b.v);
        return Dual(q, dfm::ieee_div(a.d - q * b.d, b.v));
    }
    const double r = dfm::rcp_seed(b.v), q0 = __dmul_rn(a.v, r);
    const double q = __fma_rn(__fma_rn(-q0, b.v, a.v), r, q0);
    return Dual(q, __fma_rn(-q, b.d, a.d) * __fma_rn(__fma_rn(-b.v, r, 1.0), r, r));
}
template <class CTL>
__device__ __forceinline__ Dual crcp(const Dual &b, CTL &ctl)
{
    const double q = dfm::rcp_c(b.v, ctl);
    return Dual(q, -q * q * b.d);
}
template <class CTL>
__device__ __forceinline__ double cdiv(double a, double b, CTL &ctl) { return dfm::div_c(a, b, ctl); }
template <class CTL>
__device__ __forceinline__ double crcp(double b, CTL &ctl) { return dfm::rcp_c(b, ctl); }

// exp arguments: exp(fma(a, ln T, fma(b, 1/T, c)))
enum {
    E_BETA_HI = 0,   // exp(-157809.1/T): beta_HI, zeta_HI
    E_BETA_HEI,      // exp(-285335.4/T): beta_HeI, zeta_HeI
    E_BETA_HEII,     // exp(-631515/T):   beta_HeII, zeta_HeII
    E_PSI_HI,        // exp(-118348/T)
    E_PSI_HEII,      // T^-0.397 exp(-473638/T)
    E_OMEGA1,        // T^-1.5 exp(-470000/T)
    E_OMEGA2,        // exp(-94000/T)
    E_ALPHA_HEII,    // (570670/T)^p
    E_W0,            // w = exp(z) of the Hui & Gnedin fits HG_* (their z = ln w
                     // are the arguments E_W0.. of the table; w itself is not formed)
    NEXP = E_W0 + 4
};
enum { HG_ALPHA_HII = 0, HG_ALPHA_HEIII, HG_ETA_HII, HG_ETA_HEIII, NHG };

struct ExpArg {
    double a, b, c;
};
struct HGPar {
    double A, lnT1, p, r, s;   // A lam^p / (1 + w)^s, lam = T1/T, w = (lam/l0)^r
};
struct RateTable {           // one per recombination case (A, B)
    ExpArg ea[NEXP];
    HGPar hg[NHG];
    double A_aHeII, p_aHeII;  // alpha_HeII = A (570670/T)^p
};

// Rate tables: exp(a ln T + b/T + c) arguments and the Hui &
// Gnedin parameters, case A then case B; the logarithms are of the fits'
// temperature constants and pivots.
#define RTGB_RATE_TAB_INIT {\
    { /* case A */ \
        {{0.0, -157809.1, 0.0}, {0.0, -285335.4, 0.0}, {0.0, -631515.0, 0.0}, {0.0, -118348.0, 0.0}, {-0.397, -473638.0, 0.0}, {-1.5, -470000.0, 0.0}, {0.0, -94000.0, 0.0}, {-0.654, 0.0, 8.668486417830579}, {-0.47, 0.0, 6.2568105714688285}, {-0.47, 0.0, 6.908582567206}, {-0.502, 0.0, 6.664858835981581}, {-0.502, 0.0, 7.361006797385964}},\
        {{1.269e-13, 12.662275226919286, 1.503, 0.47, 1.923}, {2.538e-13, 14.049024154019651, 1.503, 0.47, 1.923}, {1.778e-29, 12.662275226919286, 1.965, 0.502, 2.697}, {1.4224e-28, 14.049024154019651, 1.965, 0.502, 2.697}},\
        3e-14, 0.654 },\
    { /* case B */ \
        {{0.0, -157809.1, 0.0}, {0.0, -285335.4, 0.0}, {0.0, -631515.0, 0.0}, {0.0, -118348.0, 0.0}, {-0.397, -473638.0, 0.0}, {-1.5, -470000.0, 0.0}, {0.0, -94000.0, 0.0}, {-0.75, 0.0, 9.940924791090113}, {-0.407, 0.0, 4.743307143753357}, {-0.407, 0.0, 5.307713957083206}, {-0.376, 0.0, 4.456105724024312}, {-0.376, 0.0, 4.977523320614049}},\
        {{2.753e-14, 12.662275226919286, 1.5, 0.407, 2.242}, {5.506e-14, 14.049024154019651, 1.5, 0.407, 2.242}, {3.435e-30, 12.662275226919286, 1.97, 0.376, 3.72}, {2.748e-29, 14.049024154019651, 1.97, 0.376, 3.72}},\
        1.26e-14, 0.75 }\
}
// compile-time copy, from which the rate functions below are built
constexpr RateTable kRateTabCx[2] = RTGB_RATE_TAB_INIT;
#undef RTGB_RATE_TAB_INIT

// The table's constants as float pairs (hi = the double rounded to a float,
// lo = the rest rounded), made at compile time.
constexpr dfm::F2 pair_of(double x)
{
    return dfm::F2{(float)x, (float)(x - (double)(float)x)};
}

// a double rounded to the nearest float (ties away from zero) through
// integer operations: a double -> float conversion would take the FP64
// pipe.  Below the normal float range the result is 0, above it infinity
// (NaN included).  Truncating instead biases the FP32 absorption
// coefficients by half an ulp, which over a source cell's thousands of
// sub-steps moved the mixed-precision results by 1e-4.
__device__ __forceinline__ float narrow(double x)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned sign = (unsigned)(b >> 63) << 31;
    const unsigned long long a = (b & 0x7fffffffffffffffULL) + 0x10000000ULL;   // carry may raise the exponent
    const int e = (int)(a >> 52);
    if (e < 897) return __uint_as_float(sign);
    if (e > 1150) return __uint_as_float(sign | 0x7f800000u);
    return __uint_as_float(sign | ((unsigned)(e - 896) << 23) | (unsigned)((a >> 29) & 0x7fffff));
}

enum { SP_HI = 0, SP_HII, SP_HEI, SP_HEII, SP_HEIII, SP_FF, NSP };   // SP_FF: n_HII + n_HeII + 4 n_HeIII

struct CoolTerm {
    double C;
    int sq, uu, tt;   // powers (0 or 1) of sqrt T, u, T
    int e1, e2, hg;   // exponentials e[e1], e[e2] and Hui & Gnedin fit hg (-1: none)
    int amp;          // 1: times the table's amplitude of alpha_HeII
    int sp;           // density factor SP_*
    int he;           // a helium term
};

// (the paper's fits: Cen 1992 collisional ionisation and excitation, Hui &
// Gnedin 1997 recombination cooling, Black 1981 dielectronic recombination,
// bremsstrahlung; k_B T alpha_HeII for HeII recombination cooling)
#define RTGB_COOL_TERMS(X)                                                           \
    X(1.27e-21, 1, 1, 0, E_BETA_HI, -1, -1, 0, SP_HI, 0)                              \
    X(7.5e-19, 0, 1, 0, E_PSI_HI, -1, -1, 0, SP_HI, 0)                                \
    X(1.0, 0, 0, 1, -1, -1, HG_ETA_HII, 0, SP_HII, 0)                                 \
    X(1.42e-27, 1, 0, 0, -1, -1, -1, 0, SP_FF, 0)                                     \
    X(9.38e-22, 1, 1, 0, E_BETA_HEI, -1, -1, 0, SP_HEI, 1)                            \
    X(4.95e-22, 1, 1, 0, E_BETA_HEII, -1, -1, 0, SP_HEII, 1)                          \
    X(5.54e-17, 0, 1, 0, E_PSI_HEII, -1, -1, 0, SP_HEII, 1)                           \
    X(1.380649e-16, 0, 0, 1, E_ALPHA_HEII, -1, -1, 1, SP_HEII, 1)                     \
    X(1.24e-13, 0, 0, 0, E_OMEGA1, -1, -1, 0, SP_HEII, 1)                             \
    X(0.3 * 1.24e-13, 0, 0, 0, E_OMEGA1, E_OMEGA2, -1, 0, SP_HEII, 1)                 \
    X(1.0, 0, 0, 1, -1, -1, HG_ETA_HEIII, 0, SP_HEIII, 1)
#define RTGB_COOL_ROW(C, a, b, c, e1, e2, hg, amp, sp, he) {C, a, b, c, e1, e2, hg, amp, sp, he},
constexpr int kNCool = 11;
// row k at compile time (the one-thread sum, unrolled)
__host__ __device__ __forceinline__ constexpr CoolTerm cool_row(int k)
{
    constexpr CoolTerm rows[kNCool] = {RTGB_COOL_TERMS(RTGB_COOL_ROW)};
    return rows[k];
}
#undef RTGB_COOL_ROW
#undef RTGB_COOL_TERMS

// ---- rate functions ----
//   Cen (1992) collisional rates A sqrt(T) u exp(-T0/T), u = 1/(1 + sqrt(T/1e5)):
//     Cc = A, c1 = 1/2, c2 = -T0, c3 = 1, z = (ln T - ln 1e5)/2, since
//     ln u = -softplus(z);
//   Hui & Gnedin (1997) fits A lam^p / (1 + (lam/l0)^r)^s, lam = T1/T:
//     Cc = A, c0 = p ln T1, c1 = -p, c3 = s, z = r ln(lam/l0) (the table's
//     argument E_W0 + j: a = -r, c = r (ln T1 - ln l0));
//   alpha_HeII = A (570670/T)^p and the Boltzmann factors: c3 = 0;
//   a cooling term C n_s sqrt(T)^sq u^uu T^tt X1 X2 v^hg adds the exponents
//     of its factors (no term has both u and a Hui & Gnedin factor) and
//     times its density n_s after the function.
// d ln f/dT = (c1 - c2/T - c3 c4 sigma(z)) / T, sigma = e^z / (1 + e^z).
enum {
    RF_COOL0 = 0,                 // slots 0..10: the cooling terms; 11..15 zero
    RF_BETA_HI = 16, RF_ALPHA_HII, RF_BETA_HEI, RF_BETA_HEII, RF_ALPHA_HEII, RF_ALPHA_HEIII,
    NRF
};
static_assert(kNCool <= 16 && NRF <= 32, "function slots fit the tables and the masks of slots");

// The kernels take ln T relative to 2^14 K, the middle of the range that
// matters: |ln(T / 2^14 K)| is a few units where |ln T| is 9, and so are the
// pair roundings of the exponent's terms.  c0 and the reference's share of
// c1 ln T go into the factor, c4's into c5r.
constexpr int kLnTRef = 14;
constexpr double kLnTRefV = 9.704060527839234;   // 14 ln 2

struct RateFn {
    double Cc;
    dfm::F2 c0, c5;             // (with Cc: the function in terms of ln T, for rt_rate_functions)
    dfm::F2 c1, c2, c3, c4, c5r;
    dfm::F2 Cm, c34, c344;      // Cc exp(c0 + c1 14 ln 2) = Cm 2^ke, 1 <= Cm < 2; c3 c4, c3 c4^2
    int ke;
};
struct RateFnTab {
    RateFn f[32];
};

constexpr double kHalfLn1e5 = 5.756462732485114;   // ln(1e5) / 2

// e^x at compile time: Taylor's series of e^(x/2^7) - 1, then seven times
// s -> (1 + s)^2 - 1 (relative error ~1e-15)
constexpr double const_exp(double x)
{
    const double t = x / 128.0;
    double term = 1.0, sum = 0.0;   // sum = e^t - 1
    for (int n = 1; n < 24; ++n) {
        term *= t / n;
        sum += term;
    }
    for (int k = 0; k < 7; ++k) sum = sum * (2.0 + sum);   // (1 + s)^2 - 1
    return 1.0 + sum;
}
constexpr RateFn rate_fn(double Cc, double c0, double c1, double c2, double c3, double c4, double c5)
{
    double m = Cc * const_exp(c0 + c1 * kLnTRefV);
    int e = 0;
    while (m >= 2.0) { m *= 0.5; ++e; }
    while (m > 0.0 && m < 1.0) { m *= 2.0; --e; }
    return RateFn{Cc, pair_of(c0), pair_of(c5), pair_of(c1), pair_of(c2), pair_of(c3), pair_of(c4),
                  pair_of(c5 + c4 * kLnTRefV), pair_of(m), pair_of(c3 * c4), pair_of(c3 * c4 * c4), e};
}
constexpr RateFn cen_fn(double A, double T0) { return rate_fn(A, 0.0, 0.5, -T0, 1.0, 0.5, -kHalfLn1e5); }
constexpr RateFn hg_fn(const RateTable &R, int j)
{
    return rate_fn(R.hg[j].A, R.hg[j].p * R.hg[j].lnT1, -R.hg[j].p, 0.0, R.hg[j].s, R.ea[E_W0 + j].a,
                   R.ea[E_W0 + j].c);
}
constexpr RateFn cool_fn(const RateTable &R, const CoolTerm &q)
{
    double Cc = q.C, c0 = 0.0, c1 = 0.5 * q.sq + q.tt, c2 = 0.0, c3 = 0.0, c4 = 0.0, c5 = 0.0;
    if (q.e1 >= 0) { c0 += R.ea[q.e1].c; c1 += R.ea[q.e1].a; c2 += R.ea[q.e1].b; }
    if (q.e2 >= 0) { c0 += R.ea[q.e2].c; c1 += R.ea[q.e2].a; c2 += R.ea[q.e2].b; }
    if (q.hg >= 0) {
        Cc *= R.hg[q.hg].A;
        c0 += R.hg[q.hg].p * R.hg[q.hg].lnT1;
        c1 -= R.hg[q.hg].p;
        c3 = R.hg[q.hg].s;
        c4 = R.ea[E_W0 + q.hg].a;
        c5 = R.ea[E_W0 + q.hg].c;
    }
    if (q.uu) { c3 = 1.0; c4 = 0.5; c5 = -kHalfLn1e5; }
    if (q.amp) Cc *= R.A_aHeII;
    return rate_fn(Cc, c0, c1, c2, c3, c4, c5);
}
constexpr RateFnTab make_rate_fns(int cb)
{
    RateFnTab t{};
    const RateTable &R = kRateTabCx[cb];
    for (int k = 0; k < kNCool; ++k) t.f[RF_COOL0 + k] = cool_fn(R, cool_row(k));
    for (int k = kNCool; k < 16; ++k) t.f[k] = rate_fn(0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0);
    t.f[RF_BETA_HI] = cen_fn(5.85e-11, 157809.1);
    t.f[RF_ALPHA_HII] = hg_fn(R, HG_ALPHA_HII);
    t.f[RF_BETA_HEI] = cen_fn(2.38e-11, 285335.4);
    t.f[RF_BETA_HEII] = cen_fn(5.68e-12, 631515.0);
    t.f[RF_ALPHA_HEII] = rate_fn(R.A_aHeII, R.ea[E_ALPHA_HEII].c, R.ea[E_ALPHA_HEII].a, R.ea[E_ALPHA_HEII].b, 0.0,
                                 0.0, 0.0);
    t.f[RF_ALPHA_HEIII] = hg_fn(R, HG_ALPHA_HEIII);
    for (int k = NRF; k < 32; ++k) t.f[k] = rate_fn(0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0);
    return t;
}
// uniform reads (one thread, a compile-time slot): the constant cache;
// lane-indexed reads (a warp): global memory through the L1 cache, which
// serves different addresses of a warp in one request
constexpr RateFnTab kRateFnCx[2] = {make_rate_fns(0), make_rate_fns(1)};   // (compile-time queries)
static __constant__ RateFnTab c_rate_fn[2] = {make_rate_fns(0), make_rate_fns(1)};
static __device__ const RateFnTab g_rate_fn[2] = {make_rate_fns(0), make_rate_fns(1)};

// density factor and helium flag of each cooling slot
static __device__ const int g_cool_sp[16] = {SP_HI, SP_HI, SP_HII, SP_FF, SP_HEI, SP_HEII, SP_HEII, SP_HEII,
                                             SP_HEII, SP_HEII, SP_HEIII, 0, 0, 0, 0, 0};

// ln(T / 2^14 K) and 1/T of one temperature as pairs
struct TLevel {
    dfm::F2 lnT, invT;
};
// (the logarithm inline on the fast path)
template <class CTL>
__device__ __forceinline__ void t_level(double T, TLevel &L, CTL &ctl)
{
    using namespace dfm;
    if constexpr (CTL::fast) {
        ctl.odd |= !(T > 0.0) || !splittable(T);
        const F2 T2 = split(T);
        L.lnT = log2f2_inl(T2, kLnTRef);
        L.invT = rcp(T2);
    } else if (!(T > 0.0) || !splittable(T)) {   // not reached by T >= 1 K below 2^60 K
        L.lnT = split_any(log(T) - kLnTRefV);
        L.invT = split_any(1.0 / T);
    } else {
        const F2 T2 = split(T);
        L.lnT = log2f2(T2, kLnTRef);
        L.invT = rcp(T2);
    }
}
// the same from 1/T as a pair
template <class CTL>
__device__ __forceinline__ void t_level_inv(dfm::F2 invT, TLevel &L, CTL &ctl)
{
    using namespace dfm;
    L.invT = invT;
    const bool in = invT.hi > 0x1p-60f && invT.hi < 0x1p60f;
    if constexpr (CTL::fast) {
        ctl.odd |= !in;
        L.lnT = neg(log2f2_inl(in ? invT : F2{1.0f, 0.0f}, -kLnTRef));
    } else if (in) {
        L.lnT = neg(log2f2(invT, -kLnTRef));
    } else {
        L.lnT = split_any(-log(to_double(invT)) - kLnTRefV);
    }
}

// A function value y 2^m (y a normalised pair below 8, or 0), as pairs
// g = d ln f / d ln T and, for the adjoint, w = T^2 f'' / f = g^2 - g + c2/T -
// c3 c4^2 sigma (1 - sigma)
struct RateVal {
    dfm::F2 y, g, w;
    int m;
};

// Slots by the terms of their exponent, so that one thread can leave out
// what is zero (adding a zero pair or multiplying by one returns the same
// normalised pair, so both paths still give the same bits).
__host__ __device__ constexpr unsigned rf_bit(int k) { return 1u << k; }
enum { kZeroC1, kZeroC2, kZeroC3 };
constexpr unsigned rf_zero_mask(int what)
{
    unsigned m = 0;
    for (int k = 0; k < NRF; ++k) {
        bool z = true;
        for (int cb = 0; cb < 2; ++cb) {
            const RateFn &q = kRateFnCx[cb].f[k];
            const float v = what == kZeroC1 ? q.c1.hi : what == kZeroC2 ? q.c2.hi : q.c3.hi;
            z = z && v == 0.0f;
        }
        if (z) m |= rf_bit(k);
    }
    return m;
}
// slots whose softplus is that of u (c3 = 1, z = (ln T - ln 1e5)/2, the same in all of them)
constexpr unsigned rf_u_mask()
{
    unsigned m = rf_bit(RF_BETA_HI) | rf_bit(RF_BETA_HEI) | rf_bit(RF_BETA_HEII);
    for (int k = 0; k < kNCool; ++k)
        if (cool_row(k).uu) m |= rf_bit(RF_COOL0 + k);
    return m;
}
constexpr unsigned kC1Zero = rf_zero_mask(kZeroC1), kC2Zero = rf_zero_mask(kZeroC2), kC3Zero = rf_zero_mask(kZeroC3),
                   kSlotU = rf_u_mask();

// softplus(z) and sigma(z) of one function, z = c4 ln(T / 2^14 K) + c5r.  MIX (the
// mixed-precision thermochemistry, RT_MIXED32): z still in pairs, but the
// correction ln(1 + e^-|z|) < ln 2 and sigma in FP32.
template <bool MIX, class CTL>
__device__ __forceinline__ dfm::F2 rate_softplus(const RateFn &q, const TLevel &L, dfm::F2 &sig, CTL &ctl)
{
    using namespace dfm;
    const F2 z = norm(addu(mulu(L.lnT, q.c4), q.c5r));
    if constexpr (MIX) {
        const float e = __expf(-fabsf(z.hi));
        sig = F2{(z.hi >= 0.0f ? 1.0f : e) / (1.0f + e), 0.0f};
        return add(z.hi >= 0.0f ? z : F2{0.0f, 0.0f}, log1pf(e));   // max(z, 0) + ln(1 + e^-|z|)
    } else {
        return softplus2(z, sig, ctl);
    }
}

template <bool MIX>
__device__ __forceinline__ dfm::F2 rate_softplus(const RateFn &q, const TLevel &L, dfm::F2 &sig)
{
    dfm::Exact e;
    return rate_softplus<MIX>(q, L, sig, e);
}

// One function from l = softplus(z) and sigma(z).  The argument of the
// exponential is formed in pairs on every path (it reaches |20-60|, where a
// float's rounding alone is 1e-6 of the rate, and over thousands of
// sub-steps that moved N by 2e-4 of the FP64 result); MIX takes the
// exponential of the reduced argument and the log-derivative in FP32
// (relative accuracy ~2e-7).  zero: bits kZero* of the terms known to be
// zero (compile-time), one3: c3 = 1.
template <bool MIX, int DERIV>
__device__ __forceinline__ void rate_val(const RateFn &q, const TLevel &L, dfm::F2 l, dfm::F2 sig, unsigned zero,
                                         bool one3, RateVal &r)
{
    using namespace dfm;
    const F2 nil{0.0f, 0.0f};
    const F2 b = (zero >> kZeroC2 & 1) ? nil : mulu(L.invT, q.c2);
    F2 arg = (zero >> kZeroC1 & 1) ? nil : mulu(L.lnT, q.c1);
    if (!(zero >> kZeroC2 & 1)) arg = addu(arg, b);
    if (!(zero >> kZeroC3 & 1)) arg = addu(arg, neg(one3 ? l : mulu(l, q.c3)));
    arg = norm(arg);
    if (arg.hi < -1400.0f) arg = F2{-1400.0f, 0.0f};   // 0 in every use
    if constexpr (MIX) {
        const float kf = rintf(__fmul_rn(arg.hi, 1.44269504f));
        const float t = __fadd_rn(__fmaf_rn(-kf, -1.90465421e-9f, __fmaf_rn(-kf, 0.693147182f, arg.hi)), arg.lo);
        r.y = mul(q.Cm, expf(t));
        r.m = (int)kf + q.ke;
        if constexpr (DERIV > 0)
            r.g = F2{__fmaf_rn(-q.c34.hi, sig.hi, __fmaf_rn(-q.c2.hi, L.invT.hi, q.c1.hi)), 0.0f};
    } else {
        int m;
        exp_pair(arg, r.y, m);
        r.y = norm(mulu(q.Cm, r.y));
        r.m = m + q.ke;
        if constexpr (DERIV > 0) {
            F2 g = (zero >> kZeroC1 & 1) ? nil : q.c1;
            if (!(zero >> kZeroC2 & 1)) g = addu(g, neg(b));
            if (!(zero >> kZeroC3 & 1)) g = addu(g, neg(mulu(sig, q.c34)));
            r.g = norm(g);
        }
        if constexpr (DERIV > 1) {
            F2 w = addu(addu(mulu(r.g, r.g), neg(r.g)), b);
            r.w = norm(addu(w, neg(mulu(q.c344, addu(sig, neg(mulu(sig, sig)))))));
        }
    }
}
template <class CTL>
__device__ __forceinline__ double rate_f(const RateVal &r, CTL &ctl) { return dfm::to_double_c(r.y, r.m, ctl); }
__device__ __forceinline__ double rate_f(const RateVal &r) { return dfm::to_double_i(r.y, r.m); }
// df/dT = f g / T
template <class CTL>
__device__ __forceinline__ double rate_df(const RateVal &r, const TLevel &L, CTL &ctl)
{
    using namespace dfm;
    return to_double_c(norm(mulu(r.y, mulu(r.g, L.invT))), r.m, ctl);
}
// T df/dT = f g, and its T-derivative f (g + w) / T
// (the hydrogen update needs df/dT only times T: two FP64 products of an
// attempt less; 48^3 without the OTSA 10.1 -> 9.8 ms, 256^3 33.4 -> 32.9 ms)
template <class CTL>
__device__ __forceinline__ double rate_tdf(const RateVal &r, CTL &ctl)
{
    return dfm::to_double_c(dfm::norm(dfm::mulu(r.y, r.g)), r.m, ctl);
}
template <class CTL>
__device__ __forceinline__ double rate_dtdf(const RateVal &r, const TLevel &L, CTL &ctl)
{
    using namespace dfm;
    return to_double_c(norm(mulu(mulu(r.y, L.invT), addu(r.g, r.w))), r.m, ctl);
}

// values (and derivatives) of several functions at one temperature
template <typename S>
struct RatesT {
    S f[NRF], tdf[NRF];   // f, T df/dT
};
using Rates = RatesT<double>;

constexpr unsigned kNeedH = rf_bit(RF_BETA_HI) | rf_bit(RF_ALPHA_HII);   // values and derivatives
constexpr unsigned kNeedHe = rf_bit(RF_BETA_HEI) | rf_bit(RF_BETA_HEII) | rf_bit(RF_ALPHA_HEII) |
                             rf_bit(RF_ALPHA_HEIII);
constexpr unsigned kNeedHe3 = rf_bit(RF_BETA_HEII) | rf_bit(RF_ALPHA_HEIII);
constexpr unsigned kNeedRec = rf_bit(RF_ALPHA_HII) | rf_bit(RF_ALPHA_HEII) | rf_bit(RF_ALPHA_HEIII);
__host__ __device__ constexpr unsigned cool_mask(int he)
{
    unsigned m = 0;
    for (int k = 0; k < kNCool; ++k)
        if (cool_row(k).he == he) m |= rf_bit(RF_COOL0 + k);
    return m;
}

// one thread: slot k (a constant once unrolled) at level L, given the
// softplus of u
template <bool MIX, int DERIV>
__device__ __forceinline__ void rate_serial(int k, const RateFnTab &R, const TLevel &L, dfm::F2 lu, dfm::F2 su,
                                            RateVal &r, dfm::F2 &sig)
{
    const unsigned zero = (kC1Zero >> k & 1) << kZeroC1 | (kC2Zero >> k & 1) << kZeroC2 | (kC3Zero >> k & 1) << kZeroC3;
    dfm::F2 l = lu;
    sig = su;
    if (!(kSlotU & rf_bit(k)) && !(kC3Zero & rf_bit(k))) l = rate_softplus<MIX>(R.f[k], L, sig);
    rate_val<MIX, DERIV>(R.f[k], L, l, sig, zero, (kSlotU & rf_bit(k)) != 0, r);
}

// one thread: the functions in needF (derivatives of those in needD); the
// shared softplus of u once
template <bool MIX>
__device__ __forceinline__ void rates_serial(const TLevel &L, int case_b, unsigned needF, unsigned needD, Rates &r)
{
    const RateFnTab &R = c_rate_fn[case_b];
    dfm::F2 lu{0.0f, 0.0f}, su{0.0f, 0.0f};
    if (needF & kSlotU) lu = rate_softplus<MIX>(R.f[RF_BETA_HI], L, su);
#pragma unroll
    for (int k = 0; k < NRF; ++k) {
        if (needF & rf_bit(k)) {
            RateVal v;
            dfm::F2 sig;
            if (needD & rf_bit(k)) {
                rate_serial<MIX, 1>(k, R, L, lu, su, v, sig);
                dfm::Exact e;
                r.tdf[k] = rate_tdf(v, e);
            } else {
                rate_serial<MIX, 0>(k, R, L, lu, su, v, sig);
            }
            r.f[k] = rate_f(v);
        }
    }
}

// ---- teams: TS (2, 4 or 8) adjacent lanes of a warp work on one cell, holding
// the same state and sharing its rate functions ----
template <int TS>
__device__ __forceinline__ int team_lane() { return (int)(threadIdx.x & (TS - 1)); }
template <int TS>
__device__ __forceinline__ unsigned team_mask()
{
    static_assert(TS == 1 || TS == 2 || TS == 4 || TS == 8, "team sizes");
    return ((1u << TS) - 1u) << (threadIdx.x & 31u & ~(TS - 1u));
}
// ... of the shuffles and votes of an attempt.  On the fast path of teams of
// two and of the adjoint's teams of eight the whole warp runs it (teams
// without a cell on whatever they hold), with a constant full mask.  Teams of
// four, often one to a warp, run without the others (a lone cell's attempt
// took 4% longer with the idle lanes' table reads).
template <int TS>
__host__ __device__ constexpr bool whole_warp() { return TS == 2 || TS == 8; }
template <int TS, class CTL>
__device__ __forceinline__ unsigned team_mask_c()
{
    if constexpr (CTL::fast && whole_warp<TS>()) return 0xffffffffu;
    else return team_mask<TS>();
}
template <int TS>
__device__ __forceinline__ double team_get(unsigned m, double v, int src) { return __shfl_sync(m, v, src, TS); }

// one function per lane of a team, slot k, with its own softplus
template <bool MIX, int DERIV, class CTL>
__device__ __forceinline__ void rate_lane(int case_b, int k, const TLevel &L, RateVal &r, CTL &ctl)
{
    const RateFn &q = g_rate_fn[case_b].f[k];
    dfm::F2 sig;
    const dfm::F2 l = rate_softplus<MIX>(q, L, sig, ctl);
    rate_val<MIX, DERIV>(q, L, l, sig, 0u, false, r);
}

template <typename S>
struct HRatesT {      // rates needed by the x_HII update
    S beta, tbeta, alpha, talpha;   // f and T df/dT
};
template <typename S>
struct HeRatesT {
    S beta_HeI, beta_HeII, alpha_HeII, alpha_HeIII;
};
using HRates = HRatesT<double>;
using HeRates = HeRatesT<double>;

template <typename S>
__device__ __forceinline__ void h_rates_from(const RatesT<S> &t, HRatesT<S> &r)
{
    r.beta = t.f[RF_BETA_HI];
    r.tbeta = t.tdf[RF_BETA_HI];
    r.alpha = t.f[RF_ALPHA_HII];
    r.talpha = t.tdf[RF_ALPHA_HII];
}

template <typename S>
__device__ __forceinline__ void he_rates_from(const RatesT<S> &t, HeRatesT<S> &r)
{
    r.beta_HeI = t.f[RF_BETA_HEI];
    r.beta_HeII = t.f[RF_BETA_HEII];
    r.alpha_HeII = t.f[RF_ALPHA_HEII];
    r.alpha_HeIII = t.f[RF_ALPHA_HEIII];
}

// The sets of functions an attempt needs at one temperature, out of line:
// they do not depend on the group count, and inlined into every
// instantiation of the one-thread kernels they made ptxas run for minutes.
template <bool MIX>
static __device__ __noinline__ HRates h_rates_serial(TLevel L, int case_b)
{
    Rates t;
    HRates r;
    rates_serial<MIX>(L, case_b, kNeedH, kNeedH, t);
    h_rates_from(t, r);
    return r;
}
template <bool MIX>
static __device__ __noinline__ HeRates he_rates_serial(TLevel L, int case_b)
{
    Rates t;
    HeRates r;
    rates_serial<MIX>(L, case_b, kNeedHe, 0u, t);
    he_rates_from(t, r);
    return r;
}
template <bool MIX>
static __device__ __noinline__ double2 he3_rates_serial(TLevel L, int case_b)
{
    Rates t;
    rates_serial<MIX>(L, case_b, kNeedHe3, 0u, t);
    return make_double2(t.f[RF_BETA_HEII], t.f[RF_ALPHA_HEIII]);
}
// ... and by a team: lanes 0 and 1 the two hydrogen functions, lanes 0..3 (a
// team of two: twice lanes 0, 1) the four helium ones, each then in every lane
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ HRates h_rates_team(const TLevel &L, int case_b, CTL &ctl)
{
    const unsigned m = team_mask_c<TS, CTL>();
    RateVal v;
    rate_lane<MIX, 1>(case_b, team_lane<TS>() == 0 ? RF_BETA_HI : RF_ALPHA_HII, L, v, ctl);
    const double f = rate_f(v, ctl), tdf = rate_tdf(v, ctl);
    HRates r;
    r.beta = team_get<TS>(m, f, 0);
    r.tbeta = team_get<TS>(m, tdf, 0);
    r.alpha = team_get<TS>(m, f, 1);
    r.talpha = team_get<TS>(m, tdf, 1);
    return r;
}
static_assert(RF_BETA_HEII == RF_BETA_HEI + 1 && RF_ALPHA_HEII == RF_BETA_HEI + 2 && RF_ALPHA_HEIII == RF_BETA_HEI + 3,
              "the helium functions of a team's lanes");
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ HeRates he_rates_team(const TLevel &L, int case_b, CTL &ctl)
{
    const unsigned m = team_mask_c<TS, CTL>();
    RateVal v;
    rate_lane<MIX, 0>(case_b, RF_BETA_HEI + (team_lane<TS>() & 3), L, v, ctl);
    const double f = rate_f(v, ctl);
    HeRates r;
    r.beta_HeI = team_get<TS>(m, f, 0);
    r.beta_HeII = team_get<TS>(m, f, 1);
    if constexpr (TS >= 4) {
        r.alpha_HeII = team_get<TS>(m, f, 2);
        r.alpha_HeIII = team_get<TS>(m, f, 3);
    } else {   // lanes 0, 1 once more
        rate_lane<MIX, 0>(case_b, RF_BETA_HEI + 2 + team_lane<TS>(), L, v, ctl);
        const double g = rate_f(v, ctl);
        r.alpha_HeII = team_get<TS>(m, g, 0);
        r.alpha_HeIII = team_get<TS>(m, g, 1);
    }
    return r;
}
// dual numbers, by a team of eight lanes that hold the same value and each
// their own tangent (level L of the value, dT this lane's tangent of T): the
// values are those above, f carries df/dT dT and T df/dT carries its derivative
template <class CTL>
__device__ __forceinline__ HRatesT<Dual> h_rates_dual(const TLevel &L, double dT, int case_b, CTL &ctl)
{
    const unsigned m = team_mask_c<8, CTL>();
    RateVal v;
    rate_lane<false, 2>(case_b, team_lane<8>() == 0 ? RF_BETA_HI : RF_ALPHA_HII, L, v, ctl);
    const double f = rate_f(v, ctl), df = rate_df(v, L, ctl);
    const double tdf = rate_tdf(v, ctl), dtdf = rate_dtdf(v, L, ctl);
    HRatesT<Dual> r;
    r.beta = Dual(team_get<8>(m, f, 0), team_get<8>(m, df, 0) * dT);
    r.tbeta = Dual(team_get<8>(m, tdf, 0), team_get<8>(m, dtdf, 0) * dT);
    r.alpha = Dual(team_get<8>(m, f, 1), team_get<8>(m, df, 1) * dT);
    r.talpha = Dual(team_get<8>(m, tdf, 1), team_get<8>(m, dtdf, 1) * dT);
    return r;
}
template <class CTL>
__device__ __forceinline__ HeRatesT<Dual> he_rates_dual(const TLevel &L, double dT, int case_b, CTL &ctl)
{
    const unsigned m = team_mask_c<8, CTL>();
    RateVal v;
    rate_lane<false, 1>(case_b, RF_BETA_HEI + (team_lane<8>() & 3), L, v, ctl);
    const double f = rate_f(v, ctl), df = rate_df(v, L, ctl);
    HeRatesT<Dual> r;
    r.beta_HeI = Dual(team_get<8>(m, f, 0), team_get<8>(m, df, 0) * dT);
    r.beta_HeII = Dual(team_get<8>(m, f, 1), team_get<8>(m, df, 1) * dT);
    r.alpha_HeII = Dual(team_get<8>(m, f, 2), team_get<8>(m, df, 2) * dT);
    r.alpha_HeIII = Dual(team_get<8>(m, f, 3), team_get<8>(m, df, 3) * dT);
    return r;
}

// Recombination rates of HII, HeII, HeIII (the case t was evaluated with)
template <typename S>
__device__ __forceinline__ void recomb_alphas(const RatesT<S> &t, S a[3])
{
    a[0] = t.f[RF_ALPHA_HII];
    a[1] = t.f[RF_ALPHA_HEII];
    a[2] = t.f[RF_ALPHA_HEIII];
}

// Primordial cooling magnitude L (Eq. (rate_cooling), positive = cooling)
// and dL/dT: the sum of the cooling functions (collisional ionisation and
// excitation, recombination and dielectronic cooling, bremsstrahlung) each
// times its density, in a fixed pairwise order, then Compton cooling.  The
// terms, scaled by 2^kCoolExp, and their sums are float pairs (2^-46, the
// accuracy of the functions themselves is 1e-14 to 1e-12): before, 11
// functions and derivatives entered FP64 one by one, 90 of an attempt's FP64
// instructions.  The one-thread sum and the teams' sums run the same
// operations and give the same bits.
constexpr int kCoolExp = 80;
// Terms whose function is below 2^kCoolCut on this scale (6e-55 erg cm^3 s^-1) count
// as zero: with n_HII >= 1e-6 n_H, the floor of x_HII, they are below 2^-48 of the
// bremsstrahlung whatever the densities they are multiplied by.  (At -60 the
// excitation cooling of neutral gas near 2000 K was lost, up to 1e-11 of it.)
// Above it the low floats stay clear of float subnormals.
constexpr int kCoolCut = -100;

// a[i] through selects (registers, not local memory, for a lane-dependent
// i; a plain a[i] once unrolled with a constant i)
template <typename T, int N>
__device__ __forceinline__ T pick(const T (&a)[N], int i)
{
    T r = a[0];
#pragma unroll
    for (int j = 1; j < N; ++j) r = (i == j) ? a[j] : r;
    return r;
}

template <typename S>
__device__ __forceinline__ void cool_densities(const S &nHI, const S &nHII, const S &nHeI, const S &nHeII,
                                               const S &nHeIII, S n[NSP])
{
    n[SP_HI] = nHI;
    n[SP_HII] = nHII;
    n[SP_HEI] = nHeI;
    n[SP_HEII] = nHeII;
    n[SP_HEIII] = nHeIII;
    n[SP_FF] = rfma(4.0, nHeIII, radd(nHII, nHeII));
}

// a density as a pair (below 2^-70, 1e-21 of the smallest electron density
// that matters, as 0; 2^120 and above through the FP64 pipe)
__device__ __forceinline__ dfm::F2 split_density(double n);
template <class CTL>
__device__ __forceinline__ dfm::F2 split_density(double n, CTL &ctl)
{
    if constexpr (CTL::fast) {
        const unsigned h = (unsigned)((unsigned long long)__double_as_longlong(n) >> 32);
        ctl.odd |= h >= (1143u << 20);
        const dfm::F2 s = dfm::split_near(n);
        return h < (953u << 20) ? dfm::F2{0.0f, 0.0f} : s;
    } else {
        return split_density(n);
    }
}
__device__ __forceinline__ dfm::F2 split_density(double n)
{
    const unsigned h = (unsigned)((unsigned long long)__double_as_longlong(n) >> 32);
    if (h < (953u << 20)) return {0.0f, 0.0f};
    if (h >= (1143u << 20)) return dfm::split_any(n);
    return dfm::split_near(n);
}

// a term f n (scaled) and f n g, g = d ln f/d ln T
__device__ __forceinline__ void cool_term(const RateVal &r, dfm::F2 n, dfm::F2 &v, dfm::F2 &dv)
{
    using namespace dfm;
    const int e = r.m + kCoolExp;
    const float sc = e < kCoolCut ? 0.0f : pow2f(e > 100 ? 100 : e);
    v = mulu(F2{r.y.hi * sc, r.y.lo * sc}, n);
    dv = mulu(v, r.g);
}

// + Compton, varpi = comp (T - T_gamma), comp = 1.017e-37 T_gamma^4 and
// T_gamma = 2.727/a (ThermoParams::comp, ::tg); both sums times n_e
template <typename S>
__device__ __forceinline__ void cooling_close(double comp, double tg, const S &T, const S &ne, const S &Ls,
                                              const S &dLs, S &L, S &dL)
{
    L = rmul(ne, rfma(comp, radd(T, S(-tg)), Ls));
    dL = rmul(ne, radd(dLs, S(comp)));
}

// The terms' places in the sums: place t + TS r is lane t's term of round r in
// a team of TS, the last place empty.  The order gives the two terms with a
// softplus of their own places 2 and 3 beside the first two of u, so a team
// of four or eight evaluates one softplus per lane, a team of two two.
__host__ __device__ __forceinline__ constexpr int cool_at(int place)
{
    constexpr int at[12] = {0, 1, 2, 10, 4, 5, 6, 7, 8, 9, 3, -1};
    return at[place];
}
static __device__ const int g_cool_at[12] = {0, 1, 2, 10, 4, 5, 6, 7, 8, 9, 3, 11};

// the sum over the places in a fixed pairwise order: places 8 apart, 4
// apart, then 2 and 1 (the empty one left out)
__device__ __forceinline__ dfm::F2 tree_sum(const dfm::F2 (&a)[kNCool])
{
    using dfm::addu;
    const dfm::F2 s0 = addu(a[cool_at(0)], a[cool_at(8)]), s1 = addu(a[cool_at(1)], a[cool_at(9)]),
                  s2 = addu(a[cool_at(2)], a[cool_at(10)]);
    const dfm::F2 t0 = addu(s0, a[cool_at(4)]), t1 = addu(s1, a[cool_at(5)]), t2 = addu(s2, a[cool_at(6)]),
                  t3 = addu(a[cool_at(3)], a[cool_at(7)]);
    return dfm::norm(addu(addu(t0, t2), addu(t1, t3)));
}

// one thread
template <bool MIX>
__device__ __forceinline__ void cooling_sums(const TLevel &L, int case_b, bool helium, const double *n, double &Ls,
                                             double &dLs)
{
    using namespace dfm;
    const RateFnTab &R = c_rate_fn[case_b];
    F2 np[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) np[k] = split_density(n[k]);
    F2 su;
    const F2 lu = rate_softplus<MIX>(R.f[RF_BETA_HI], L, su);
    F2 a[kNCool], b[kNCool];
#pragma unroll
    for (int k = 0; k < kNCool; ++k) {
        const CoolTerm q = cool_row(k);
        a[k] = b[k] = F2{0.0f, 0.0f};
        if (helium || !q.he) {
            RateVal v;
            F2 sig;
            rate_serial<MIX, 1>(k, R, L, lu, su, v, sig);
            cool_term(v, np[q.sp], a[k], b[k]);
        }
    }
    Ls = to_double_i(tree_sum(a), -kCoolExp);
    dLs = to_double_i(norm(mulu(tree_sum(b), L.invT)), -kCoolExp);
}

// (out of line, as the rate sets above)
template <bool MIX>
static __device__ __noinline__ double2 cooling_sums_serial(int case_b, bool helium, double T, double nHI, double nHII,
                                                           double nHeI, double nHeII, double nHeIII)
{
    TLevel Lv;
    dfm::Exact e;
    t_level(T, Lv, e);
    double n[NSP], Ls, dLs;
    cool_densities(nHI, nHII, nHeI, nHeII, nHeIII, n);
    cooling_sums<MIX>(Lv, case_b, helium, n, Ls, dLs);
    return make_double2(Ls, dLs);
}
template <bool MIX>
__device__ __forceinline__ void cooling_serial(int case_b, double comp, double tg, bool helium, double T, double ne,
                                               double nHI, double nHII, double nHeI, double nHeII, double nHeIII,
                                               double &L, double &dL)
{
    const double2 s = cooling_sums_serial<MIX>(case_b, helium, T, nHI, nHII, nHeI, nHeII, nHeIII);
    cooling_close(comp, tg, T, ne, s.x, s.y, L, dL);
}

// a team of TS = 2 or 4: places t, t + TS, ..., the last sums over shuffles,
// in the order of tree_sum
__device__ __forceinline__ dfm::F2 team_add(unsigned mask, dfm::F2 a, int m)
{
    return dfm::addu(a, dfm::F2{__shfl_xor_sync(mask, a.hi, m), __shfl_xor_sync(mask, a.lo, m)});
}
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ double2 cooling_sums_team(int case_b, bool helium, double T, double nHI, double nHII,
                                                     double nHeI, double nHeII, double nHeIII, CTL &ctl)
{
    using namespace dfm;
    static_assert(TS == 2 || TS == 4, "team sizes");
    const unsigned mask = team_mask_c<TS, CTL>();
    const int t = team_lane<TS>();
    const RateFn *R = g_rate_fn[case_b].f;
    TLevel L;
    t_level(T, L, ctl);
    double n[NSP];
    cool_densities(nHI, nHII, nHeI, nHeII, nHeIII, n);
    // the softplus of u: lane 0's of round 0 (a team of two: of both lanes);
    // places 2 and 3 have their own, places 7 to 11 none (c3 = c3 c4 = 0)
    F2 l, sig;
    l = rate_softplus<MIX>(R[g_cool_at[t]], L, sig, ctl);
    F2 lu = l, su = sig;
    if constexpr (TS == 4) {
        lu = F2{__shfl_sync(mask, l.hi, 0, TS), __shfl_sync(mask, l.lo, 0, TS)};
        su = F2{__shfl_sync(mask, sig.hi, 0, TS), __shfl_sync(mask, sig.lo, 0, TS)};
    }
    constexpr int NR = 12 / TS;
    F2 v[NR], dv[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
        const int k = g_cool_at[t + TS * r];
        const bool own = r * TS < 4;   // the round has a softplus of its own
        if (own && r > 0) l = rate_softplus<MIX>(R[k], L, sig, ctl);
        RateVal q;
        rate_val<MIX, 1>(R[k], L, own ? l : lu, own ? sig : su, r * TS >= 8 ? 1u << kZeroC3 : 0u, false, q);
        cool_term(q, split_density(pick(n, g_cool_sp[k]), ctl), v[r], dv[r]);
        if (k >= kNCool || (!helium && (cool_mask(1) >> k & 1))) v[r] = dv[r] = F2{0.0f, 0.0f};
    }
    // places 8 apart, 4 apart, 2 and 1 apart
#pragma unroll
    for (int r = 0; r < 4 / TS; ++r) {
        v[r] = addu(addu(v[r], v[r + 8 / TS]), v[r + 4 / TS]);
        dv[r] = addu(addu(dv[r], dv[r + 8 / TS]), dv[r + 4 / TS]);
    }
    F2 s = v[0], ds = dv[0];
    if constexpr (TS == 2) {
        s = addu(s, v[1]);
        ds = addu(ds, dv[1]);
    } else {
        s = team_add(mask, s, 2);
        ds = team_add(mask, ds, 2);
    }
    s = norm(team_add(mask, s, 1));
    ds = norm(team_add(mask, ds, 1));
    return make_double2(to_double_c(s, -kCoolExp, ctl), to_double_c(norm(mulu(ds, L.invT)), -kCoolExp, ctl));
}

// dual numbers, by a team of eight (same values, a tangent per lane): places
// t and t + 8; the values as above.  With the sums over the species s of
// F_s = sum f and their T-derivatives, the tangents are dL = sum F_s dn_s +
// L_T dT and dL_T = sum F_s' dn_s + L_TT dT.
template <class CTL>
__device__ __forceinline__ void cooling_dual(int case_b, double comp, double tg, bool helium, const Dual &T,
                                             const Dual &ne, const Dual &nHI, const Dual &nHII, const Dual &nHeI,
                                             const Dual &nHeII, const Dual &nHeIII, Dual &L, Dual &dL, CTL &ctl)
{
    using namespace dfm;
    const unsigned mask = team_mask_c<8, CTL>();
    const int t = team_lane<8>();
    const RateFn *R = g_rate_fn[case_b].f;
    TLevel Lv;
    t_level(T.v, Lv, ctl);
    Dual n[NSP];
    cool_densities(nHI, nHII, nHeI, nHeII, nHeIII, n);
    double nv[NSP];
#pragma unroll
    for (int k = 0; k < NSP; ++k) nv[k] = n[k].v;
    F2 v[2], dv[2], d2[2];
    double f[2], df[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
        const int k = r ? (t < 4 ? g_cool_at[t + 8] : kNCool) : g_cool_at[t];
        F2 sig{0.0f, 0.0f}, l{0.0f, 0.0f};
        if (r == 0) l = rate_softplus<false>(R[k], Lv, sig, ctl);   // (none in places 8 to 11)
        RateVal q;
        rate_val<false, 2>(R[k], Lv, l, sig, r ? 1u << kZeroC3 : 0u, false, q);
        cool_term(q, split_density(pick(nv, g_cool_sp[k]), ctl), v[r], dv[r]);
        d2[r] = mulu(v[r], q.w);
        f[r] = rate_f(q, ctl);
        df[r] = rate_df(q, Lv, ctl);
        if (k >= kNCool || (!helium && (cool_mask(1) >> k & 1))) {
            v[r] = dv[r] = d2[r] = F2{0.0f, 0.0f};
            f[r] = df[r] = 0.0;
        }
    }
    F2 s = addu(v[0], v[1]), ds = addu(dv[0], dv[1]), d2s = addu(d2[0], d2[1]);
#pragma unroll
    for (int m = 4; m >= 1; m >>= 1) {
        s = team_add(mask, s, m);
        ds = team_add(mask, ds, m);
        d2s = team_add(mask, d2s, m);
    }
    const double Ls = to_double_c(norm(s), -kCoolExp, ctl);
    const double dLs = to_double_c(norm(mulu(norm(ds), Lv.invT)), -kCoolExp, ctl);
    const double d2Ls = to_double_c(norm(mulu(mulu(d2s, Lv.invT), Lv.invT)), -kCoolExp, ctl);
    double tL = dLs * T.d, tdL = d2Ls * T.d;
#pragma unroll
    for (int p = 0; p < kNCool; ++p) {
        const int sp = cool_row(cool_at(p)).sp;
        tL = ::fma(team_get<8>(mask, f[p / 8], p % 8), n[sp].d, tL);
        tdL = ::fma(team_get<8>(mask, df[p / 8], p % 8), n[sp].d, tdL);
    }
    cooling_close(comp, tg, T, ne, Dual(Ls, tL), Dual(dLs, tdL), L, dL);
}

}  // namespace rtgb
