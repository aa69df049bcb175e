// One thermo_step of the per-cell thermochemistry (paper App. A) and one
// attempt of its sub-cycling loop (Sec. 3.3.1), shared by the forward
// kernels (thermo.cu) and the adjoint's differentiated recomputation
// (adjoint.cu).  The scalar type S is double, or Dual for the adjoint.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "dual.cuh"
#include "rates.cuh"
#include "rt_internal.h"

namespace rtgb {
namespace thermo_detail {

constexpr double kEV = 1.602176634e-12;
constexpr double kEps0 = 13.60 * kEV, kEps1 = 24.59 * kEV, kEps2 = 54.42 * kEV;
constexpr double kFloorN = 1e-30;
constexpr double kXMin = 1e-6;
constexpr double kNeFloor = 1e-6;
constexpr double kTFloor = 1.0;

// Photon groups a lane holds: all G of them (PT = 1, or dual numbers), or
// those of its place in a team of PT lanes, group r PT + t in place r.
template <typename S = double>
__host__ __device__ constexpr int lane_groups(int G, int PT)
{
    return std::is_same<S, double>::value ? (G + PT - 1) / PT : G;
}

template <int NG, typename S = double>
struct CellState {
    S x, y2, y3, T;
    S N[NG];
    S Fs[NG];         // accumulated flux scale prod 1/(1 + h D_i)
    S Nd[NG];         // smoothed RT: photon density rate Ndot_i (Sec. 3.4)
    S Fb[NG];         // smoothed RT: weight of Fdot_i in F, sum h prod 1/(1 + h D_i)
};

template <typename S = double>
struct IsoRates {     // quantities of a cell fixed over its sub-steps
    HRatesT<S> h;     // rates at the fixed temperature of an isothermal cell
    HeRatesT<S> he;
    S nHe, K, nef;    // n_He, (gamma - 1) X / (k_B n_H), the n_e floor 1e-6 n_H
};

template <typename S = double>
struct CoolCache {    // quantities of the current state at t, kept over rejected attempts
    S L, dL;          // cooling and dL/dT
    S rj[3];          // without the OTSA: (alpha^A_j - alpha^B_j) n_j n_e, j = HII, HeII, HeIII
    bool valid, rvalid;
};

template <typename S>
__device__ __forceinline__ void cell_constants(const ThermoParams &p, const S &nH, IsoRates<S> &iso)
{
    iso.nHe = nH * p.he_ratio;
    dfm::Exact e;
    iso.K = cdiv(S(p.kfac), nH, e);
    iso.nef = kNeFloor * nH;
}

// y2 + 2 y3, electrons per helium nucleus
template <typename S>
__device__ __forceinline__ S he_electrons(const S &y2, const S &y3)
{
    return rfma(2.0, y3, y2);
}

// n_e given q = he_electrons
template <typename S>
__device__ __forceinline__ S ne_of(const S &nHII, const S &q, const S &nHe)
{
    return rfma(q, nHe, nHII);
}

// 1/mu = X (1 + x) + (1 - X)(1 + y2 + 2 y3)/4, mu the mean particle mass in
// m_H (App. A): X x + md_he(q), md_he(q) = X + (1 - X)(1 + q)/4
template <typename S>
__device__ __forceinline__ S md_he(const ThermoParams &p, const S &q)
{
    return rfma(p.mu_w, q, S(p.mu_0));
}
template <typename S>
__device__ __forceinline__ S mu_den(const ThermoParams &p, const S &x, const S &mhe)
{
    return rfma(p.X, x, mhe);
}

// Comparisons, minima and maxima of doubles through their bit patterns, on
// the integer pipe (a GB300 warp issues one FP64 instruction, compares and
// min/max included, per ~64 cycles).  For doubles >= +0 the signed 64-bit
// order of the bits is the order of the values, and every negative double
// orders below them, so these are exact wherever at most one operand can be
// negative; a NaN orders above +infinity.
constexpr long long kInfBits = 0x7ff0000000000000LL;

__device__ __forceinline__ long long dbits(double x) { return __double_as_longlong(x); }

// max(x, c), min(x, c) for c >= +0 and any x (dual numbers: fmax, fmin)
template <typename S, typename C>
__device__ __forceinline__ S max0(const S &x, C c)
{
    if constexpr (std::is_same<S, double>::value && std::is_same<C, double>::value)
        return __longlong_as_double(max(dbits(x), dbits(c)));
    else
        return fmax(x, c);
}

template <typename S, typename C>
__device__ __forceinline__ S min0(const S &x, C c)
{
    if constexpr (std::is_same<S, double>::value && std::is_same<C, double>::value)
        return __longlong_as_double(min(dbits(x), dbits(c)));
    else
        return fmin(x, c);
}

// 2 h and h / 2 of a positive normal h: the exponent moved by one (exact)
__device__ __forceinline__ double twice(double h)
{
    return (dbits(h) >> 52) < 2046 ? __longlong_as_double(dbits(h) + (1LL << 52)) : 2.0 * h;
}

__device__ __forceinline__ double half(double h)
{
    return (dbits(h) >> 52) > 1 ? __longlong_as_double(dbits(h) - (1LL << 52)) : 0.5 * h;
}

// fl(a / b) > t and fl(a / b) < t (a >= 0, b > 0), decided exactly as the
// rounded quotient would decide them: the product t b settles everything
// more than 8 ulps away from it (for doubles, by their bits; the rounding
// of t b and of the quotient is within 2 ulps), and the quotient itself is
// formed only inside that band (or for a NaN, which then compares false as
// the quotient would).  The 10% rule's decisions thus match a statement of
// it that divides, including at exact ties (a sub-cycled cell whose photon
// density grows linearly from zero meets relative changes of exactly 1/10
// and 1/20).  The quotient is kept out of line so that the compiler does
// not evaluate it on the common path.
template <typename S>
__device__ __noinline__ bool quotient_gt(S a, S b, double t)
{
    return a / b > t;
}

template <typename S>
__device__ __noinline__ bool quotient_lt(S a, S b, double t)
{
    return a / b < t;
}

template <typename S>
__device__ __forceinline__ bool ratio_gt(const S &a, const S &b, double t)
{
    const S tb = t * b;
    if constexpr (std::is_same<S, double>::value) {
        const long long ai = dbits(a), ti = dbits(tb);
        if (ai > ti + 8 && ai <= kInfBits) return true;
        if (ai < ti - 8) return false;
    } else {
        if (a > tb * (1.0 + 1e-15)) return true;
        if (a < tb * (1.0 - 1e-15)) return false;
    }
    return quotient_gt<S>(a, b, t);
}

template <typename S>
__device__ __forceinline__ bool ratio_lt(const S &a, const S &b, double t)
{
    const S tb = t * b;
    if constexpr (std::is_same<S, double>::value) {
        const long long ai = dbits(a), ti = dbits(tb);
        if (ai < ti - 8) return true;
        if (ai > ti + 8 && ai <= kInfBits) return false;
    } else {
        if (a < tb * (1.0 - 1e-15)) return true;
        if (a > tb * (1.0 + 1e-15)) return false;
    }
    return quotient_lt<S>(a, b, t);
}

// The change of a checked quantity from `o` to `n` against its 10% and 5%
// limits, relative to max(o, floor): in FP32 (the floats nearest to the two
// are within 2^-24, so 1e-5 around the limits is undecided by far), and
// there exactly as the rounded quotient decides.  An FP64 difference and two
// products per check before.
template <typename S>
__device__ __noinline__ bool change_gt(S n, S o, S floor_, double t)
{
    return ratio_gt(fabs(n - o), max0(o, floor_), t);
}
template <typename S>
__device__ __noinline__ bool change_lt(S n, S o, S floor_, double t)
{
    return ratio_lt(fabs(n - o), max0(o, floor_), t);
}
// (the fast path only notes what it cannot decide, and a broken limit)
template <typename S, class CTL>
__device__ __forceinline__ bool change_ok(const S &n, const S &o, const S &floor_, bool &small, CTL &ctl)
{
    const float of = dfm::near_float(val(o));
    const float d = fabsf(__fsub_rn(dfm::near_float(val(n)), of));
    const float den = fmaxf(of, dfm::near_float(val(floor_)));
    const bool ok = d < 0.099999f * den, bad = d > 0.100001f * den;
    const bool sm = d < 0.049999f * den, not_sm = d > 0.050001f * den;
    if constexpr (CTL::fast) {
        ctl.reject |= bad;
        ctl.odd |= !(ok || bad) || !(sm || not_sm);
        small = small && sm;
        return true;
    } else {
        if (!ok) {
            if (bad) return false;
            if (change_gt<S>(n, o, floor_, 0.1)) return false;
        }
        small = small && (sm || (!not_sm && change_lt<S>(n, o, floor_, 0.05)));
        return true;
    }
}
// |a| > t b for a first-order term a (b > 0)
template <typename S>
__device__ __noinline__ bool term_gt(S a, S b, double t)
{
    return ratio_gt(fabs(a), b, t);
}
template <typename S>
__device__ __noinline__ bool term_lt(S a, S b, double t)
{
    return ratio_lt(fabs(a), b, t);
}
// |a| <= 0.1 b, and with `small` also whether |a| < 0.05 b
template <typename S, class CTL>
__device__ __forceinline__ bool term_ok(const S &a, const S &b, CTL &ctl, bool *small = nullptr)
{
    const float d = fabsf(dfm::near_float(val(a))), den = dfm::near_float(val(b));
    const bool ok = d < 0.099999f * den, bad = d > 0.100001f * den;
    const bool sm = d < 0.049999f * den, not_sm = d > 0.050001f * den;
    if constexpr (CTL::fast) {
        ctl.reject |= bad;
        ctl.odd |= !(ok || bad) || (small && !(sm || not_sm));
        if (small) *small = *small && sm;
        return true;
    } else {
        if (!ok && (bad || term_gt<S>(a, b, 0.1))) return false;
        if (small) *small = *small && (sm || (!not_sm && term_lt<S>(a, b, 0.05)));
        return true;
    }
}

// Rates at one temperature level, by one thread or by a team of TS lanes
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void h_rates(const TLevel &L, double, int case_b, HRates &r, CTL &ctl)
{
    if constexpr (TS > 1) r = h_rates_team<TS, MIX>(L, case_b, ctl);
    else r = h_rates_serial<MIX>(L, case_b);
}
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void he_rates(const TLevel &L, double, int case_b, HeRates &r, CTL &ctl)
{
    if constexpr (TS > 1) r = he_rates_team<TS, MIX>(L, case_b, ctl);
    else r = he_rates_serial<MIX>(L, case_b);
}
// (only beta_HeII and alpha_HeIII; one thread)
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void he3_rates(const TLevel &L, double, int case_b, HeRates &r, CTL &ctl)
{
    const double2 t = he3_rates_serial<MIX>(L, case_b);
    r.beta_HeII = t.x;
    r.alpha_HeIII = t.y;
}

// What an attempt of a team makes of the rates at one temperature, each lane
// from its own function before the shuffles: an FP64 instruction takes a warp
// 64 cycles whatever its lanes hold, so the lanes' terms share one (each a
// fused multiply-add with a factor 1 or an addend 0 where a lane has none:
// the bits of the one-thread path).
// With the sums of photons_team about 24 of an attempt's 135 FP64
// instructions less: 128^3 with 16 bright sources, one lone cell's chain of
// 2448 attempts 19.4 -> 17.3 ms; 48^3 without the OTSA 10.9 -> 10.2 ms; 256^3
// 37.5 -> 34.4 ms.
// The densities n_HI, n_HeI, n_HeII, n_HeIII:
template <int TS, class CTL>
__device__ __forceinline__ void densities_team(double nH, double nHe, double xI, double yI, double y2, double y3,
                                               double &nHI, double &nHeI, double &nHeII, double &nHeIII)
{
    const unsigned m = team_mask_c<TS, CTL>();
    const int t = team_lane<TS>();
    const double n = t == 0 ? nH : nHe;
    if constexpr (TS >= 4) {
        const double d = rmul(n, t == 0 ? xI : t == 1 ? yI : t == 2 ? y2 : y3);
        nHI = team_get<TS>(m, d, 0);
        nHeI = team_get<TS>(m, d, 1);
        nHeII = team_get<TS>(m, d, 2);
        nHeIII = team_get<TS>(m, d, 3);
    } else {
        const double d = rmul(n, t == 0 ? xI : yI), e = rmul(nHe, t == 0 ? y2 : y3);
        nHI = team_get<TS>(m, d, 0);
        nHeI = team_get<TS>(m, d, 1);
        nHeII = team_get<TS>(m, e, 0);
        nHeIII = team_get<TS>(m, e, 1);
    }
}
// The cooling L and dL/dT of the sums (cooling_close):
template <int TS, class CTL>
__device__ __forceinline__ void cooling_close_team(double comp, double tg, double T, double ne, double Ls, double dLs,
                                                   double &L, double &dL)
{
    const unsigned m = team_mask_c<TS, CTL>();
    const bool l = team_lane<TS>() == 0;
    const double z = rmul(ne, rfma(comp, l ? radd(T, -tg) : 1.0, l ? Ls : dLs));
    L = team_get<TS>(m, z, 0);
    dL = team_get<TS>(m, z, 1);
}
// Hydrogen: beta, alpha, dC = n_H beta + f T dbeta/dT, dD = n_H alpha + f T
// dalpha/dT
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void h_terms_team(const TLevel &L, int case_b, double nH, double f, double &beta,
                                             double &alpha, double &dC, double &dD, CTL &ctl)
{
    const unsigned m = team_mask_c<TS, CTL>();
    RateVal v;
    rate_lane<MIX, 1>(case_b, team_lane<TS>() == 0 ? RF_BETA_HI : RF_ALPHA_HII, L, v, ctl);
    const double r = rate_f(v, ctl), d = rfma(f, rate_tdf(v, ctl), rmul(nH, r));
    beta = team_get<TS>(m, r, 0);
    alpha = team_get<TS>(m, r, 1);
    dC = team_get<TS>(m, d, 0);
    dD = team_get<TS>(m, d, 1);
}
// HeI and HeII: D1 = beta_HeI n_e + Gamma_1, P3 = y3 alpha_HeIII n_e, num1 =
// yI + h y2 alpha_HeII n_e, den1 = 1 + h D1, den2 = 1 + h ((beta_HeII +
// alpha_HeII) n_e + Gamma_2)
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void he_terms_team(const TLevel &L, int case_b, double y2, double y3, double yI, double ne,
                                              double gam1, double gam2, double h, double &D1, double &P3,
                                              double &num1, double &den1, double &den2, CTL &ctl)
{
    const unsigned m = team_mask_c<TS, CTL>();
    const int t = team_lane<TS>();
    RateVal v;
    rate_lane<MIX, 0>(case_b, RF_BETA_HEI + t, L, v, ctl);
    const double r = rate_f(v, ctl);
    if constexpr (TS >= 4) {   // lanes beta_HeI, beta_HeII, alpha_HeII, alpha_HeIII
        const double a2 = team_get<TS>(m, r, 2);
        const double u = rfma(t < 2 ? 1.0 : t == 2 ? y2 : y3, r, t == 1 ? a2 : 0.0);
        const double w = rfma(u, ne, t == 0 ? gam1 : t == 1 ? gam2 : 0.0);
        const double z = rfma(w, h, t == 2 ? yI : 1.0);
        D1 = team_get<TS>(m, w, 0);
        P3 = team_get<TS>(m, w, 3);
        den1 = team_get<TS>(m, z, 0);
        den2 = team_get<TS>(m, z, 1);
        num1 = team_get<TS>(m, z, 2);
    } else {   // beta_HeI, beta_HeII, then alpha_HeII, alpha_HeIII
        rate_lane<MIX, 0>(case_b, RF_BETA_HEI + 2 + t, L, v, ctl);
        const double a = rate_f(v, ctl), a2 = team_get<TS>(m, a, 0);
        const double w = rfma(radd(r, t == 0 ? 0.0 : a2), ne, t == 0 ? gam1 : gam2);
        const double z = rfma(w, h, 1.0);
        const double P = rmul(rmul(t == 0 ? y2 : y3, a), ne);
        D1 = team_get<TS>(m, w, 0);
        P3 = team_get<TS>(m, P, 1);
        den1 = team_get<TS>(m, z, 0);
        den2 = team_get<TS>(m, z, 1);
        num1 = team_get<TS>(m, rfma(P, h, yI), 0);
    }
}
// HeIII: C3 = y2 (beta_HeII n_e + Gamma_2), den3 = 1 + h alpha_HeIII n_e
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void he3_terms_team(const TLevel &L, int case_b, double y2, double ne, double gam2,
                                               double h, double &C3, double &den3, CTL &ctl)
{
    const unsigned m = team_mask_c<TS, CTL>();
    const bool b = team_lane<TS>() == 0;
    RateVal v;
    rate_lane<MIX, 0>(case_b, b ? RF_BETA_HEII : RF_ALPHA_HEIII, L, v, ctl);
    const double w = rfma(rate_f(v, ctl), ne, b ? gam2 : 0.0);
    const double z = rfma(w, b ? y2 : h, b ? 0.0 : 1.0);
    C3 = team_get<TS>(m, z, 0);
    den3 = team_get<TS>(m, z, 1);
}
// dual numbers, a team of eight: the level of the value, dT the tangent of T
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void h_rates(const TLevel &L, double dT, int case_b, HRatesT<Dual> &r, CTL &ctl)
{
    static_assert(TS == 8 && !MIX, "dual rates: teams of eight, FP64");
    r = h_rates_dual(L, dT, case_b, ctl);
}
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void he_rates(const TLevel &L, double dT, int case_b, HeRatesT<Dual> &r, CTL &ctl)
{
    r = he_rates_dual(L, dT, case_b, ctl);
}
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void he3_rates(const TLevel &L, double dT, int case_b, HeRatesT<Dual> &r, CTL &ctl)
{
    r = he_rates_dual(L, dT, case_b, ctl);
}

// The level of T = (T/mu') mu_j given 1/mu_j = md and 1/(T/mu') = iT as a
// pair (the temperatures of steps 3 and 4 enter their rates only through
// 1/T and ln T): 1/T = md iT in pair arithmetic; and the derivative of a
// dual T = Tmu1 / md.
template <class CTL>
__device__ __forceinline__ dfm::F2 inv_pair(double x, CTL &ctl)
{
    const bool in = (x > 0.0) && dfm::splittable(x);
    if constexpr (CTL::fast) {
        ctl.odd |= !in;
        return dfm::rcp2(dfm::split(x));
    } else {
        if (!in) return dfm::split_any(1.0 / x);
        return dfm::rcp2(dfm::split(x));
    }
}
template <class CTL>
__device__ __forceinline__ dfm::F2 md_pair(double md, CTL &ctl)
{
    if constexpr (CTL::fast) {
        ctl.odd |= !dfm::splittable(md);
        return dfm::split(md);
    } else {
        return dfm::split_any(md);
    }
}
template <class CTL>
__device__ __forceinline__ double level_mu(const Dual &md, dfm::F2 iT, const Dual &Tmu1, TLevel &L, CTL &ctl)
{
    t_level_inv(dfm::norm(dfm::mulu(md_pair(md.v, ctl), iT)), L, ctl);
    return cdiv(Tmu1, md, ctl).d;
}
template <class CTL>
__device__ __forceinline__ double level_mu(double md, dfm::F2 iT, double, TLevel &L, CTL &ctl)
{
    t_level_inv(dfm::norm(dfm::mulu(md_pair(md, ctl), iT)), L, ctl);
    return 0.0;
}

// (alpha^A_j - alpha^B_j) n_j n_e of HII, HeII, HeIII at temperature T
// (Eq. (cool_N_cr)); out of line: it only runs without the OTSA, and
// inlined its two rate tables would raise the register count of every
// kernel
template <bool MIX>
static __device__ __noinline__ void recomb_rates(double T, double nHII, double nHeII, double nHeIII, double ne,
                                                 double *rj)
{
    double aA[3], aB[3];
    TLevel L;
    dfm::Exact e;
    t_level(T, L, e);
    Rates t;
    rates_serial<MIX>(L, 0, kNeedRec, 0u, t);
    recomb_alphas(t, aA);
    rates_serial<MIX>(L, 1, kNeedRec, 0u, t);
    recomb_alphas(t, aB);
    rj[0] = (aA[0] - aB[0]) * nHII * ne;
    rj[1] = (aA[1] - aB[1]) * nHeII * ne;
    rj[2] = (aA[2] - aB[2]) * nHeIII * ne;
}

// ... by a team: lane j species j, both cases; the same operations
template <int TS, bool MIX, class CTL>
__device__ __forceinline__ void recomb_rates_team(double T, double nHII, double nHeII, double nHeIII, double ne,
                                                  double *rj, CTL &ctl)
{
    const unsigned m = team_mask_c<TS, CTL>();
    TLevel L;
    t_level(T, L, ctl);
#pragma unroll
    for (int j0 = 0; j0 < 3; j0 += TS) {
        const int j = j0 + team_lane<TS>();
        const int k = j == 0 ? RF_ALPHA_HII : j == 1 ? RF_ALPHA_HEII : RF_ALPHA_HEIII;
        RateVal a, b;
        rate_lane<MIX, 0>(0, k, L, a, ctl);
        rate_lane<MIX, 0>(1, k, L, b, ctl);
        const double r = (rate_f(a, ctl) - rate_f(b, ctl)) * (j == 0 ? nHII : j == 1 ? nHeII : nHeIII) * ne;
#pragma unroll
        for (int i = 0; i < TS; ++i)
            if (j0 + i < 3) rj[j0 + i] = team_get<TS>(m, r, i);
    }
}

// Photon update of one group, Eq. (SIE photons): N_i' = (N_i + h C_i)/(1 + h D_i)
// (C_i = 0 under the OTSA; smoothed RT adds the rate Ndot_i), F_i scaled by
// 1/(1 + h D_i), D_i = c_r sum_j sigma^N_ij n_j with the backward absorber
// densities; with the group's 10% and 5% checks on N_i and the factors of its
// terms of the photo-ionisation rates N_i' c_r sigma^N_ij and of the
// photoheating N_i' q, q = c_r sum_j n_j (egy_i sigma^E_ij - eps_j sigma^N_ij).
// Products and sums are rounded as written; the terms enter their sums over
// the groups by fused multiply-adds (with c_r in the coefficients 13 FP64
// instructions of 187 less in the one-thread pass, 256^3: 17.2 -> 16.5 ms, and 5
// of 110 in a team's, 256^3: 34.4 -> 33.4 ms).
template <typename S>
struct PhotonTerms {
    S Nn, Fs, Fb, q;
    bool ok, small;
};

template <bool MIX, bool SM, typename S, class CTL>
__device__ __forceinline__ void photon_group(const ThermoParams &p, int i, const S &N, const S &Fs, const S &Nd,
                                             const S &Fb, const S &Crec, const S &nHI, const S &nHeI,
                                             const S &nHeII, double h, PhotonTerms<S> &o, CTL &ctl)
{
    S inv;
    if constexpr (MIX) {
        // absorption coefficient in FP32; the update itself in FP64, since
        // a cell may take thousands of sub-steps and FP32 roundings of N
        // would accumulate past the stated 1e-4 (doubles narrowed and the
        // float widened through integer operations, not FP64-pipe
        // conversions)
        const float Df = __fadd_rn(__fadd_rn(__fmul_rn(narrow(p.crs[i][0]), narrow(nHI)),
                                             __fmul_rn(narrow(p.crs[i][1]), narrow(nHeI))),
                                   __fmul_rn(narrow(p.crs[i][2]), narrow(nHeII)));
        inv = crcp(rfma(h, dfm::widen(Df), 1.0), ctl);
    } else {
        const S D = rfma(p.crs[i][2], nHeII, rfma(p.crs[i][1], nHeI, rmul(nHI, p.crs[i][0])));
        inv = crcp(rfma(h, D, S(1.0)), ctl);
    }
    // smoothed RT: N + h Ndot rounded step by step, so a cell growing
    // linearly from zero meets its relative changes 1/k exactly
    S Nn;
    if constexpr (SM) Nn = rmul(radd(N, rmul(Nd + Crec, h)), inv);
    else if (p.emit) Nn = rmul(rfma(h, Crec, N), inv);
    else Nn = rmul(N, inv);
    o.small = true;
    o.ok = change_ok(Nn, N, S(kFloorN), o.small, ctl);
    o.Nn = Nn;
    o.Fs = rmul(Fs, inv);
    if constexpr (SM) o.Fb = rmul(radd(Fb, S(h)), inv);
    o.q = rfma(p.hq[i][2], nHeII, rfma(p.hq[i][1], nHeI, rmul(nHI, p.hq[i][0])));
}

// The photon stage of an attempt by a team of PT lanes (each with its own
// groups), filling the lanes' new N_i and flux scales and, in every lane, the
// photo-ionisation rates gam_j and the photoheating, each summed over the
// groups in one lane (a team of two: two in each); false when a group
// breaks the 10% rule.  The recombination photons C_i (without the OTSA) come
// from cc.rj.
template <int G, int PT, bool MIX, bool SM, class CTL>
__device__ __forceinline__ bool photons_team(const ThermoParams &p, const CellState<lane_groups<>(G, PT)> &s,
                                             const CoolCache<double> &cc, double nHI, double nHeI, double nHeII,
                                             double h, CellState<lane_groups<>(G, PT)> &o, double &gam0, double &gam1,
                                             double &gam2, double &heat, bool &sm, CTL &ctl)
{
    constexpr int NG = lane_groups<>(G, PT);
    const unsigned mask = team_mask_c<PT, CTL>();
    const int t = team_lane<PT>();
    bool ok = true, small = true;
    PhotonTerms<double> pt[NG];
#pragma unroll
    for (int r = 0; r < NG; ++r) {
        const bool mine = r * PT + t < G;
        const int gi = mine ? r * PT + t : 0;
        double Crec = 0.0;
        if (p.emit) {
#pragma unroll
            for (int j = 0; j < 3; ++j)
                if (mine && p.rec_g[j] == gi) Crec += cc.rj[j];
        }
        // (a lane without a group here runs group 0 on zeros, which changes nothing)
        photon_group<MIX, SM>(p, gi, s.N[r], s.Fs[r], s.Nd[r], s.Fb[r], Crec, nHI, nHeI, nHeII, h, pt[r], ctl);
        ok = ok && (pt[r].ok || !mine);
        small = small && (pt[r].small || !mine);
        o.N[r] = pt[r].Nn;
        o.Fs[r] = pt[r].Fs;
        if constexpr (SM) {
            o.Fb[r] = pt[r].Fb;
            o.Nd[r] = s.Nd[r];
        }
    }
    if constexpr (CTL::fast) {   // (decided for the whole team at the end)
        sm = sm && small;
    } else {
        ok = __all_sync(mask, ok);
        sm = sm && (__all_sync(mask, small) != 0);
    }
    constexpr int NS = 4 / PT;   // sums per lane: t NS, t NS + 1, ... of gam0, gam1, gam2, heat
    double sum[NS];
#pragma unroll
    for (int i = 0; i < G; ++i) {
        const double Nn = team_get<PT>(mask, pt[i / PT].Nn, i % PT), q = team_get<PT>(mask, pt[i / PT].q, i % PT);
#pragma unroll
        for (int k = 0; k < NS; ++k) {
            const int j = t * NS + k;
            const double w = j == 3 ? q : p.crs[i][j < 3 ? j : 2];
            sum[k] = i == 0 ? rmul(w, Nn) : rfma(w, Nn, sum[k]);
        }
    }
    gam0 = team_get<PT>(mask, sum[0], 0);
    gam1 = team_get<PT>(mask, sum[1 % NS], 1 / NS);
    gam2 = team_get<PT>(mask, sum[2 % NS], 2 / NS);
    heat = team_get<PT>(mask, sum[3 % NS], 3 / NS);
    return ok;
}

template <int G, bool MIX, bool SM, typename S, class CTL>
__device__ __forceinline__ bool photons_serial(const ThermoParams &p, const CellState<G, S> &s,
                                               const CoolCache<S> &cc, const S &nHI, const S &nHeI, const S &nHeII,
                                               double h, CellState<G, S> &o, S &gam0, S &gam1, S &gam2, S &heat,
                                               bool &sm, CTL &ctl)
{
    PhotonTerms<S> pt;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        S Crec = 0.0;
        if (p.emit) {
#pragma unroll
            for (int j = 0; j < 3; ++j)
                if (p.rec_g[j] == i) Crec += cc.rj[j];
        }
        photon_group<MIX, SM>(p, i, s.N[i], s.Fs[i], s.Nd[i], s.Fb[i], Crec, nHI, nHeI, nHeII, h, pt, ctl);
        if (!pt.ok) return false;
        sm = sm && pt.small;
        o.N[i] = pt.Nn;
        o.Fs[i] = pt.Fs;
        if constexpr (SM) {
            o.Fb[i] = pt.Fb;
            o.Nd[i] = s.Nd[i];
        }
        if (i == 0) {
            gam0 = rmul(pt.Nn, p.crs[i][0]);
            gam1 = rmul(pt.Nn, p.crs[i][1]);
            gam2 = rmul(pt.Nn, p.crs[i][2]);
            heat = rmul(pt.Nn, pt.q);
        } else {
            gam0 = rfma(p.crs[i][0], pt.Nn, gam0);
            gam1 = rfma(p.crs[i][1], pt.Nn, gam1);
            gam2 = rfma(p.crs[i][2], pt.Nn, gam2);
            heat = rfma(pt.q, pt.Nn, heat);
        }
    }
    return true;
}

// One thermo_step over h.  Returns true and fills `o` when the 10% rule
// holds; `small` then tells whether every checked change stayed below 5%.
// The checks |dX| / den > 0.1 go through ratio_gt / ratio_lt (a division
// only near the threshold).
// MIX (RT_MIXED32): the rates' softplus corrections and exponentials and
// the absorption coefficients in FP32 (rates.cuh, rate_softplus, rate_val); the
// photon, T/mu, x_HII and helium updates and 1 - x in FP64.
//
// S is double, or Dual for the adjoint's differentiated recomputation
// (values bit-identical to the double path; MIX only with double).
// TS: 1, one thread, or 2 or 4, a team of lanes that hold the same cell,
// share its rate functions and each update their own photon groups; the same
// operations in the same order, so the same bits.  Dual: teams of eight lanes
// with the same values and a tangent each; they share the rate functions.
// CTL: Exact, or Fast (teams, evolving T, with helium): no branches but that of
// the recombination photons; the result counts unless ctl.odd or ctl.reject is
// set in a lane of the team.
template <int G, int TS, bool MIX, typename S, bool SM, class CTL>
__device__ __forceinline__ bool attempt(const ThermoParams &p, const S &nH, const CellState<lane_groups<S>(G, TS), S> &s,
                                        double h, const IsoRates<S> &iso, CoolCache<S> &cc,
                                        CellState<lane_groups<S>(G, TS), S> &o, bool &small, CTL &ctl)
{
    constexpr bool fast = CTL::fast;
    const bool isothermal = !fast && p.isothermal, helium = fast || p.helium;
    constexpr bool dual = !std::is_same<S, double>::value;
    static_assert(dual ? TS == 8 : TS == 1 || TS == 2 || TS == 4, "team sizes");
    static_assert(!MIX || sizeof(S) == sizeof(double), "the mixed path is not differentiated");
    const S nHe = iso.nHe;
    const S x = s.x, y2 = s.y2, y3 = s.y3;
    const S q0 = he_electrons(y2, y3);
    const S xI = radd(S(1.0), -x);
    const S nHII = rmul(nH, x);
    const S yI = radd(radd(S(1.0), -y2), -y3);
    S nHI, nHeI, nHeII, nHeIII;
    constexpr bool team = TS > 1 && !dual;
    if constexpr (team) {
        densities_team<TS, CTL>(nH, nHe, xI, yI, y2, y3, nHI, nHeI, nHeII, nHeIII);
    } else {
        nHI = rmul(nH, xI);
        nHeI = rmul(nHe, yI);
        nHeII = rmul(nHe, y2);
        nHeIII = rmul(nHe, y3);
    }
    const S ne = ne_of(nHII, q0, nHe);
    const S mhe = md_he(p, q0);
    bool sm = true;
    S gam0 = 0.0, gam1 = 0.0, gam2 = 0.0, heat = 0.0;

    // cooling at T(t) and the state at t (step 2 below), first: it depends on
    // nothing this sub-step computes, so its rate functions can overlap the
    // photon update; kept over rejected attempts
    // recombination photons without the OTSA, Eq. (cool_N_cr), at T(t) with
    // the backward abundances; group i gains C_i = sum_j [rec_g[j] == i] rj[j]
    if constexpr (!dual) {   // (the adjoint needs the OTSA)
        if (p.emit && (fast || !cc.rvalid)) {
            if constexpr (TS > 1) recomb_rates_team<TS, MIX>(s.T, nHII, nHeII, nHeIII, ne, cc.rj, ctl);
            else recomb_rates<MIX>(s.T, nHII, nHeII, nHeIII, ne, cc.rj);
            cc.rvalid = true;
        }
    }

    if (fast || (!isothermal && !cc.valid)) {
        if constexpr (dual) {
            cooling_dual(p.case_b, p.comp, p.tg, helium, s.T, ne, nHI, nHII, nHeI, nHeII, nHeIII, cc.L, cc.dL,
                         ctl);
        } else if constexpr (TS > 1) {
            const double2 c = cooling_sums_team<TS, MIX>(p.case_b, helium, s.T, nHI, nHII, nHeI, nHeII, nHeIII, ctl);
            cooling_close_team<TS, CTL>(p.comp, p.tg, s.T, ne, c.x, c.y, cc.L, cc.dL);
        } else {
            cooling_serial<MIX>(p.case_b, p.comp, p.tg, helium, s.T, ne, nHI, nHII, nHeI, nHeII, nHeIII, cc.L,
                                cc.dL);
        }
        cc.valid = true;
    }

    // 1. photons: group i's update depends on no other group, so the lanes of
    // a team take a group each; one thread loops over the groups; both call
    // photon_group and sum the groups' terms in the same order (rounded as
    // written), so they give the same bits
    {
        bool ok;
        if constexpr (TS > 1 && !dual)
            ok = photons_team<G, TS, MIX, SM>(p, s, cc, nHI, nHeI, nHeII, h, o, gam0, gam1, gam2, heat, sm, ctl);
        else ok = photons_serial<G, MIX, SM>(p, s, cc, nHI, nHeI, nHeII, h, o, gam0, gam1, gam2, heat, sm, ctl);
        if (!ok) return false;
    }

    // 2. temperature: T/mu + K h (Lambda) / (1 + mu (dL/dT) K h), Lambda =
    // heating - cooling, d Lambda/d(T/mu) = -mu dL/dT
    S mden, mu, Tmu1 = 0.0;
    if (!isothermal) {
        mden = mu_den(p, x, mhe);
        mu = crcp(mden, ctl);
        const S Tmu = rmul(s.T, mden);
        const S Kh = rmul(iso.K, h);
        const S num = rmul(radd(heat, -cc.L), Kh);
        const S dT = cdiv(num, rfma(rmul(mu, cc.dL), Kh, S(1.0)), ctl);
        Tmu1 = radd(Tmu, dT);
        if (!term_ok(num, Tmu, ctl)) return false;
        if (!term_ok(dT, Tmu, ctl, &sm)) return false;
    }
    // 1/(T/mu') as a pair, for the temperatures (T/mu') mu_j of steps 3 and 4
    const dfm::F2 iT = isothermal ? dfm::F2{0.0f, 0.0f} : inv_pair(val(Tmu1), ctl);

    // 3. hydrogen: C = beta n_e + Gamma, D = alpha n_e and their derivatives
    S beta, alpha, dC, dD;
    // d/dx at constant T/mu' through T = (T/mu') mu: - n_e (T/mu') mu^2 X d/dT =
    // - n_e mu X (T d/dT)
    const S f = isothermal ? S(0.0) : rmul(rmul(ne, mu), -p.X);
    if (team && !isothermal) {
        if constexpr (team) {
            TLevel L;
            level_mu(mden, iT, Tmu1, L, ctl);
            h_terms_team<TS, MIX>(L, p.case_b, nH, f, beta, alpha, dC, dD, ctl);
        }
    } else {
        HRatesT<S> hr;
        if (isothermal) {
            hr = iso.h;
        } else {
            TLevel L;
            const double dT = level_mu(mden, iT, Tmu1, L, ctl);
            h_rates<TS, MIX>(L, dT, p.case_b, hr, ctl);
        }
        beta = hr.beta;
        alpha = hr.alpha;
        dC = rmul(nH, hr.beta);
        dD = rmul(nH, hr.alpha);
        if (!isothermal) {
            dC = rfma(f, hr.tbeta, dC);
            dD = rfma(f, hr.talpha, dD);
        }
    }
    const S C = rfma(beta, ne, gam0);
    const S CD = rfma(alpha, ne, C);   // C + D
    // h (C - x (C + D)) and 1 - h J, J = dC - C - D - x (dC + dD)
    S hx, den;
    if constexpr (team) {
        const unsigned m = team_mask_c<TS, CTL>();
        const bool j = team_lane<TS>() == 0;
        const double v = rfma(-x, j ? radd(dC, dD) : CD, j ? radd(dC, -CD) : C);
        const double z = rfma(j ? -v : v, h, j ? 1.0 : 0.0);
        den = team_get<TS>(m, z, 0);
        hx = team_get<TS>(m, z, 1);
    } else {
        const S J = rfma(-x, radd(dC, dD), radd(dC, -CD));
        hx = rmul(rfma(-x, CD, C), h);
        den = rfma(-J, S(h), S(1.0));
    }
    S x1 = radd(x, cdiv(hx, den, ctl));
    x1 = min0(max0(x1, kXMin), 1.0);
    if (!change_ok(x1, x, S(kXMin), sm, ctl)) return false;
    if (!term_ok(hx, max0(x, kXMin), ctl)) return false;

    // 4. helium
    S y2n = y2, y3n = y3;
    const S nHII1 = rmul(x1, nH);
    if (helium) {
        const S ne2 = ne_of(nHII1, q0, nHe);
        const S hs(h);
        S D1, P3, num1, den1, den2;
        if (team && !isothermal) {
            if constexpr (team) {
                TLevel L;
                level_mu(mu_den(p, x1, mhe), iT, Tmu1, L, ctl);
                he_terms_team<TS, MIX>(L, p.case_b, y2, y3, yI, ne2, gam1, gam2, h, D1, P3, num1, den1, den2, ctl);
            }
        } else {
            HeRatesT<S> r2;
            if (isothermal) {
                r2 = iso.he;
            } else {
                TLevel L;
                const double dT = level_mu(mu_den(p, x1, mhe), iT, Tmu1, L, ctl);
                he_rates<TS, MIX>(L, dT, p.case_b, r2, ctl);
            }
            D1 = rfma(r2.beta_HeI, ne2, gam1);
            P3 = rmul(rmul(y3, r2.alpha_HeIII), ne2);
            num1 = rfma(rmul(rmul(y2, r2.alpha_HeII), ne2), hs, yI);
            den1 = rfma(D1, hs, S(1.0));
            den2 = rfma(rfma(radd(r2.beta_HeII, r2.alpha_HeII), ne2, gam2), hs, S(1.0));
        }
        const S yI1 = cdiv(num1, den1, ctl);
        const S C2 = rfma(yI1, D1, P3);
        y2n = cdiv(rfma(C2, hs, y2), den2, ctl);
        const S q1 = he_electrons(y2n, y3);
        const S ne3 = ne_of(nHII1, q1, nHe);
        S C3, den3;
        if (team && !isothermal) {
            if constexpr (team) {
                TLevel L;
                level_mu(mu_den(p, x1, md_he(p, q1)), iT, Tmu1, L, ctl);
                he3_terms_team<TS, MIX>(L, p.case_b, y2n, ne3, gam2, h, C3, den3, ctl);
            }
        } else {
            HeRatesT<S> r3;
            if (isothermal) {
                r3 = iso.he;
            } else {
                TLevel L;
                const double dT = level_mu(mu_den(p, x1, md_he(p, q1)), iT, Tmu1, L, ctl);
                he3_rates<TS, MIX>(L, dT, p.case_b, r3, ctl);
            }
            C3 = rmul(y2n, rfma(r3.beta_HeII, ne3, gam2));
            den3 = rfma(rmul(r3.alpha_HeIII, ne3), hs, S(1.0));
        }
        y3n = cdiv(rfma(C3, hs, y3), den3, ctl);
        // conservation: lower the largest fraction (HeI largest: no change);
        // (the fractions are positive or zero: compared by their bits)
        const long long bI = dbits(val(yI1)), b2 = dbits(val(y2n)), b3 = dbits(val(y3n));
        const bool two = b2 >= bI && b2 >= b3, three = !two && b3 >= bI;
        const S rest = radd(radd(S(1.0), -yI1), two ? -y3n : -y2n);
        y2n = two ? rest : y2n;
        y3n = three ? rest : y3n;
        y2n = min0(max0(y2n, 0.0), 1.0);
        y3n = min0(max0(y3n, 0.0), 1.0);
    }
    const S q2 = he_electrons(y2n, y3n);
    if (!change_ok(ne_of(nHII1, q2, nHe), ne, iso.nef, sm, ctl)) return false;
    const S Tf = isothermal ? s.T : cdiv(Tmu1, mu_den(p, x1, md_he(p, q2)), ctl);
    o.x = x1;
    o.y2 = y2n;
    o.y3 = y3n;
    o.T = max0(Tf, kTFloor);
    small = sm;
    return true;
}

// One attempt of the sub-cycling loop; returns true when the cell is done.
// Teams of two and eight: called by whole warps; `have`: the lane's team has a
// cell.
template <int G, int TS, bool MIX, typename S = double, bool SM = false>
__device__ __forceinline__ bool subcycle_once(const ThermoParams &p, const S &nH,
                                              CellState<lane_groups<S>(G, TS), S> &st, double &t_left, double &dt_tc,
                                              int &att, const IsoRates<S> &iso, CoolCache<S> &cc, bool have = true)
{
    // t_left, dt_tc > 0: compared through their bits
    double h = (dbits(dt_tc) < dbits(t_left)) ? dt_tc : t_left;
    att += have;
    CellState<lane_groups<S>(G, TS), S> o;
    bool small = false, ok = false, decided = false;
    if constexpr (TS > 1) {
        // (a retry evaluates the cooling again, to the same bits: beside teams
        // that need theirs it takes no longer, and the warp stays together)
        if (!p.isothermal && p.helium) {
            dfm::Fast f;
            attempt<G, TS, MIX, S, SM>(p, nH, st, h, iso, cc, o, small, f);
            const unsigned m = team_mask<TS>(), all = team_mask_c<TS, dfm::Fast>();
            const bool odd = (__ballot_sync(all, f.odd) & m) != 0, reject = (__ballot_sync(all, f.reject) & m) != 0;
            small = (__ballot_sync(all, !small) & m) == 0;
            // (a broken limit rejects whatever else was odd, but an odd value may itself have broken it)
            decided = !odd;
            ok = decided && !reject;
        }
    }
    if (!have) return true;
    if (!decided) {
        // (nothing of an undecided fast attempt is kept for the exact one)
        if constexpr (TS > 1)
            if (!p.isothermal && p.helium) cc.valid = cc.rvalid = false;
        dfm::Exact e;
        small = false;
        ok = attempt<G, TS, MIX, S, SM>(p, nH, st, h, iso, cc, o, small, e);
    }
    if (ok) {
        st = o;
        cc.valid = false;
        cc.rvalid = false;
        t_left = (dbits(h) == dbits(t_left)) ? 0.0 : t_left - h;
        dt_tc = small ? twice(h) : h;
    } else {
        dt_tc = half(h);
    }
    return dbits(t_left) <= 0;
}

}  // namespace thermo_detail
}  // namespace rtgb
