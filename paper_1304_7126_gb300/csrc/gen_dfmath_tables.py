"""Writes dfmath_tables.h: the tables and split constants of the
double-float exp, log and softplus in dfmath.cuh, each value split into a pair of
floats (hi = the value rounded to a float, lo = the rest rounded to a
float) from a 60-digit mpmath evaluation.  Run from this folder:
    python gen_dfmath_tables.py > dfmath_tables.h
"""
import math

import mpmath
import numpy as np

mpmath.mp.dps = 60


def f32(v):
    return float(np.float32(float(v)))


def pair(v):
    hi = f32(v)
    lo = f32(mpmath.mpf(v) - mpmath.mpf(hi))
    return hi, lo


def round_bits(v, bits):
    """v rounded to `bits` significant bits (exact in a float)."""
    m, e = math.frexp(float(v))
    return math.ldexp(round(m * 2 ** bits) / 2 ** bits, e)


def lit(x):
    return "%sf" % float(x).hex() if x != 0.0 else "0.0f"


def main():
    ln2 = mpmath.log(2)
    out = ["// Generated by gen_dfmath_tables.py; do not edit.", "#pragma once", ""]
    # exp: k = rint(x 64 / ln2), r = x - k ln2/64 with ln2/64 = L1 + L2 + L3;
    # L1 has 7 significant bits so that k L1 is exact for |k| < 2^17
    L = ln2 / 64
    L1 = round_bits(L, 7)
    L2 = f32(L - mpmath.mpf(L1))
    L3 = f32(L - mpmath.mpf(L1) - mpmath.mpf(L2))
    out.append("constexpr float kDfInvL = %s;   // 64 / ln 2" % lit(f32(64 / ln2)))
    out.append("constexpr float kDfL1 = %s;   // ln2/64 = L1 + L2 + L3, L1 7 bits" % lit(L1))
    out.append("constexpr float kDfL2 = %s;" % lit(L2))
    out.append("constexpr float kDfL3 = %s;" % lit(L3))
    # log: e ln2 with ln2 = N1 + N2 + N3, N1 13 bits so that e N1 is exact for |e| < 2^11
    N1 = round_bits(ln2, 13)
    N2 = f32(ln2 - mpmath.mpf(N1))
    N3 = f32(ln2 - mpmath.mpf(N1) - mpmath.mpf(N2))
    out.append("constexpr float kDfLn2A = %s;   // ln 2 = A + B + C, A 13 bits" % lit(N1))
    out.append("constexpr float kDfLn2B = %s;" % lit(N2))
    out.append("constexpr float kDfLn2C = %s;" % lit(N3))
    third = pair(mpmath.mpf(1) / 3)
    out.append("constexpr float kDfThirdHi = %s, kDfThirdLo = %s;   // 1/3" % (lit(third[0]), lit(third[1])))
    out.append("")
    out.append("// 2^(j/64), j = 0..63: {hi, lo}")
    out.append("static __device__ const float2 kDfExp2Tab[64] = {")
    rows = []
    for j in range(64):
        hi, lo = pair(mpmath.power(2, mpmath.mpf(j) / 64))
        rows.append("    {%s, %s}" % (lit(hi), lit(lo)))
    out.append(",\n".join(rows))
    out.append("};")
    out.append("")
    out.append("// F_j = 1 + j/128, j = 0..128: {ln F hi, ln F lo, 1/F hi, 1/F lo}")
    out.append("static __device__ const float4 kDfLogTab[129] = {")
    rows = []
    for j in range(129):
        F = 1 + mpmath.mpf(j) / 128
        lh, ll = pair(mpmath.log(F))
        ih, il = pair(1 / F)
        rows.append("    {%s, %s, %s, %s}" % (lit(lh), lit(ll), lit(ih), lit(il)))
    out.append(",\n".join(rows))
    out.append("};")
    out.append("")
    # softplus(z) = ln(1 + e^z) on [SP_LO, SP_HI): on each interval of width
    # SP_W the polynomial of degree SP_DEG in t = z - (interval middle) that
    # interpolates softplus at the Chebyshev points of the interval
    out.append("// ln(1 + e^z) on [%d, %d): interval k = [%d + k/%d, %d + (k+1)/%d), coefficients"
               % (SP_LO, SP_HI, SP_LO, SP_PER, SP_LO, SP_PER))
    out.append("// c_0..c_%d of the interpolating polynomial in t = z - (the interval's middle),"
               % SP_DEG)
    out.append("// at the Chebyshev points of the interval: {hi, lo}")
    out.append("constexpr int kDfSpLo = %d, kDfSpPer = %d, kDfSpN = %d, kDfSpDeg = %d;"
               % (SP_LO, SP_PER, SP_N, SP_DEG))
    out.append("static __device__ const __align__(16) float2 kDfSoftplusTab[%d][%d] = {" % (SP_N, SP_DEG + 1))
    rows = []
    for k in range(SP_N):
        coef = softplus_coefficients(k)
        rows.append("    {" + ", ".join("{%s, %s}" % (lit(a), lit(b)) for a, b in (pair(c) for c in coef)) + "}")
    out.append(",\n".join(rows))
    out.append("};")
    print("\n".join(out))


SP_LO, SP_HI, SP_PER, SP_DEG = -16, 16, 32, 7
SP_N = (SP_HI - SP_LO) * SP_PER


def softplus(z):
    return mpmath.log1p(mpmath.exp(z))


def softplus_coefficients(k):
    """Monomial coefficients in t of the degree-SP_DEG polynomial through
    softplus at the Chebyshev points of interval k."""
    h = mpmath.mpf(1) / (2 * SP_PER)
    mid = SP_LO + (mpmath.mpf(k) + mpmath.mpf(1) / 2) / SP_PER
    n = SP_DEG + 1
    ts = [h * mpmath.cos((2 * i + 1) * mpmath.pi / (2 * n)) for i in range(n)]
    A = mpmath.matrix([[t ** j for j in range(n)] for t in ts])
    b = mpmath.matrix([softplus(mid + t) for t in ts])
    c = mpmath.lu_solve(A, b)
    return [c[j] for j in range(n)]


if __name__ == "__main__":
    main()
