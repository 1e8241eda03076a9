#!/usr/bin/env python3
"""Writes phi_table.h: piecewise polynomials of the two functions of z = delta / sigma
that the FP64 pair arithmetic needs (pair_math64.cuh),
  F(z) = phi(z) / Phi(z)   and   G(z) = log Phi(z),
phi and Phi the standard normal density and distribution function, on the
nodes c = i / 64, i = 0 .. 640 (z up to 10): degree 7 in t = z - c, |t| <= 1/128,
each the polynomial that interpolates the function at the 8 Chebyshev points
of its interval (computed with 60 digits).  The degree and the split of the
coefficients keep the relative error of both functions near FP64's rounding up
to z = 10, where they are 1e-22: a term of degree k is at most (z t)^k / k! of
the value, so the FP32 rounding of those of degree 5 and up stays below 4e-16
of it at z = 8 and 1.1e-15 at z = 10.  A node is 14 words of 64 bits, low half first:
  F's coefficients of t^4, t^3, t^2, t, 1 and G's of 1 and of t^4, t^3, t^2, t
  in FP64; in FP32 {F's of t^7, t^6}, {F's of t^5, G's of t^5}, {G's of t^7,
  t^6}; an unused word (a row is then a whole number of 16-byte loads).

Usage: python gen_phi_table.py > phi_table.h
"""
import struct

from mpmath import cos, erfc, exp, log, mp, mpf, nint, pi, sqrt

mp.dps = 60
PER_UNIT, NODES, DEG = 64, 641, 7
HALF = mpf(1) / (2 * PER_UNIT)


def cdf(z):
    return erfc(-z / sqrt(2)) / 2


def f(z):
    return exp(-z * z / 2) / sqrt(2 * pi) / cdf(z)


def g(z):
    return log(cdf(z)) if z < 1 else log(1 - erfc(z / sqrt(2)) / 2)


CHEB = [HALF * cos((2 * k + 1) * pi / (2 * (DEG + 1))) for k in range(DEG + 1)]


def fit(fn, c):
    """Monomial coefficients (in t) of the interpolant at the Chebyshev points: Newton's divided differences, expanded."""
    d = [fn(c + t) for t in CHEB]
    for k in range(1, DEG + 1):
        for j in range(DEG, k - 1, -1):
            d[j] = (d[j] - d[j - 1]) / (CHEB[j] - CHEB[j - k])
    poly = [d[DEG]]
    for k in range(DEG - 1, -1, -1):
        shifted = [mpf(0)] + poly
        poly = [a - CHEB[k] * b for a, b in zip(shifted, poly + [mpf(0)])]
        poly[0] += d[k]
    return poly


def f64(x):
    return struct.unpack("<Q", struct.pack("<d", float(x)))[0]


def f32(lo, hi):
    return struct.unpack("<Q", struct.pack("<ff", float(lo), float(hi)))[0]


def main():
    worst = [mpf(0), mpf(0)]
    rows = []
    for i in range(NODES):
        c = mpf(i) / PER_UNIT
        co = []
        for q, fn in enumerate((f, g)):
            p = fit(fn, c)
            for u in (-1, mpf(-7) / 10, mpf(-1) / 4, mpf(1) / 3, mpf(8) / 10, 1):
                t = u * HALF
                v = sum(a * t ** k for k, a in enumerate(p))
                worst[q] = max(worst[q], abs(v / fn(c + t) - 1))
            co.append(p)
        a, b = co
        rows.append([f64(v) for v in (a[4], a[3], a[2], a[1], a[0], b[0], b[4], b[3], b[2], b[1])] +
                    [f32(a[7], a[6]), f32(a[5], b[5]), f32(b[7], b[6]), 0])
    print("// Generated by gen_phi_table.py -- do not edit.")
    print("// Node i, t = z - i/64: F = phi/Phi and G = log Phi as degree-7 polynomials (layout: see the generator);")
    print("// largest relative error before the coefficients' rounding: F %.1e, G %.1e." % (worst[0], worst[1]))
    print("#pragma once")
    print("constexpr int kPhiPerUnit = %d, kPhiNodes = %d, kPhiDeg = %d, kPhiRow = 14;" % (PER_UNIT, NODES, DEG))
    # pairs of words, so that the type carries the alignment of 16-byte loads
    print("__device__ const ulonglong2 g_phi_table[kPhiNodes * kPhiRow / 2] = {")
    for r in rows:
        print(",".join("{0x%016xull,0x%016xull}" % (r[k], r[k + 1]) for k in range(0, len(r), 2)) + ",")
    print("};")


if __name__ == "__main__":
    main()
