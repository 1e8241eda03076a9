#!/usr/bin/env python3
"""Writes phi_table.h: piecewise polynomials of the two functions of z = delta / sigma
that the FP64 pair arithmetic needs (pair_math64.cuh),
  F(z) = phi(z) / Phi(z)   and   G(z) = log Phi(z),
phi and Phi the standard normal density and distribution function, on the
nodes c = i / 64, i = 0 .. 608 (z up to 9.5): degree 5 in t = z - c, |t| <= 1/128,
each the polynomial that interpolates the function at the 6 Chebyshev points
of its interval (computed with 40 digits).  A node is 10 words of 64 bits, low
half first:
  F's coefficients of t^3, t^2, t, 1 and G's of t^3, t^2, t in FP64, G's
  constant as an integer in units of 2^-52, {F's of t^5, F's of t^4} and
  {G's of t^5, G's of t^4} in FP32 (t^4 <= 3.7e-9: their rounding is below
  1e-16 of the value).

Usage: python gen_phi_table.py > phi_table.h
"""
import struct

from mpmath import cos, erfc, exp, log, mp, mpf, nint, pi, sqrt

mp.dps = 40
PER_UNIT, NODES, DEG = 64, 609, 5
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
                worst[q] = max(worst[q], abs(v - fn(c + t)))
            co.append(p)
        a, b = co
        rows.append([f64(a[3]), f64(a[2]), f64(a[1]), f64(a[0]), f64(b[3]), f64(b[2]), f64(b[1]),
                     int(nint(b[0] * 2 ** 52)) & (2 ** 64 - 1), f32(a[5], a[4]), f32(b[5], b[4])])
    print("// Generated by gen_phi_table.py -- do not edit.")
    print("// Node i, t = z - i/64: F = phi/Phi and G = log Phi as degree-5 polynomials (layout: see the generator);")
    print("// largest absolute error before the coefficients' rounding: F %.1e, G %.1e." % (worst[0], worst[1]))
    print("#pragma once")
    print("constexpr int kPhiPerUnit = %d, kPhiNodes = %d, kPhiDeg = %d, kPhiRow = 10;" % (PER_UNIT, NODES, DEG))
    # pairs of words, so that the type carries the alignment of 16-byte loads
    print("__device__ const ulonglong2 g_phi_table[kPhiNodes * kPhiRow / 2] = {")
    for r in rows:
        print(",".join("{0x%016xull,0x%016xull}" % (r[k], r[k + 1]) for k in range(0, len(r), 2)) + ",")
    print("};")


if __name__ == "__main__":
    main()
