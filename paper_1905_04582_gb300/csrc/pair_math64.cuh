// FP64 per-pair arithmetic of Eq. (2) and Eq. (9) of arXiv:1905.04582, shared
// by the FP64 pair pass (pair_kernel.cu), the allocation-free entry point
// (noalloc.cu) and the held-out densities (heldout.cu).
//
// What bounds it: GB300 issues one FP64 warp instruction per SM sub-partition
// every 64 cycles, so a pair costs its FP64 instructions and everything else
// (integer, FP32, shared memory, MUFU) is nearly free beside them.  With
// CUDA's sqrt, division, erfc, exp and log1p a pair took about 187 of them at
// D = 2; the forms below take 19, and 14 more where Phi matters:
//  - 1/delta and delta: one cubic (Halley) step from the hardware's
//    reciprocal-root seed, then delta corrected by its own residual
//    d^2 - s^2, which an FMA gives exactly: 8, for a root and a division;
//  - phi/Phi and log Phi as functions of z alone, piecewise polynomials of
//    degree 7 on nodes 1/64 apart up to z = 10 (phi_table.h), the table in
//    shared memory: 14, for an exp, an erfc, a division and a log1p.  Both keep
//    their relative precision all the way, so that a pair with y = delta, whose
//    weight is phi/Phi alone, is as good as with CUDA's functions: largest
//    relative error against 50 digits 2e-16 up to z = 7 and 7e-16 at z = 10
//    (the former forms: 2e-15 and 4e-15 for phi/Phi, 1e-14 for log Phi).  The
//    powers from the fifth on are summed in FP32: at most (z t)^5 / 5! of the
//    value, 2.4e-8 at z = 10, their rounding is part of these errors;
//  - beyond z = 10 (phi/Phi < 8e-23) the two terms are added where that can
//    change a bit (phi_far): next to a residual (y - delta) / sigma of 2^-10
//    and more, and mostly below, they vanish in the rounding of the term they
//    would be added to;
//  - y, an FP32 value, widened by moving bits (a conversion instruction would
//    cost as much as an FMA).
// Measured (GB300, whole calls, 187 instructions -> these): L, dL/dX and
// dL/dsigma at N = 5392, D = 2, caller's order, 4.35 -> 1.05 ms; the
// allocation-free call at N = 3001, D = 3, 2.84 -> 0.63 ms.  (Degree 5 with two
// powers in FP32, log Phi's constants in units of 2^-52 and nothing beyond
// z = 9.5 took 0.97 and 0.57 ms: absolute errors of 1e-17, but no relative
// precision beyond z = 4.)
#pragma once

#include <cstdint>
#include <cstring>

namespace mds {
namespace {

#include "phi_table.h"

constexpr int kPhiBytes = kPhiNodes * kPhiRow * 8;  // 71,792
static_assert(kPhiDeg == 7 && kPhiPerUnit == 64 && kPhiRow == 14 && kPhiNodes == 641 && kPhiBytes % 16 == 0,
              "phi_eval is written for this table");

static_assert(alignof(decltype(g_phi_table)) >= 16, "phi_table_load reads it 16 bytes at a time");

// The table into shared memory (16-byte aligned), by all threads of the CTA;
// the caller synchronises.
__device__ __forceinline__ void phi_table_load(double *tab) {
    ulonglong2 *dst = reinterpret_cast<ulonglong2 *>(tab);
    for (int i = threadIdx.x; i < kPhiBytes / 16; i += blockDim.x) dst[i] = g_phi_table[i];
}

// sigma in the forms the pair needs.
struct Sigma64 {
    double inv_s;        // 1 / sigma
    double inv_s_nodes;  // 64 / sigma
    double neg_s;        // -sigma
    uint32_t near_hi;    // high word of 10 sigma: delta with a larger high word is beyond the table
    uint32_t tiny_hi;    // high word of 2^-10 sigma
};

// On the host, for a kernel argument: three divisions a thread would cost as
// much as a pair or two.
inline Sigma64 sigma64(double sigma) {
    const double near = 10.0 * sigma, tiny = 0x1p-10 * sigma;
    uint64_t bn, bt;
    std::memcpy(&bn, &near, sizeof(bn));
    std::memcpy(&bt, &tiny, sizeof(bt));
    return Sigma64{1.0 / sigma, 64.0 / sigma, -sigma, static_cast<uint32_t>(bn >> 32), static_cast<uint32_t>(bt >> 32)};
}

// An FP32 value as FP64: the exponent re-biased and the mantissa moved, for
// normal positive numbers (a dissimilarity); anything else is converted.
__device__ __forceinline__ double widen(float y) {
    const uint32_t b = __float_as_uint(y);
    if (b - 0x00800000u < 0x7f000000u)
        return __hiloint2double(static_cast<int>((b >> 3) + 0x38000000u), static_cast<int>(b << 29));
    return static_cast<double>(y);
}

// The same for a number of either sign (a coordinate).
__device__ __forceinline__ double widen_signed(float v) {
    const uint32_t b = __float_as_uint(v), m = b & 0x7fffffffu;
    if (m - 0x00800000u < 0x7f000000u)
        return __hiloint2double(static_cast<int>((b & 0x80000000u) | ((m >> 3) + 0x38000000u)),
                                static_cast<int>(b << 29));
    return static_cast<double>(v);
}

// delta = sqrt(d2) and 1 / delta for d2 >= 1e-300 (the caller starts its sum
// of squares there: coincident points get delta = 1e-150, below every
// rounding, and a gradient term of exactly 0).  With r the seed and
// e = 1 - d2 r^2: 1/sqrt(d2) = r (1 + e/2 + 3 e^2/8 + ...).
__device__ __forceinline__ void root64(double d2, double &del, double &inv) {
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d2));
    const double t = d2 * r;
    const double e = fma(-t, r, 1.0);
    const double q = e * fma(e, 0.375, 0.5);
    inv = fma(r, q, r);
    const double s = fma(t, q, t);
    const double half_inv = __hiloint2double(__double2hiint(inv) - 0x00100000, __double2loint(inv));
    del = fma(fma(-s, s, d2), half_inv, s);
}

// Whether the table has this delta (a compare of high words).
__device__ __forceinline__ bool phi_near(const Sigma64 &sg, double del) {
    return static_cast<uint32_t>(__double2hiint(del)) <= sg.near_hi;
}

// The node of z = del / sigma, phi_near(del): its index, and t = z - i / 64.
__device__ __forceinline__ uint32_t phi_node(const Sigma64 &sg, double del, double &t) {
    // z * 64 to the nearest integer (the low bits of a sum with 1.5 * 2^52); at most 640 as
    // phi_near bounds z, and cut there whatever the input
    const uint32_t i = min(static_cast<uint32_t>(__double2loint(fma(del, sg.inv_s_nodes, 6755399441055744.0))),
                           static_cast<uint32_t>(kPhiNodes - 1));
    // -i / 64: an FP32 number (exact), widened
    const float cf = (__uint_as_float(0x4B000000u | i) - 8388608.0f) * (1.0f / 64.0f);
    const double nc =
        __hiloint2double(static_cast<int>(i ? (__float_as_uint(cf) >> 3) + 0xB8000000u : 0u), 0);
    t = fma(del, sg.inv_s, nc);
    return i;
}

// t in FP32 (truncated; 0 below the FP32 range): the same bits, moved.
__device__ __forceinline__ float narrow(double t) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(t)), lo = static_cast<uint32_t>(__double2loint(t));
    const uint32_t m = hi & 0x7fffffffu;
    const uint32_t b = (hi & 0x80000000u) | ((m - 0x38000000u) << 3) | (lo >> 29);
    return m < 0x38100000u ? 0.f : __uint_as_float(b);
}

// G = log Phi(z) in two parts, slope * t + g0, for a sum that takes an FMA and
// an addition.
struct PhiLog {
    double slope, t, g0;
};

template <bool WANT_F, bool WANT_G>
__device__ __forceinline__ void phi_parts(const double *tab, const Sigma64 &sg, double del, bool near, double &F,
                                          PhiLog &G) {
    double t;
    const double2 *row = reinterpret_cast<const double2 *>(tab + phi_node(sg, del, t) * kPhiRow);
    t = near ? t : 0.0;
    const double2 mid = row[2];                                         // F's and G's of 1
    const float4 high = *reinterpret_cast<const float4 *>(row + 5);     // F's of t^7, t^6, t^5, G's of t^5
    const float tf = narrow(t);
    if constexpr (WANT_F) {
        const double2 f43 = row[0], f21 = row[1];
        const double u = widen_signed(fmaf(fmaf(high.x, tf, high.y), tf, high.z));
        F = fma(fma(fma(fma(fma(u, t, f43.x), t, f43.y), t, f21.x), t, f21.y), t, mid.x);
        F = near ? F : 0.0;
    }
    if constexpr (WANT_G) {
        const double2 g43 = row[3], g21 = row[4];
        const float2 top = *reinterpret_cast<const float2 *>(row + 6);  // G's of t^7, t^6
        const double u = widen_signed(fmaf(fmaf(top.x, tf, top.y), tf, high.w));
        G.slope = fma(fma(fma(fma(u, t, g43.x), t, g43.y), t, g21.x), t, g21.y);
        G.t = t;
        G.g0 = near ? mid.y : 0.0;
    }
}

// F = phi(z)/Phi(z) and G at z = del / sigma; 0 where near is false (near:
// phi_near(del)); WANT_G false leaves G alone.
template <bool WANT_G>
__device__ __forceinline__ void phi_eval(const double *tab, const Sigma64 &sg, double del, bool near, double &F,
                                         PhiLog &G) {
    phi_parts<true, WANT_G>(tab, sg, del, near, F, G);
}

// log Phi(z) alone, phi_near(del).
__device__ __forceinline__ double phi_log(const double *tab, const Sigma64 &sg, double del) {
    double F;
    PhiLog G;
    phi_parts<false, true>(tab, sg, del, true, F, G);
    return fma(G.slope, G.t, G.g0);
}

// Whether phi_far may have something to add beyond the table: w = y - delta
// below 2^-10 sigma (a compare of high words).
__device__ __forceinline__ bool phi_tiny(const Sigma64 &sg, double w) {
    return (static_cast<uint32_t>(__double2hiint(w)) & 0x7fffffffu) <= sg.tiny_hi;
}

// F and log Phi beyond the table (z >= 10, where F = phi and log Phi = -Q, the
// upper tail, to 1e-22 of themselves), for lanes with `in`: those with
// phi_tiny(w).  0 where adding them cannot change a bit: with u = w / sigma,
// F against u and Q against u^2 / 2 both stay below 2^-54 of what they are
// added to when Q <= phi(z) / 10 <= 2^-55 u^2, that is when
// log2 u^2 >= 51 - 0.7213 z^2 (0.7213 < 1 / (2 ln 2); exponents alone for u).
template <bool WANT_G>
__device__ __forceinline__ void phi_far(const Sigma64 &sg, double del, double w, bool in, double &F, double &G) {
    constexpr double kInvSqrt2Pi = 0.39894228040143267794, kInvSqrt2 = 0.70710678118654752440;
    const double z = del * sg.inv_s;
    const float zf = narrow(z);
    const int e = ((__double2hiint(w) >> 20) & 0x7ff) + ((__double2hiint(sg.inv_s) >> 20) & 0x7ff) - 2046;
    F = 0.0;
    G = 0.0;
    if (in && static_cast<float>(2 * e) < 51.f - 0.7213f * zf * zf) {
        F = exp(-0.5 * z * z) * kInvSqrt2Pi;
        if constexpr (WANT_G) G = -0.5 * erfc(z * kInvSqrt2);
    }
}

}  // namespace
}  // namespace mds
