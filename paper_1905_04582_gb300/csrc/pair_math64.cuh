// FP64 per-pair arithmetic of Eq. (2) and Eq. (9) of arXiv:1905.04582, shared
// by the FP64 pair pass (pair_kernel.cu), the allocation-free entry point
// (noalloc.cu) and the held-out densities (heldout.cu).
//
// What bounds it: GB300 issues one FP64 warp instruction per SM sub-partition
// every 64 cycles, so a pair costs its FP64 instructions and everything else
// (integer, FP32, shared memory, MUFU) is nearly free beside them.  With
// CUDA's sqrt, division, erfc, exp and log1p a pair took about 187 of them at
// D = 2; the forms below take 19, and 11 more where Phi matters:
//  - 1/delta and delta: one cubic (Halley) step from the hardware's
//    reciprocal-root seed, then delta corrected by its own residual
//    d^2 - s^2, which an FMA gives exactly: 8, for a root and a division;
//  - phi/Phi and log Phi as functions of z alone, piecewise polynomials of
//    degree 5 on nodes 1/64 apart (phi_table.h, absolute error 9e-18), the
//    table in shared memory: 11, for an exp, an erfc, a division and a log1p.
//    The two highest powers are FP32 (t^4 <= 3.7e-9 takes their rounding below
//    1e-16 of F and G; errors against 40 digits: F 1.3e-17 rms as in FP64
//    throughout), t and their sum carried over by moving bits; G's constant is
//    summed as an integer, so that its last step is the sum's own FMA.
//    What matters is their absolute error: beside phi/Phi the weight holds
//    (delta - y)/sigma, whose rounding is at least 2^-53 z;
//  - beyond z = 9.5 both are dropped: phi/Phi < 1.1e-20 there, five orders
//    below half an ulp of delta/sigma (1e-15), the rounding of the term it
//    would be added to, and |log Phi| < 1.1e-21 against terms whose sum is
//    rounded at 1e-16;
//  - y, an FP32 value, widened by moving bits (a conversion instruction would
//    cost as much as an FMA).
// Measured (GB300, whole calls, the errors against 64 bits unchanged): L,
// dL/dX and dL/dsigma at N = 5392, D = 2, caller's order, 4.35 -> 0.97 ms (1.00
// with every power in FP64); the allocation-free call at N = 3001, D = 3,
// 2.84 -> 0.57 ms.
#pragma once

#include <cstdint>
#include <cstring>

namespace mds {
namespace {

#include "phi_table.h"

constexpr int kPhiBytes = kPhiNodes * kPhiRow * 8;  // 48,720
static_assert(kPhiDeg == 5 && kPhiPerUnit == 64 && kPhiRow == 10 && kPhiBytes % 16 == 0,
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
    uint32_t near_hi;    // high word of 9.5 sigma: delta with a larger high word is beyond the table
};

// On the host, for a kernel argument: three divisions a thread would cost as
// much as a pair or two.
inline Sigma64 sigma64(double sigma) {
    const double near = 9.5 * sigma;
    uint64_t bits;
    std::memcpy(&bits, &near, sizeof(bits));
    return Sigma64{1.0 / sigma, 64.0 / sigma, -sigma, static_cast<uint32_t>(bits >> 32)};
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

// Whether phi/Phi and log Phi are kept at this delta (a compare of high words).
__device__ __forceinline__ bool phi_near(const Sigma64 &sg, double del) {
    return static_cast<uint32_t>(__double2hiint(del)) <= sg.near_hi;
}

// The node of z = del / sigma, phi_near(del): its index, and t = z - i / 64.
__device__ __forceinline__ uint32_t phi_node(const Sigma64 &sg, double del, double &t) {
    // z * 64 to the nearest integer (the low bits of a sum with 1.5 * 2^52); at most 608 as
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

// G = log Phi(z) in two parts: slope * t + units * 2^-52.
struct PhiLog {
    double slope, t;
    int64_t units;
};
constexpr double kPhiUnit = 0x1p-52;

template <bool WANT_F, bool WANT_G>
__device__ __forceinline__ void phi_parts(const double *tab, const Sigma64 &sg, double del, bool near, double &F,
                                          PhiLog &G) {
    double t;
    const double2 *row = reinterpret_cast<const double2 *>(tab + phi_node(sg, del, t) * kPhiRow);
    t = near ? t : 0.0;
    const float4 high = *reinterpret_cast<const float4 *>(row + 4);
    const float tf = narrow(t);
    if constexpr (WANT_F) {
        const double2 f32 = row[0], f10 = row[1];
        const double u = widen_signed(fmaf(high.x, tf, high.y));
        F = fma(fma(fma(fma(u, t, f32.x), t, f32.y), t, f10.x), t, f10.y);
        F = near ? F : 0.0;
    }
    if constexpr (WANT_G) {
        const double2 g32 = row[2], g10 = row[3];
        const double u = widen_signed(fmaf(high.z, tf, high.w));
        G.slope = fma(fma(fma(u, t, g32.x), t, g32.y), t, g10.x);
        G.t = t;
        G.units = near ? __double_as_longlong(g10.y) : 0;
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
    return fma(G.slope, G.t, static_cast<double>(G.units) * kPhiUnit);
}

}  // namespace
}  // namespace mds
