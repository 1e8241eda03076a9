// One quarter tile (64 rows x 16 columns) by one warp: the pair arithmetic of
// the chunked pass (chunk_kernel.cu), its lane mappings and its row and column
// sums, shared with the small-problem trajectory (small_traj.cu).
#pragma once

#include <cfloat>
#include <cstdint>

#include "mds_internal.h"
#include "pair_math.cuh"

namespace mds {
namespace {

// x / 2 for a normal, positive FP32 x: one less in the exponent field (an
// integer subtraction on the ALU pipe instead of an FP32 multiply).
__device__ __forceinline__ float half_of(float x) { return __int_as_float(__float_as_int(x) - 0x00800000); }

// Geometry of two pairs (rows r, r+1 packed) against one column: the exact
// split differences per coordinate, delta, 1 / delta and the
// residual-corrected e = y - delta (see mds_internal.h, Split).
template <int D>
__device__ __forceinline__ void geom2(const float4 (&xi)[D], const float4 (&xj)[D], float2 y2, float2 (&s)[D],
                                      float2 &d2, float2 &inv, float2 &del, float2 &e) {
    if constexpr (D == 1) {
        geom_line(xi[0], xj[0], y2, s[0], d2, inv, del, e);
        return;
    }
    float2 d2h, cr;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float2 dh = add2(f2(xi[k].x, xi[k].y), f2(xj[k].x, xj[k].y));  // exact
        const float2 dl = add2(f2(xi[k].z, xi[k].w), f2(xj[k].z, xj[k].w));
        s[k] = add2(dh, dl);  // x_i - x_j, rounded once
        if (k == 0) {
            d2h = mul2(dh, dh);
            cr = fma2(dl, add2(s[k], dh), f2(FLT_MIN, FLT_MIN));
        } else {
            d2h = fma2(dh, dh, d2h);           // exact
            cr = fma2(dl, add2(s[k], dh), cr);  // Dl (2 Dh + Dl)
        }
    }
    d2 = add2(d2h, cr);
    inv = f2(rsqrt_approx(d2.x), rsqrt_approx(d2.y));
    del = f2(sqrt_approx(d2.x), sqrt_approx(d2.y));
    // delta_true = del + res / (2 del), res = (d2h - del^2) + cr
    const float2 res = add2(fma2(neg2(del), del, d2h), cr);
    const float2 hinv = f2(half_of(inv.x), half_of(inv.y));
    e = fma2(neg2(res), hinv, add2(y2, neg2(del)));
}

// Both-sided accumulation of the scaled gradient weight wi' = -sigma^2 w / delta
// (INIT: the column sums start here, a multiply instead of zeroing them).
template <int D, bool INIT = false>
__device__ __forceinline__ void accum2(float2 wi, const float2 (&s)[D], float2 (&racc)[D], float2 (&cacc)[D]) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
        racc[k] = fma2(wi, s[k], racc[k]);
        cacc[k] = INIT ? mul2(wi, s[k]) : fma2(wi, s[k], cacc[k]);
    }
}

// The full body: Phi via the Mills ratio (pair_kernel.cu), e^2, phi'/Phi
// delta and the product of 1/Phi accumulated; MASKED zeroes the pairs with
// vmask = 0.
template <int D, bool MASKED, bool INIT = false>
__device__ __forceinline__ void body_full(const PairArgs &a, const float4 (&xi)[D], const float4 (&xj)[D], float2 y2,
                                          float2 vmask, float2 (&racc)[D], float2 (&cacc)[D], float2 &e2, float2 &md,
                                          float2 &prod) {
    float2 s[D], d2, inv, del, e;
    geom2<D>(xi, xj, y2, s, d2, inv, del, e);
    const float2 ea = mul2(d2, a.c_phi);
    const float2 ph = f2(ex2_approx(ea.x), ex2_approx(ea.y));  // exp(-z^2 / 2)
    float2 pn = fma2(a.mp[3], del, a.mp[2]);
    pn = fma2(pn, del, a.mp[1]);
    pn = fma2(pn, del, a.mp[0]);
    float2 dd = fma2(a.md[3], del, a.md[2]);
    dd = fma2(dd, del, a.md[1]);
    dd = fma2(dd, del, a.md[0]);
    const float2 den = fma2(ph, pn, dd);  // D Phi
    const float2 rden = f2(rcp_approx(den.x), rcp_approx(den.y));
    float2 ip = mul2(dd, rden);  // 1 / Phi
    float2 mm = mul2(ph, ip);    // sqrt(2 pi) phi / Phi
    if (MASKED) {
        e = mul2(e, vmask);
        mm = mul2(mm, vmask);
        ip = f2(vmask.x != 0.f ? ip.x : 1.f, vmask.y != 0.f ? ip.y : 1.f);
    }
    prod = mul2(prod, ip);
    e2 = fma2(e, e, e2);
    md = fma2(mm, del, md);
    // wi' = (e - sigma phi'/sqrt(2 pi)) / delta
    accum2<D, INIT>(mul2(fma2(mm, a.c_m2, e), inv), s, racc, cacc);
}

// The far body (every pair of the warp's block at z >= z_c): the Phi terms
// are below FP32 resolution and dropped (pair_math.cuh, pair2_far).
template <int D, bool INIT = false>
__device__ __forceinline__ void body_far(const float4 (&xi)[D], const float4 (&xj)[D], float2 y2, float2 (&racc)[D],
                                         float2 (&cacc)[D], float2 &e2) {
    float2 s[D], d2, inv, del, e;
    geom2<D>(xi, xj, y2, s, d2, inv, del, e);
    e2 = fma2(e, e, e2);
    accum2<D, INIT>(mul2(e, inv), s, racc, cacc);
}

// Whether every pair of the warp's 64 rows x 8 columns lies at squared
// distance >= far_d2 (the columns in the {-xh, -xl} form).
template <int D>
__device__ __forceinline__ bool block_far2(const float *box, const float2 (&c)[2][D], float far_d2) {
    float g0 = 0.f, g1 = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        const float lo = box[k], hi = box[D + k];
        const float c0 = -(c[0][k].x + c[0][k].y), c1 = -(c[1][k].x + c[1][k].y);
        const float d0 = fmaxf(fmaxf(lo - c0, c0 - hi), 0.f);
        const float d1 = fmaxf(fmaxf(lo - c1, c1 - hi), 0.f);
        g0 = fmaf(d0, d0, g0);
        g1 = fmaf(d1, d1, g1);
    }
    return __all_sync(0xffffffffu, fminf(g0, g1) >= far_d2);
}

// Place of value v (column v / D, coordinate v % D) where columns lie S floats apart.
template <int D, int S>
__device__ __forceinline__ int sum_at(int v) {
    return S == D ? v : v / D * S + v % D;
}

// One tile for this lane (8 rows x 4 columns, column pairs in turn; see
// pair_math.cuh tile_f32).  Returns the column pairs that took the far body.
// NQ < 4: a unit of fewer rows (16 NQ, the pointers and row_rel set to its
// first); S: floats between the column sums of neighbouring columns.
template <int D, bool MASKED, bool HELDOUT, int NQ = 4, int S = D>
__device__ __forceinline__ int tile_chunk(const PairArgs &a, const float4 *ys, const float2 *xjs, const float4 *xis,
                                          int lane, int row_rel, int col_lo, int64_t ncol_valid, float2 (&racc)[NQ][D],
                                          float *colp, float2 &e2, float2 &md, float2 &prod, const float *box) {
    constexpr int V = 2 * D;
    constexpr int P = Pow2<V>::value;
    const int la = lane & 7, lb = lane >> 3;
    int n_far = 0;
#pragma unroll 1
    for (int cp = 0; cp < 2; ++cp) {
        float2 cj[2][D];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int k = 0; k < D; ++k) cj[e][k] = xjs[(4 * lb + 2 * cp + e) * D + k];
        float4 xj[2][D];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int k = 0; k < D; ++k) xj[e][k] = make_float4(cj[e][k].x, cj[e][k].x, cj[e][k].y, cj[e][k].y);
        float2 cacc[2][D];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int k = 0; k < D; ++k) cacc[e][k] = f2(0.f, 0.f);
        bool far = false;
        if constexpr (!MASKED) far = block_far2<D>(box, cj, a.far_d2);
        if (far) {
            ++n_far;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const float4 yv = ys[(2 * q + cp) * 32 + (lane ^ (cp << 2))];
                float4 xi[D];
#pragma unroll
                for (int k = 0; k < D; ++k) xi[k] = xis[k * 32 + la + 8 * q];
                body_far<D>(xi, xj[0], f2(yv.x, yv.y), racc[q], cacc[0], e2);
                body_far<D>(xi, xj[1], f2(yv.z, yv.w), racc[q], cacc[1], e2);
            }
        } else {
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                const float4 yv = ys[(2 * q + cp) * 32 + (lane ^ (cp << 2))];
                float4 xi[D];
#pragma unroll
                for (int k = 0; k < D; ++k) xi[k] = xis[k * 32 + la + 8 * q];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 y2 = e == 0 ? f2(yv.x, yv.y) : f2(yv.z, yv.w);
                    float2 vm = f2(1.f, 1.f);
                    if (MASKED) {
                        // rows r, r+1 of the row pair, column c (tile-relative,
                        // rows shifted so that the diagonal test is c > r); with
                        // a cross-validation fold, a held-out pair carries y < 0
                        const int r = row_rel + 2 * (la + 8 * q);
                        const int c = col_lo + 4 * lb + 2 * cp + e;
                        const bool cv = c < ncol_valid;
                        if (HELDOUT)
                            vm = f2((cv && c > r && y2.x >= 0.f) ? 1.f : 0.f, (cv && c > r + 1 && y2.y >= 0.f) ? 1.f : 0.f);
                        else
                            vm = f2((cv && c > r) ? 1.f : 0.f, (cv && c > r + 1) ? 1.f : 0.f);
                    }
                    body_full<D, MASKED>(a, xi, xj[e], y2, vm, racc[q], cacc[e], e2, md, prod);
                }
            }
        }
        // column sums over the tile's 64 rows: 3-level transpose over the row lanes
        float colv[P];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int k = 0; k < D; ++k) colv[e * D + k] = cacc[e][k].x + cacc[e][k].y;
#pragma unroll
        for (int i = V; i < P; ++i) colv[i] = 0.f;
        lane_reduce<P, 3>(colv, lane, 0);
        bool writer;
        const int base = reduced_base<P, 3>(lane, 0, writer);
        constexpr int kHeld = P >= 8 ? P / 8 : 1;
        if (writer) {
#pragma unroll
            for (int i = 0; i < kHeld; ++i)
                if (base + i < V) colp[(4 * lb + 2 * cp) * S + sum_at<D, S>(base + i)] = colv[i];
        }
    }
    return n_far;
}

// One tile for this lane in the tall mapping (D <= 2): lane 4b + a takes the
// 16 rows 2(a + 4q) + {0, 1}, q = 0..7, against the 2 columns 2b, 2b + 1 of
// the warp's 16: one block test, one load of the column locations and one
// 2-level column transpose per tile.  ybe / ybo: the lane's float4 index in
// the warp's Y quarter for even / odd q (tile layout, mds_internal.h), plus
// (q / 2) * 64.  Returns the 64 x 8 blocks of the warp that took the far body
// (0 or 2).
// NQ < 8: a unit of fewer rows (8 NQ), as in tile_chunk.
template <int D, bool MASKED, bool HELDOUT, int NQ = 8, int S = D>
__device__ __forceinline__ int tile_tall(const PairArgs &a, const float4 *ys, const float2 *xjs, const float4 *xis,
                                         int lane, int ybe, int ybo, int row_rel, int col_lo, int64_t ncol_valid,
                                         float2 (&racc)[NQ][D], float *colp, float2 &e2, float2 &md, float2 &prod,
                                         const float *box) {
    constexpr int V = 2 * D;
    constexpr int P = Pow2<V>::value;
    const int la = lane & 3, lb = lane >> 2;
    float2 cj[2][D];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int k = 0; k < D; ++k) cj[e][k] = xjs[(2 * lb + e) * D + k];
    float4 xj[2][D];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int k = 0; k < D; ++k) xj[e][k] = make_float4(cj[e][k].x, cj[e][k].x, cj[e][k].y, cj[e][k].y);
    float2 cacc[2][D];
    bool far = false;
    if constexpr (!MASKED) far = block_far2<D>(box, cj, a.far_d2);
    if (far) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 yv = ys[(q >> 1) * 64 + ((q & 1) ? ybo : ybe)];
            float4 xi[D];
#pragma unroll
            for (int k = 0; k < D; ++k) xi[k] = xis[k * 32 + la + 4 * q];
            if (q == 0) {
                body_far<D, true>(xi, xj[0], f2(yv.x, yv.y), racc[q], cacc[0], e2);
                body_far<D, true>(xi, xj[1], f2(yv.z, yv.w), racc[q], cacc[1], e2);
            } else {
                body_far<D>(xi, xj[0], f2(yv.x, yv.y), racc[q], cacc[0], e2);
                body_far<D>(xi, xj[1], f2(yv.z, yv.w), racc[q], cacc[1], e2);
            }
        }
    } else {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const float4 yv = ys[(q >> 1) * 64 + ((q & 1) ? ybo : ybe)];
            float4 xi[D];
#pragma unroll
            for (int k = 0; k < D; ++k) xi[k] = xis[k * 32 + la + 4 * q];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float2 y2 = e == 0 ? f2(yv.x, yv.y) : f2(yv.z, yv.w);
                float2 vm = f2(1.f, 1.f);
                if (MASKED) {
                    const int r = row_rel + 2 * (la + 4 * q);
                    const int c = col_lo + 2 * lb + e;
                    const bool cv = c < ncol_valid;
                    if (HELDOUT)
                        vm = f2((cv && c > r && y2.x >= 0.f) ? 1.f : 0.f, (cv && c > r + 1 && y2.y >= 0.f) ? 1.f : 0.f);
                    else
                        vm = f2((cv && c > r) ? 1.f : 0.f, (cv && c > r + 1) ? 1.f : 0.f);
                }
                if (q == 0)
                    body_full<D, MASKED, true>(a, xi, xj[e], y2, vm, racc[q], cacc[e], e2, md, prod);
                else
                    body_full<D, MASKED>(a, xi, xj[e], y2, vm, racc[q], cacc[e], e2, md, prod);
            }
        }
    }
    // column sums over the tile's 64 rows: 2-level transpose over the row lanes
    float colv[P];
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int k = 0; k < D; ++k) colv[e * D + k] = cacc[e][k].x + cacc[e][k].y;
#pragma unroll
    for (int i = V; i < P; ++i) colv[i] = 0.f;
    lane_reduce<P, 2>(colv, lane, 0);
    bool writer;
    const int base = reduced_base<P, 2>(lane, 0, writer);
    constexpr int kHeld = P >= 4 ? P / 4 : 1;
    if (writer) {
#pragma unroll
        for (int i = 0; i < kHeld; ++i)
            if (base + i < V) colp[2 * lb * S + sum_at<D, S>(base + i)] = colv[i];
    }
    return far ? 2 : 0;
}

// Row sums of one segment in the tall mapping into the warp's partial slot:
// sums over the 8 column lanes of each row (3-level lane transpose).
template <int D, int NQ = 8, int S = D>
__device__ __forceinline__ void flush_rows_tall(float2 (&racc)[NQ][D], int lane, float *rp) {
    constexpr int VR = 2 * NQ * D;
    static_assert(VR % 8 == 0, "three halvings of the values");
    float rv[VR];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int k = 0; k < D; ++k) {
            rv[(q * D + k) * 2 + 0] = racc[q][k].x;
            rv[(q * D + k) * 2 + 1] = racc[q][k].y;
            racc[q][k] = f2(0.f, 0.f);
        }
    lane_reduce<VR, 3>(rv, lane, 2);
    bool writer;
    const int base = reduced_base<VR, 3>(lane, 2, writer);
    const int la = lane & 3;
#pragma unroll
    for (int i = 0; i < VR / 8; ++i) {
        const int v = base + i;
        const int h = v & 1, k = (v >> 1) % D, q = (v >> 1) / D;
        rp[(2 * (la + 4 * q) + h) * S + k] = rv[i];
    }
}

// A warp's row sums of one segment (its 16 columns of every tile) into its
// partial slot rp[64 * D]: sums over the 4 column lanes of each row
// (lane transpose), then one store per value.
template <int D, int NQ = 4, int S = D>
__device__ __forceinline__ void flush_rows(float2 (&racc)[NQ][D], int lane, float *rp) {
    constexpr int VR = 2 * NQ * D;
    static_assert(VR % 4 == 0, "two halvings of the values");
    float rv[VR];
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
        for (int k = 0; k < D; ++k) {
            rv[(q * D + k) * 2 + 0] = racc[q][k].x;
            rv[(q * D + k) * 2 + 1] = racc[q][k].y;
            racc[q][k] = f2(0.f, 0.f);
        }
    lane_reduce<VR, 2>(rv, lane, 3);
    bool writer;
    const int base = reduced_base<VR, 2>(lane, 3, writer);
    const int la = lane & 7;
#pragma unroll
    for (int i = 0; i < VR / 4; ++i) {
        const int v = base + i;
        const int h = v & 1, k = (v >> 1) % D, q = (v >> 1) / D;
        rp[(2 * (la + 8 * q) + h) * S + k] = rv[i];
    }
}

}  // namespace
}  // namespace mds
