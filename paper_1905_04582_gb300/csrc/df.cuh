// Double-float sums and the split location layouts, shared by the reduction
// (reduce_kernel.cu) and the small-problem trajectory (small_traj.cu).
#pragma once

#include <cstdint>

#include "mds_internal.h"

namespace mds {
namespace {

// ------------------------------------------------- double-float accumulator

// hi + lo with |lo| <= ulp(hi)/2, updated with Knuth's two-sum.
struct DF {
    float hi, lo;
};

__device__ __forceinline__ void df_add(DF &a, float v) {
    const float s = __fadd_rn(a.hi, v);
    const float bp = __fsub_rn(s, a.hi);
    const float err = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bp)), __fsub_rn(v, bp));
    a.hi = s;
    a.lo = __fadd_rn(a.lo, err);
}

__device__ __forceinline__ void df_add(DF &a, const DF &b) {
    df_add(a, b.hi);
    a.lo = __fadd_rn(a.lo, b.lo);
}

__device__ __forceinline__ float df_float(const DF &a) { return __fadd_rn(a.hi, a.lo); }

// Double-float product a * (b.x + b.y): the exact product of the leading
// parts by an FMA (Dekker's two-product), the cross terms added to its
// error, then a fast two-sum (|p| >= |t|) into (hi, lo); relative error
// about 2^-44, the precision of the double-float sums themselves.
__device__ __forceinline__ DF df_mul(const DF &a, float2 b) {
    const float p = __fmul_rn(a.hi, b.x);
    const float e = __fmaf_rn(a.hi, b.x, -p);
    const float t = __fmaf_rn(a.hi, b.y, __fmaf_rn(a.lo, b.x, e));
    const float hi = __fadd_rn(p, t);
    return DF{hi, __fsub_rn(t, __fsub_rn(hi, p))};
}
__device__ __forceinline__ double df_double(const DF &a) { return static_cast<double>(a.hi) + static_cast<double>(a.lo); }

__device__ __forceinline__ DF df_shfl_xor(const DF &a, int o) {
    return DF{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}

// Rewrite slot k, coordinate kk of the FP32C split layouts from value v.
__device__ __forceinline__ void write_split_slot(const XState &xs, const Split &sp, int64_t k, int d, int kk,
                                                 float v) {
    const float h = __fsub_rn(__fadd_rn(v, sp.magic), sp.magic);  // nearest multiple of q
    const float l = __fsub_rn(v, h);                               // exact
    float *xr = reinterpret_cast<float *>(xs.xrow + (((k >> 6) * d + kk) * 32 + ((k >> 1) & 31)));
    xr[k & 1] = h;
    xr[2 + (k & 1)] = l;
    xs.xcol[k * d + kk] = make_float4(-h, -h, -l, -l);
    if (xs.xcol2) xs.xcol2[k * d + kk] = make_float2(-h, -l);
}

}  // namespace
}  // namespace mds
