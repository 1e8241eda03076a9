// Cross-validation folds (arXiv:1905.04582, section 2.4 "Model selection").
//
// A fold holds out a set of observations y_ij; the model is trained on the
// rest (the pair pass skips pairs whose tile-packed y is negative) and the
// held-out pairs are scored by the log pointwise predictive density,
// estimated from S posterior draws as
//   lpd-hat = sum_ij log( (1/S) sum_s p(y_ij | X_s, sigma_s) ),
// p the truncated-normal density of Eq. (1):
//   log p(y | delta, sigma) = -log(sqrt(2 pi) sigma) - (y - delta)^2 / (2 sigma^2)
//                             - log Phi(delta / sigma).
// The estimate is accumulated one draw at a time as a running log-sum-exp per
// pair (max m and scaled sum s, so no exp underflows), in FP64: the held-out
// set is small next to the M pairs of the pass and is scored once per draw.
#include <cmath>
#include <cstdint>

#include "mds_internal.h"
#include "pair_math64.cuh"

namespace mds {
namespace {

constexpr int kHoThreads = 256;
constexpr int kLpdThreads = 512;
constexpr int kSms = 152;  // GB300

__device__ __forceinline__ double to_double(double v) { return v; }
__device__ __forceinline__ double to_double(float v) { return widen_signed(v); }

__global__ void ho_mark_kernel(float *y, const int64_t *off, int64_t count, float *ho_y, unsigned char *tile_ho) {
    for (int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < count;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int64_t o = off[k];
        ho_y[k] = y[o];
        y[o] = -1.0f;
        tile_ho[o / kTileElems] = 1;
    }
}

__global__ void ho_restore_kernel(float *y, const int64_t *off, int64_t count, const float *ho_y) {
    for (int64_t k = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; k < count;
         k += static_cast<int64_t>(gridDim.x) * blockDim.x)
        y[off[k]] = ho_y[k];
}

// lp = log p(y | delta, sigma) of every held-out pair.  Bound by the FP64 pipe
// like the FP64 pair pass, so it takes that pass's forms (pair_math64.cuh):
// delta without a square root, log Phi from the table, the constants of sigma
// from the host; about 26 FP64 instructions a pair at D = 3 where CUDA's
// sqrt, divisions, erfc and log1p took about 220.  Two CTAs per SM, each with
// the table in shared memory and a contiguous share of the pairs.  Measured
// (GB300, the whole fold: gradient, one draw, sum): N = 2999, D = 3, 225,000
// held-out pairs 221 -> 104 us, the waits and the sum's one launch included.
template <typename T>
__global__ void __launch_bounds__(kLpdThreads, 2)
    lpd_accumulate_kernel(const T *x, int d, const int2 *pairs, const float *ho_y, int64_t count, Sigma64 sg,
                          double log_norm, bool first, double *lse_m, double *lse_s, unsigned *err) {
    extern __shared__ __align__(16) unsigned char lpd_smem[];
    double *tab = reinterpret_cast<double *>(lpd_smem);
    phi_table_load(tab);
    __syncthreads();
    // a contiguous share per CTA: every SM then ends with the same number of
    // warps (in a grid stride the last round filled some SMs and not others)
    const int64_t per = (count + gridDim.x - 1) / gridDim.x;
    const int64_t k1 = min(count, (blockIdx.x + 1) * per);
    for (int64_t k = blockIdx.x * per + threadIdx.x; k < k1; k += kLpdThreads) {
        const int2 p = pairs[k];
        const float y = ho_y[k];
        const T *xi = x + static_cast<int64_t>(p.x) * d, *xj = x + static_cast<int64_t>(p.y) * d;
        double d2 = 1e-300;  // see root64
        for (int c = 0; c < d; ++c) {
            const double t = to_double(xi[c]) - to_double(xj[c]);
            d2 = fma(t, t, d2);
        }
        double delta, inv;
        root64(d2, delta, inv);
        const double u = (widen(y) - delta) * sg.inv_s;
        double lp = fma(-0.5 * u, u, log_norm);
        // beyond the table Phi is 1 - 8e-24 at least: no factor of a density
        if (phi_near(sg, delta)) lp -= phi_log(tab, sg, delta);
        if (!isfinite(lp)) atomicOr(err, kErrNonfinite);
        if (first) {
            lse_m[k] = lp;
            lse_s[k] = 1.0;
        } else {
            const double m = lse_m[k];
            if (lp > m) {
                lse_s[k] = lse_s[k] * exp(m - lp) + 1.0;
                lse_m[k] = lp;
            } else {
                lse_s[k] += exp(lp - m);
            }
        }
    }
}

// Block sum in a fixed order, in thread 0: shuffles, then the warps' sums.
__device__ __forceinline__ double block_sum(double v, double *sm) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = sm[threadIdx.x % (kHoThreads / 32)];
    if (threadIdx.x < 32) {
#pragma unroll
        for (int o = kHoThreads / 64; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    }
    __syncthreads();
    return t;
}

// Block b sums the terms k = b kHoThreads + thread, in steps of the grid; the
// last block to finish (a ticket that wraps to 0 for the next launch) sums the
// kLpdParts partials, all in a fixed order, into out (pinned host memory).
__global__ void __launch_bounds__(kHoThreads)
    lpd_sum_kernel(const double *lse_m, const double *lse_s, int64_t count, double log_draws, double *part,
                   unsigned *ticket, double *out) {
    __shared__ double sm[kHoThreads / 32];
    __shared__ bool last;
    double v = 0.0;
    for (int64_t k = static_cast<int64_t>(blockIdx.x) * kHoThreads + threadIdx.x; k < count;
         k += static_cast<int64_t>(kLpdParts) * kHoThreads) {
        // log 1 = 0 is left out: after the first draw every s is 1, and the FP64 log (about 40 instructions) would be
        // most of this kernel
        const double sc = lse_s[k];
        v += lse_m[k] - log_draws;
        if (sc != 1.0) v += log(sc);
    }
    const double t = block_sum(v, sm);
    if (threadIdx.x == 0) {
        part[blockIdx.x] = t;
        __threadfence();
        last = atomicInc(ticket, kLpdParts - 1) == kLpdParts - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    v = 0.0;
    for (int k = threadIdx.x; k < kLpdParts; k += kHoThreads) v += __ldcg(part + k);
    const double total = block_sum(v, sm);
    if (threadIdx.x == 0) *out = total;
}

int grid_of(int64_t count) {
    const int64_t g = (count + kHoThreads - 1) / kHoThreads;
    return static_cast<int>(g < 4096 ? (g > 0 ? g : 1) : 4096);
}

}  // namespace

cudaError_t launch_ho_mark(float *y, const int64_t *off, int64_t count, float *ho_y, unsigned char *tile_ho,
                           cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    ho_mark_kernel<<<grid_of(count), kHoThreads, 0, s>>>(y, off, count, ho_y, tile_ho);
    return cudaGetLastError();
}

cudaError_t launch_ho_restore(float *y, const int64_t *off, int64_t count, const float *ho_y, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    ho_restore_kernel<<<grid_of(count), kHoThreads, 0, s>>>(y, off, count, ho_y);
    return cudaGetLastError();
}

cudaError_t launch_lpd_accumulate(const void *x, bool fp64, int d, const int2 *pairs, const float *ho_y,
                                  int64_t count, double sigma, bool first, double *lse_m, double *lse_s,
                                  unsigned *err, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    const Sigma64 sg = sigma64(sigma);
    const double log_norm = -0.91893853320467274178 - std::log(sigma);  // -log(sqrt(2 pi) sigma)
    const int64_t blocks = (count + kLpdThreads - 1) / kLpdThreads;
    const int grid = static_cast<int>(blocks < 2 * kSms ? blocks : 2 * kSms);
    cudaError_t e = raise_dyn_smem(fp64 ? reinterpret_cast<const void *>(lpd_accumulate_kernel<double>)
                                        : reinterpret_cast<const void *>(lpd_accumulate_kernel<float>),
                                   kPhiBytes);
    if (e != cudaSuccess) return e;
    if (fp64)
        lpd_accumulate_kernel<double><<<grid, kLpdThreads, kPhiBytes, s>>>(
            static_cast<const double *>(x), d, pairs, ho_y, count, sg, log_norm, first, lse_m, lse_s, err);
    else
        lpd_accumulate_kernel<float><<<grid, kLpdThreads, kPhiBytes, s>>>(
            static_cast<const float *>(x), d, pairs, ho_y, count, sg, log_norm, first, lse_m, lse_s, err);
    return cudaGetLastError();
}

cudaError_t launch_lpd_sum(const double *lse_m, const double *lse_s, int64_t count, double draws, double *part,
                           unsigned *ticket, double *out, cudaStream_t s) {
    lpd_sum_kernel<<<kLpdParts, kHoThreads, 0, s>>>(lse_m, lse_s, count, std::log(draws), part, ticket, out);
    return cudaGetLastError();
}

}  // namespace mds
