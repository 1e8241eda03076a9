// Allocation-free evaluation of the likelihood and its gradients.
//
// Some callers cannot let a library allocate device memory: a host program
// that budgets every byte of the GPU itself, code that runs inside a memory
// allocator's own callback (where a nested cudaMalloc could deadlock or
// recurse), or a real-time loop that must not allocate after start-up.  For
// them, mds_loglik_grad_noalloc() evaluates L, dL/dX and dL/dsigma from
// caller-owned device buffers and allocates nothing: its only scratch is the
// fixed file-scope array below, which every GPU that loads this library
// holds until the process exits.
//
// Work split: a CTA takes whole rows i of the full N x N matrix Y, in steps of
// the grid; its threads stride over j != i, so every pair is
// visited twice (once per end, as the per-row gradient sums of the paper's
// Algorithm 2) and no column partials are needed.  The per-pair arithmetic is
// that of the FP64 path (pair_math64.cuh), bound by the FP64 pipe; log Phi
// and the other scalar terms are evaluated only for j > i.  A whole CTA per
// row rather than a warp: the rows then come in pieces small enough to end
// together on 152 SMs.  The CTAs are resident all at once, two or three per SM,
// and load the table once; how many, by what the last round leaves idle
// (row_blocks): at D = 2 two and three per SM take 354 and 367 us at N = 2400,
// 955 and 925 at N = 4000.  (With a shorter table, a CTA per row left to the
// scheduler took 400 us at N = 2400 against 351 for resident ones.)  Each
// block writes its partial sums of the scalar terms into the scratch array; a
// second, single-block kernel sums them in a fixed order.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <mutex>

#include "mds.h"
#include "mds_internal.h"
#include "pair_math.cuh"
#include "pair_math64.cuh"

namespace mds {
namespace {

constexpr int kNaWarps = 4;
constexpr int kNaThreads = 32 * kNaWarps;
constexpr int kNaMaxBlocks = 8192;
constexpr int64_t kNaMaxN = 65536;
constexpr int kNaParts = 4;                       // e^2, m*delta, log Phi, spare

// The scratch: per-block partial sums, then the three final sums.
static __device__ __align__(256) double g_noalloc_scratch[kNaMaxBlocks * kNaParts + kNaParts];

constexpr int kMaxDevices = 64;
std::mutex g_na_mu;
double *g_na_ptr[kMaxDevices] = {};
int g_na_sms[kMaxDevices] = {};

// Row sums: gradient in units of -sigma^2 (see pair_f64_kernel), then the scalars.
template <int D>
struct RowSums {
    double v[Pow2<D + 3>::value];
};

// Pairs (i, j) of row i for j in [lo, hi), a thread each in turn; SCALARS: their scalar terms too.
template <int D, bool SCALARS>
__device__ __forceinline__ void row_part(const double *tab, const Sigma64 &sg, const double (&xi)[D],
                                         const double *x, const float *yrow, int64_t lo, int64_t hi, RowSums<D> &acc) {
    for (int64_t j0 = lo; j0 < hi; j0 += kNaThreads) {
        const bool in = j0 + threadIdx.x < hi;
        const int64_t j = in ? j0 + threadIdx.x : lo;
        double dl[D];
        double d2 = 1e-300;  // see root64
#pragma unroll
        for (int k = 0; k < D; ++k) {
            dl[k] = xi[k] - x[j * D + k];
            d2 = fma(dl[k], dl[k], d2);
        }
        double del, inv;
        root64(d2, del, inv);
        double w = in ? widen(yrow[j]) - del : 0.0;  // y - delta
        if constexpr (SCALARS) acc.v[D] = fma(w, w, acc.v[D]);
        const bool near = in && phi_near(sg, del);
        if (__any_sync(0xffffffffu, near)) {
            double F;
            PhiLog G;
            phi_eval<SCALARS>(tab, sg, del, near, F, G);
            if constexpr (SCALARS) {
                acc.v[D + 1] = fma(F, del, acc.v[D + 1]);
                acc.v[D + 2] = fma(G.slope, G.t, acc.v[D + 2]) + G.g0;
            }
            w = fma(F, sg.neg_s, w);
        }
        const bool tiny = in && !near && phi_tiny(sg, w);
        if (__any_sync(0xffffffffu, tiny)) {
            double F, G;
            phi_far<SCALARS>(sg, del, w, tiny, F, G);
            if constexpr (SCALARS) {
                acc.v[D + 1] = fma(F, del, acc.v[D + 1]);
                acc.v[D + 2] += G;
            }
            w = fma(F, sg.neg_s, w);
        }
        w *= inv;
#pragma unroll
        for (int k = 0; k < D; ++k) acc.v[k] = fma(w, dl[k], acc.v[k]);
    }
}

template <int D>
__global__ void __launch_bounds__(kNaThreads, 3) noalloc_rows_kernel(int64_t n, const float *y, int64_t ld,
                                                                     const double *x, Sigma64 sg, double *grad,
                                                                     double *part) {
    constexpr int V = D + 3, P = Pow2<V>::value;
    extern __shared__ __align__(16) unsigned char na_smem[];
    double *tab = reinterpret_cast<double *>(na_smem);
    __shared__ double red[kNaWarps][V];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    phi_table_load(tab);
    __syncthreads();
    double scalar = 0.0;  // threads D .. D + 2: the block's sums of the scalar terms
    for (int64_t i = blockIdx.x; i < n; i += gridDim.x) {
        RowSums<D> acc;
#pragma unroll
        for (int q = 0; q < P; ++q) acc.v[q] = 0.0;
        double xi[D];
#pragma unroll
        for (int k = 0; k < D; ++k) xi[k] = x[i * D + k];
        const float *yrow = y + i * ld;
        row_part<D, false>(tab, sg, xi, x, yrow, 0, i, acc);
        row_part<D, true>(tab, sg, xi, x, yrow, i + 1, n, acc);
        lane_reduce<P, 5>(acc.v, lane, 0);
        bool writer;
        const int base = reduced_base<P, 5>(lane, 0, writer);
        if (writer && base < V) red[warp][base] = acc.v[0];
        __syncthreads();
        if (tid < V) {
            double v = red[0][tid];
#pragma unroll
            for (int w = 1; w < kNaWarps; ++w) v += red[w][tid];
            if (tid < D)
                grad[i * D + tid] = sg.inv_s * sg.inv_s * v;
            else
                scalar += v;
        }
        __syncthreads();  // red is free for the next row
    }
    if (tid >= D && tid < V) part[blockIdx.x * kNaParts + tid - D] = scalar;
}

// Sums the per-block partials in a fixed order into the three final slots.
__global__ void noalloc_sum_kernel(int nblocks, double *part) {
    __shared__ double sm[3][256];
    double acc[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < nblocks; b += 256)
        for (int q = 0; q < 3; ++q) acc[q] += part[b * kNaParts + q];
    for (int q = 0; q < 3; ++q) sm[q][threadIdx.x] = acc[q];
    __syncthreads();
    for (int o = 128; o >= 1; o >>= 1) {
        if (threadIdx.x < o)
            for (int q = 0; q < 3; ++q) sm[q][threadIdx.x] += sm[q][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x < 3) part[kNaMaxBlocks * kNaParts + threadIdx.x] = sm[threadIdx.x][0];
}

// CTAs for n rows: k per SM, k = 3 (as many as the table leaves room for) or 2.
// An SM's FP64 pipes are shared, so its time is k times its largest CTA's
// number of rows, ceil(n / (k SMs)): the k with the smaller product, more CTAs
// (latency) where they are equal.
int64_t row_blocks(int64_t n, int sms) {
    int64_t best = 0, cost = 0;
    for (int64_t k = 3; k >= 2; --k) {
        const int64_t c = k * ((n + k * sms - 1) / (k * sms));
        if (best == 0 || c < cost) {
            best = k;
            cost = c;
        }
    }
    return std::min<int64_t>(n, std::min<int64_t>(best * sms, kNaMaxBlocks));
}

template <int D>
cudaError_t raise_smem_d() {
    return cudaFuncSetAttribute(noalloc_rows_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPhiBytes);
}

// The kernels' shared memory limit, for every D at once: a later call neither
// sets an attribute nor grows a host table.
cudaError_t raise_smem_all() {
    cudaError_t (*const raise[])() = {raise_smem_d<1>, raise_smem_d<2>, raise_smem_d<3>, raise_smem_d<4>,
                                      raise_smem_d<5>, raise_smem_d<6>, raise_smem_d<7>, raise_smem_d<8>};
    for (auto f : raise) {
        const cudaError_t e = f();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Device address of the scratch array on the current device (looked up once
// per device; host code cannot use the symbol itself as a device pointer).
int scratch_address(double **out, int *sms) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        mds::set_thread_error("mds_loglik_grad_noalloc: cudaGetDevice: %s", cudaGetErrorString(e));
        return MDS_ERR_CUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) {
        mds::set_thread_error("mds_loglik_grad_noalloc: device ordinal %d beyond %d", dev, kMaxDevices);
        return MDS_ERR_UNSUPPORTED;
    }
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p) {
            mds::set_thread_error("mds_loglik_grad_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
            return MDS_ERR_CUDA;
        }
        e = cudaDeviceGetAttribute(&g_na_sms[dev], cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) {
            mds::set_thread_error("mds_loglik_grad_noalloc: cudaDeviceGetAttribute: %s", cudaGetErrorString(e));
            return MDS_ERR_CUDA;
        }
        e = raise_smem_all();
        if (e != cudaSuccess) {
            mds::set_thread_error("mds_loglik_grad_noalloc: shared memory: %s", cudaGetErrorString(e));
            return MDS_ERR_CUDA;
        }
        g_na_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_na_ptr[dev];
    *sms = g_na_sms[dev];
    return MDS_OK;
}

}  // namespace
}  // namespace mds

using namespace mds;

extern "C" int mds_loglik_grad_noalloc(int64_t n, int32_t d, const float *y, int64_t ld, const double *x,
                                       double sigma, double *grad, double *loglik, double *dlogl_dsigma,
                                       void *stream) {
    if (n < 2 || d < 1 || d > MDS_MAX_D || !y || !x || !grad || ld < n || !(sigma > 0.0) || !std::isfinite(sigma)) {
        mds::set_thread_error("mds_loglik_grad_noalloc: invalid argument (need 2 <= N, 1 <= D <= %d, ld >= N, "
                              "sigma > 0, non-NULL y, x, grad)", MDS_MAX_D);
        return MDS_ERR_INVALID_ARG;
    }
    if (n > kNaMaxN) {
        mds::set_thread_error("mds_loglik_grad_noalloc: N = %lld exceeds the maximum %lld of the fixed scratch",
                              static_cast<long long>(n), static_cast<long long>(kNaMaxN));
        return MDS_ERR_INVALID_ARG;
    }
    double *part = nullptr;
    int sms = 0;
    int st = scratch_address(&part, &sms);
    if (st != MDS_OK) return st;
    const int64_t nblocks = row_blocks(n, sms);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const Sigma64 sg = sigma64(sigma);
    switch (d) {
#define MDS_NA_CASE(DD)                                                                                           \
    case DD:                                                                                                      \
        noalloc_rows_kernel<DD>                                                                                   \
            <<<static_cast<int>(nblocks), kNaThreads, kPhiBytes, s>>>(n, y, ld, x, sg, grad, part);              \
        break;
        MDS_NA_CASE(1) MDS_NA_CASE(2) MDS_NA_CASE(3) MDS_NA_CASE(4)
        MDS_NA_CASE(5) MDS_NA_CASE(6) MDS_NA_CASE(7) MDS_NA_CASE(8)
#undef MDS_NA_CASE
        default: break;
    }
    noalloc_sum_kernel<<<1, 256, 0, s>>>(static_cast<int>(nblocks), part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        mds::set_thread_error("mds_loglik_grad_noalloc: launch: %s", cudaGetErrorString(e));
        return MDS_ERR_CUDA;
    }
    if (loglik || dlogl_dsigma) {
        double sums[3];
        e = cudaMemcpyAsync(sums, part + kNaMaxBlocks * kNaParts, sizeof(sums), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            mds::set_thread_error("mds_loglik_grad_noalloc: %s", cudaGetErrorString(e));
            return MDS_ERR_CUDA;
        }
        const double m = 0.5 * static_cast<double>(n) * static_cast<double>(n - 1);
        const double sum_r = sums[0] / (2.0 * sigma * sigma) + sums[2];
        const double ll = -m * std::log(sigma) - sum_r;
        const double ds = -m / sigma + sums[0] / (sigma * sigma * sigma) + sums[1] / (sigma * sigma);
        if (loglik) *loglik = ll;
        if (dlogl_dsigma) *dlogl_dsigma = ds;
        if (!std::isfinite(ll) || !std::isfinite(ds)) {
            mds::set_thread_error("mds_loglik_grad_noalloc: non-finite result");
            return MDS_ERR_NONFINITE;
        }
    }
    return MDS_OK;
}
