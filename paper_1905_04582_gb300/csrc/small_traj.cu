// Steps of a trajectory of a small problem in one launch: a cluster of 16
// CTAs keeps the tiles of Y, the split locations, the positions and the
// momenta in shared memory and runs kick-drift steps, each an evaluation of
// the gradient (Eq. (9) of arXiv:1905.04582) and the leapfrog update
// (section 2.3, Eq. (7)).
//
// At these sizes a step as two launches (pair pass, reduction) is latency:
// the hand-overs, the table of chunks, the rings' first copies, the partial
// sums' way through L2.  Here a step is the pair arithmetic of one quarter
// tile after another per warp (the tile functions of the chunked pass, so the
// same terms), a cluster barrier, the gather of each item's partial sums out
// of the CTAs' shared memory (16 lanes an item, double-float sums as in the
// reduction), the update, the new split locations written into all 16 CTAs (a
// lane each), and a second cluster barrier.  What bounds it: the latency of
// one quarter tile's chain and of the two barriers for the smallest problems,
// the FP32 pipes of 16 SMs for the largest, which is where the rule ends
// (small_traj_fits).  Measured (GB300, a step inside an HMC iteration, this
// kernel against pass and reduction): N = 200 at D = 1, 2, 3, 6: 2.9, 3.8,
// 4.5, 8.7 us against 4.9, 5.9, 6.8, 9.4; N = 50, D = 2: 2.7 against 6.0.
#include <cooperative_groups.h>

#include <cstdint>

#include "chunk_tile.cuh"
#include "df.cuh"
#include "mds_internal.h"
#include "pair_math.cuh"

namespace mds {
namespace {

namespace cg = cooperative_groups;

constexpr int kStCtas = 16;      // CTAs of the cluster (and lanes per item)
constexpr int kStWarps = 8;      // warps per CTA
constexpr int kStThreads = 32 * kStWarps;
constexpr int kStMaxUnits = (4 * kStMaxBlocks * (kStMaxBlocks + 1) / 2 + kStCtas - 1) / kStCtas;

// Shared memory of a CTA: its quarter tiles of Y, their row and column sums,
// all split locations, and the state of the items it updates.
struct StLayout {
    int units, xi, xj, y, rowp, colp, own, bytes;
    __host__ __device__ StLayout(int nt, int d) {
        units = (4 * nt * (nt + 1) / 2 + kStCtas - 1) / kStCtas;
        const int slots = (nt * kTile + kStCtas - 1) / kStCtas;
        xi = 0;                                  // [nt][d][32] float4
        xj = xi + nt * d * 32 * 16;              // [nt * 64][d] float2
        y = xj + nt * kTile * d * 8;             // [units][1024]
        rowp = y + units * kWarpTileElems * 4;   // [units][64][d]
        colp = rowp + units * kTile * d * 4;     // [units][16][d]
        own = colp + units * kWarpCols * d * 4;  // [slots][2][d]: x, p
        bytes = own + slots * 2 * d * 4;
    }
};

template <int D>
__global__ void __launch_bounds__(kStThreads, 1) small_traj_kernel(const __grid_constant__ SmallTrajArgs a) {
    constexpr bool kTall = D <= 2;
    constexpr int kRP = kTall ? 8 : 4;
    extern __shared__ __align__(128) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank());
    const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, lane = tid & 31;
    const PairArgs &pa = a.pair;
    const ReduceArgs &ra = a.reduce;
    const int nt = pa.nt;
    const int n = static_cast<int>(pa.n);
    const StLayout L(nt, D);
    float4 *const xi_s = reinterpret_cast<float4 *>(smem + L.xi);
    float2 *const xj_s = reinterpret_cast<float2 *>(smem + L.xj);
    float *const y_s = reinterpret_cast<float *>(smem + L.y);
    float *const rowp_s = reinterpret_cast<float *>(smem + L.rowp);
    float *const colp_s = reinterpret_cast<float *>(smem + L.colp);
    float *const own_s = reinterpret_cast<float *>(smem + L.own);
    __shared__ float box_s[kStWarps][2 * D];
    __shared__ short2 ij_s[kStMaxUnits];  // row and column block of each local unit
    const int units_all = 4 * nt * (nt + 1) / 2;
    pdl_trigger();
    for (int l = tid; rank + l * kStCtas < units_all; l += kStThreads) {
        const int t = (rank + l * kStCtas) >> 2;
        int I = 0;
        while (I + 1 < nt && tile_index(I + 1, I + 1, nt) <= t) ++I;
        ij_s[l] = make_short2(static_cast<short>(I), static_cast<short>(I + (t - tile_index(I, I, nt))));
    }
    // unit u (quarter u % 4 of tile u / 4) is local unit u / 16 of CTA u % 16;
    // Y does not change: it may stream in while the kernel before drains
    for (int l = warp; rank + l * kStCtas < units_all; l += kStWarps) {
        const int u = rank + l * kStCtas;
        const float4 *src = reinterpret_cast<const float4 *>(pa.y + static_cast<int64_t>(u) * kWarpTileElems);
        float4 *dst = reinterpret_cast<float4 *>(y_s + l * kWarpTileElems);
#pragma unroll
        for (int i = 0; i < kWarpTileElems / 4 / 32; ++i) dst[i * 32 + lane] = src[i * 32 + lane];
    }
    const Split sp = *ra.xs.split;  // changes only at a trajectory's end and where the caller sets locations
    pdl_wait();
    for (int i = tid; i < nt * D * 32; i += kStThreads) xi_s[i] = __ldcg(pa.xrow + i);
    for (int i = tid; i < nt * kTile * D; i += kStThreads) xj_s[i] = __ldcg(pa.xcol2 + i);
    // the slots this CTA updates: [k0, k1), 16 lanes each
    const int per = (n + kStCtas - 1) / kStCtas;
    const int k0 = min(n, rank * per), k1 = min(n, k0 + per);
    const int sub = lane & 15, grp = tid >> 4;
    for (int k = k0 + grp; k < k1; k += kStThreads / 16) {
        if (sub < D) {
            const int64_t it = ra.perm ? ra.perm[k] : k;
            own_s[((k - k0) * 2 + 0) * D + sub] = __ldcg(reinterpret_cast<const float *>(ra.xs.x) + it * D + sub);
            own_s[((k - k0) * 2 + 1) * D + sub] = __ldcg(reinterpret_cast<const float *>(ra.p) + it * D + sub);
        }
    }
    const int tla = lane & 3, tlb = lane >> 2;
    const int ybe = (tlb & 1) * 32 + 8 * (tlb >> 1) + (tla | ((tlb & 1) << 2));
    const int ybo = (tlb & 1) * 32 + 8 * (tlb >> 1) + (tla | ((~tlb & 1) << 2));
    const bool ragged = n % kTile != 0;
    const float eps = static_cast<float>(ra.eps), lambda = static_cast<float>(ra.lambda);
    float xmax = 0.f;
    bool bad = false;
    cluster.sync();
    for (int step = 0; step < a.n_steps; ++step) {
        // ---- the quarter tiles of this CTA
        for (int l = warp; rank + l * kStCtas < units_all; l += kStWarps) {
            const int u = rank + l * kStCtas, t = u >> 2, w = u & 3;
            const int I = ij_s[l].x, J = ij_s[l].y;
            const float4 *ys = reinterpret_cast<const float4 *>(y_s + l * kWarpTileElems);
            const float2 *xjs = xj_s + (J * kTile + w * kWarpCols) * D;
            const float4 *xis = xi_s + I * 32 * D;
            float *rp = rowp_s + l * kTile * D, *cp = colp_s + l * kWarpCols * D;
            float2 racc[kRP][D];
#pragma unroll
            for (int q = 0; q < kRP; ++q)
#pragma unroll
                for (int k = 0; k < D; ++k) racc[q][k] = f2(0.f, 0.f);
            float2 e2 = f2(0.f, 0.f), md = f2(0.f, 0.f), prod = f2(1.f, 1.f);  // not used by these steps
            const bool masked = J == I || (ragged && J == nt - 1) || (pa.tile_ho && pa.tile_ho[t]);
            const int row_rel = (I - J) * kTile;
            const int64_t ncv = n - J * kTile;
            if (!masked) {
                float b[2 * D];
                row_box<D>(xis, lane, b);
                __syncwarp();
                if (lane == 0)
#pragma unroll
                    for (int i = 0; i < 2 * D; ++i) box_s[warp][i] = b[i];
                __syncwarp();
            }
            if constexpr (kTall) {
                if (masked)
                    tile_tall<D, true, true>(pa, ys, xjs, xis, lane, ybe, ybo, row_rel, w * kWarpCols, ncv, racc, cp,
                                             e2, md, prod, box_s[warp]);
                else
                    tile_tall<D, false, false>(pa, ys, xjs, xis, lane, ybe, ybo, row_rel, w * kWarpCols, ncv, racc,
                                               cp, e2, md, prod, box_s[warp]);
                flush_rows_tall<D>(racc, lane, rp);
            } else {
                if (masked)
                    tile_chunk<D, true, true>(pa, ys, xjs, xis, lane, row_rel, w * kWarpCols, ncv, racc, cp, e2, md,
                                              prod, box_s[warp]);
                else
                    tile_chunk<D, false, false>(pa, ys, xjs, xis, lane, row_rel, w * kWarpCols, ncv, racc, cp, e2, md,
                                                prod, box_s[warp]);
                flush_rows<D>(racc, lane, rp);
            }
        }
        cluster.sync();
        // ---- each item's sums, update, and the new locations to every CTA
        for (int kb = k0; kb < k1; kb += kStThreads / 16) {
            const int k = kb + grp;
            const bool in = k < k1;
            const int B = in ? k >> 6 : 0, r = k & (kTile - 1);
            DF acc[D];
#pragma unroll
            for (int d = 0; d < D; ++d) acc[d] = DF{0.f, 0.f};
            if (in) {
                // row partials: the 4 (nt - B) units of row block B, one after another
                const int ub = 4 * static_cast<int>(tile_index(B, B, nt)), R = 4 * (nt - B), C = B + 1;
#pragma unroll 4
                for (int i = sub; i < R + C; i += 16) {
                    int u;
                    const float *src;
                    float sign;
                    if (i < R) {
                        u = ub + i;
                        src = rowp_s + ((u >> 4) * kTile + r) * D;
                        sign = -1.f;
                    } else {
                        const int I = i - R;
                        u = 4 * static_cast<int>(tile_index(I, B, nt)) + (r >> 4);
                        src = colp_s + ((u >> 4) * kWarpCols + (r & 15)) * D;
                        sign = 1.f;
                    }
                    const float *rem = cluster.map_shared_rank(src, u & 15);
#pragma unroll
                    for (int d = 0; d < D; ++d) df_add(acc[d], sign * rem[d]);
                }
            }
#pragma unroll
            for (int o = 8; o >= 1; o >>= 1)
#pragma unroll
                for (int d = 0; d < D; ++d) df_add(acc[d], df_shfl_xor(acc[d], o));
            float xn[D];
            if (in && sub == 0) {
                float *own = own_s + (k - k0) * 2 * D;
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const DF v = df_mul(acc[d], ra.part_scale_df);
                    bad = bad || !isfinite(v.hi);
                    const float xv = own[d];
                    const float tg = v.hi - lambda * xv;
                    const float pn = own[D + d] + eps * tg;
                    xn[d] = xv + eps * pn;
                    own[d] = xn[d];
                    own[D + d] = pn;
                    xmax = fmaxf(xmax, fabsf(xn[d]));
                }
            }
#pragma unroll
            for (int d = 0; d < D; ++d) xn[d] = __shfl_sync(0xffffffffu, xn[d], lane & 16);
            if (in) {
                float *xr = reinterpret_cast<float *>(cluster.map_shared_rank(xi_s, sub));
                float2 *xc = cluster.map_shared_rank(xj_s, sub);
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    const float h = __fsub_rn(__fadd_rn(xn[d], sp.magic), sp.magic);  // nearest multiple of q
                    const float lo = __fsub_rn(xn[d], h);                              // exact
                    float *q = xr + ((B * D + d) * 32 + (r >> 1)) * 4 + (r & 1);
                    q[0] = h;
                    q[2] = lo;
                    xc[k * D + d] = make_float2(-h, -lo);
                }
            }
        }
        cluster.sync();
    }
    // ---- the state back: x, p, and the split layouts from this CTA's items
    if (bad) atomicOr(ra.err, kErrNonfinite);
    if (xmax > sp.bound) atomicMax(ra.xs.xmax_bits, __float_as_uint(xmax));
    for (int e = tid; e < (k1 - k0) * D; e += kStThreads) {
        const int k = k0 + e / D, d = e % D;
        const int64_t it = ra.perm ? ra.perm[k] : k;
        const float xv = own_s[(k - k0) * 2 * D + d];
        reinterpret_cast<float *>(ra.xs.x)[it * D + d] = xv;
        reinterpret_cast<float *>(ra.p)[it * D + d] = own_s[(k - k0) * 2 * D + D + d];
        write_split_slot(ra.xs, sp, k, D, d, xv);
    }
}

template <int D>
cudaError_t prepare_d(int smem) {
    const void *fn = reinterpret_cast<const void *>(small_traj_kernel<D>);
    cudaError_t e = raise_dyn_smem(fn, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

template <int D>
cudaError_t launch_small_d(const SmallTrajArgs &a, cudaStream_t s) {
    const int smem = StLayout(a.pair.nt, D).bytes;
    cudaError_t e = prepare_d<D>(smem);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kStCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kStCtas);
    cfg.blockDim = dim3(kStThreads);
    cfg.dynamicSmemBytes = static_cast<size_t>(smem);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, small_traj_kernel<D>, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// Whether a cluster can be resident on this device (16 SMs of one GPC).
template <int D>
bool resident_d(int nt) {
    const int smem = StLayout(nt, D).bytes;
    if (prepare_d<D>(smem) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kStCtas;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kStCtas);
    cfg.blockDim = dim3(kStThreads);
    cfg.dynamicSmemBytes = static_cast<size_t>(smem);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, small_traj_kernel<D>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters >= 1;
}

#define MDS_ST_SWITCH(D, F, ...)       \
    switch (D) {                       \
        case 1: return F<1>(__VA_ARGS__); \
        case 2: return F<2>(__VA_ARGS__); \
        case 3: return F<3>(__VA_ARGS__); \
        case 4: return F<4>(__VA_ARGS__); \
        case 5: return F<5>(__VA_ARGS__); \
        case 6: return F<6>(__VA_ARGS__); \
        case 7: return F<7>(__VA_ARGS__); \
        case 8: return F<8>(__VA_ARGS__); \
        default: break;                \
    }

}  // namespace

// The rule: up to the number of row blocks at which a step here still takes
// less time than a pass and a reduction over the whole chip (measured, us a
// step, here against there): D = 1, N = 400 4.6 / 5.2, N = 500 5.5 / 5.1;
// D = 2, N = 200 3.8 / 5.9, N = 300 6.0 / 6.1; D = 3, N = 200 4.5 / 6.8,
// N = 300 6.4 / 7.0; D = 4, N = 200 6.0 / 8.0, N = 300 8.3 / 7.9; D = 6,
// N = 100 5.5 / 9.8, N = 200 8.7 / 9.4; D = 8, N = 100 7.4 / 12.0, N = 200
// 11.3 / 11.9.
bool small_traj_fits(int64_t nt, int d) {
    if (d < 1 || d > 8 || nt > (d == 1 ? kStMaxBlocks : d <= 4 ? 4 : 3)) return false;
    if (StLayout(static_cast<int>(nt), d).bytes > kStMaxSmem) return false;
    MDS_ST_SWITCH(d, resident_d, static_cast<int>(nt))
    return false;
}

cudaError_t launch_small_traj(const SmallTrajArgs &a, int d, cudaStream_t s) {
    MDS_ST_SWITCH(d, launch_small_d, a, s)
    return cudaErrorInvalidValue;
}

}  // namespace mds
