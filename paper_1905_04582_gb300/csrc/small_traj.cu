// Whole trajectories of a small problem in one launch: a cluster of 16 CTAs
// keeps the tiles of Y, the split locations, positions, momenta and gradients
// in shared memory and runs HMC iterations (arXiv:1905.04582, section 2.3,
// Eq. (6)-(9)): momentum draw, half kick and drift, an evaluation of the
// gradient per step with the leapfrog update, the energies, and the
// Metropolis decision, from which every CTA goes on to the next iteration.
//
// At these sizes a step as two launches (pair pass, reduction) is latency:
// the hand-overs, the table of chunks, the rings' first copies, the partial
// sums' way through L2; and the trajectory's start and end are two launches
// more.  Here a step is the pair arithmetic of half a quarter tile (32 rows x
// 16 columns) per warp, the tile functions of the chunked pass, so the same
// terms; a cluster barrier; the gather of each item's partial sums out of the
// CTAs' shared memory (16 lanes an item, double-float sums as in the
// reduction); the update, the new split locations written into all 16 CTAs (a
// lane each); and a second cluster barrier.  Halves rather than whole quarter
// tiles: the chain of one unit is what a step waits for (quarter tiles took
// 3.8 us a step at N = 200, D = 2).  What bounds it: the latency of that chain
// and of the two barriers for the smallest problems, the FP32 pipes of 16 SMs
// for the largest, which is where the rule ends (small_traj_fits).
// Measured (GB300, a step inside an HMC iteration, this kernel against pass
// and reduction): N = 200 at D = 1, 2, 3, 6: 3.2, 4.1, 5.2, 8.0 us against
// 4.9, 6.0, 6.9, 9.7; N = 50, D = 2: 2.6 against 6.0; start and end of an
// iteration: about 5 against 18 us.  10 iterations of 10 steps at N = 200,
// D = 2, the whole call: 818 -> 540 us.
#include <cooperative_groups.h>

#include <cstdint>

#include "chunk_tile.cuh"
#include "df.cuh"
#include "mds_internal.h"
#include "pair_math.cuh"
#include "philox.cuh"

namespace mds {
namespace {

namespace cg = cooperative_groups;

constexpr int kStCtas = 16;  // CTAs of the cluster (and lanes per item)
constexpr int kStMaxUnits = (8 * kStMaxBlocks * (kStMaxBlocks + 1) / 2 + kStCtas - 1) / kStCtas;
constexpr int kUnitElems = kWarpTileElems / 2;
constexpr int kUnitRows = kTile / 2;

// 128 registers at 16 warps hold the bodies up to D = 4.
template <int D>
__host__ __device__ constexpr int st_warps() {
    return D <= 4 ? 16 : 8;
}

// What the CTAs exchange at a trajectory's end, a row per CTA.
enum StPart : int { kPartKe0 = 0, kPartXx0, kPartKe1, kPartXx1, kPartE2, kPartMd, kPartLp, kPartXmax, kStParts };

// Shared memory of a CTA: its units of Y, their row and column sums, all
// split locations, and the state of the items it updates.
struct StLayout {
    int units, slots, xi, xj, y, rowp, colp, own, g0, g1, bytes;
    __host__ __device__ StLayout(int nt, int d) {
        units = (8 * nt * (nt + 1) / 2 + kStCtas - 1) / kStCtas;
        slots = (nt * kTile + kStCtas - 1) / kStCtas;
        xi = 0;                                  // [nt][d][32] float4
        xj = xi + nt * d * 32 * 16;              // [nt * 64][d] float2
        y = xj + nt * kTile * d * 8;             // [units][512]
        rowp = y + units * kUnitElems * 4;       // [units][32][d]
        colp = rowp + units * kUnitRows * d * 4; // [units][16][d]
        own = colp + units * kWarpCols * d * 4;  // x, p, x at the start: [3][slots * d]
        g0 = own + slots * 3 * d * 4;            // gradient at the start (hi, lo): [slots * d] float2
        g1 = g0 + slots * d * 8;                 // gradient at the end
        bytes = g1 + slots * d * 8;
    }
};

// Sum of a double-float over the warp into sm[i] (the caller adds the warps'
// parts after a barrier).
template <int W>
__device__ __forceinline__ void warp_part(DF v, DF (*sm)[W], int i) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) df_add(v, df_shfl_xor(v, o));
    if ((threadIdx.x & 31) == 0) sm[i][threadIdx.x >> 5] = v;
}

template <int D>
__global__ void __launch_bounds__(32 * st_warps<D>(), 1) small_traj_kernel(const __grid_constant__ SmallTrajArgs a) {
    constexpr bool kTall = D <= 2;
    constexpr int kNQ = kTall ? 4 : 2;  // row pairs per lane of a unit
    constexpr int kWarps = st_warps<D>(), kThreads = 32 * kWarps;
    extern __shared__ __align__(128) unsigned char smem[];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank());
    const int tid = static_cast<int>(threadIdx.x), warp = tid >> 5, lane = tid & 31;
    const PairArgs &pa = a.pair;
    const ReduceArgs &ra = a.reduce;
    const TrajArgs &ta = a.traj;
    const AcceptArgs &ac = a.accept;
    const int nt = pa.nt;
    const int n = static_cast<int>(pa.n);
    const StLayout L(nt, D);
    float4 *const xi_s = reinterpret_cast<float4 *>(smem + L.xi);
    float2 *const xj_s = reinterpret_cast<float2 *>(smem + L.xj);
    float *const y_s = reinterpret_cast<float *>(smem + L.y);
    float *const rowp_s = reinterpret_cast<float *>(smem + L.rowp);
    float *const colp_s = reinterpret_cast<float *>(smem + L.colp);
    const int sd = L.slots * D;
    float *const x_s = reinterpret_cast<float *>(smem + L.own), *const p_s = x_s + sd, *const x0_s = p_s + sd;
    float2 *const g0_s = reinterpret_cast<float2 *>(smem + L.g0), *const g1_s = reinterpret_cast<float2 *>(smem + L.g1);
    __shared__ float box_s[kWarps][2 * D];
    __shared__ short4 unit_s[kStMaxUnits];  // row block, column block, half, quarter of each local unit
    __shared__ DF part_s[kStParts][kWarps];
    __shared__ double all_s[kStCtas][kStParts];  // every CTA's sums
    __shared__ double sum_s[kStParts];
    __shared__ double logu_s;
    __shared__ int keep_s;
    const int units_all = 8 * nt * (nt + 1) / 2;
    pdl_trigger();
    // unit u: tile u / 8, rows 32 ((u / 4) % 2) on, quarter u % 4; local unit u / 16 of CTA u % 16.
    // Y does not change: it may stream in while the kernel before drains
    for (int l = tid; rank + l * kStCtas < units_all; l += kThreads) {
        const int u = rank + l * kStCtas, t = u >> 3;
        int I = 0;
        while (I + 1 < nt && tile_index(I + 1, I + 1, nt) <= t) ++I;
        unit_s[l] = make_short4(static_cast<short>(I), static_cast<short>(I + (t - tile_index(I, I, nt))),
                                static_cast<short>((u >> 2) & 1), static_cast<short>(u & 3));
    }
    for (int l = warp; rank + l * kStCtas < units_all; l += kWarps) {
        const int u = rank + l * kStCtas;
        const float4 *src = reinterpret_cast<const float4 *>(pa.y + static_cast<int64_t>(u >> 3) * kTileElems +
                                                             (u & 3) * kWarpTileElems + ((u >> 2) & 1) * kUnitElems);
        float4 *dst = reinterpret_cast<float4 *>(y_s + l * kUnitElems);
#pragma unroll
        for (int i = 0; i < kUnitElems / 4 / 32; ++i) dst[i * 32 + lane] = src[i * 32 + lane];
    }
    pdl_wait();
    Split sp = *ra.xs.split;
    const int64_t iter0 = ta.counters[kIter], il0 = ta.counters[kIterLocal];
    double ll = ac.scal[kLogLik], sum_r = ac.scal[kSumR], ds = ac.scal[kDSigma];  // at the current x
    const double prior = ac.scal[kPriorLogp];
    for (int i = tid; i < nt * D * 32; i += kThreads) xi_s[i] = __ldcg(pa.xrow + i);
    for (int i = tid; i < nt * kTile * D; i += kThreads) xj_s[i] = __ldcg(pa.xcol2 + i);
    // the slots this CTA updates: [k0, k1), 16 lanes each in the gather
    const int per = (n + kStCtas - 1) / kStCtas;
    const int k0 = min(n, rank * per), k1 = min(n, k0 + per), nown = (k1 - k0) * D;
    const int sub = lane & 15, grp = tid >> 4;
    for (int e = tid; e < nown; e += kThreads) {
        const int k = k0 + e / D;
        const int64_t g = (ra.perm ? static_cast<int64_t>(ra.perm[k]) : k) * D + e % D;
        x_s[e] = __ldcg(reinterpret_cast<const float *>(ra.xs.x) + g);
        p_s[e] = __ldcg(reinterpret_cast<const float *>(ra.p) + g);
        g0_s[e] = __ldcg(reinterpret_cast<const float2 *>(ra.grad) + g);
    }
    const int tla = lane & 3, tlb = lane >> 2;
    const int ybe = (tlb & 1) * 32 + 8 * (tlb >> 1) + (tla | ((tlb & 1) << 2));
    const int ybo = (tlb & 1) * 32 + 8 * (tlb >> 1) + (tla | ((~tlb & 1) << 2));
    const bool ragged = n % kTile != 0;
    const float eps = static_cast<float>(ra.eps), half_eps = static_cast<float>(0.5 * ra.eps);
    const float lambda = static_cast<float>(ra.lambda);
    float xmax = 0.f;
    unsigned bits = 0;  // error bits
    int64_t accepted = 0;
    // split locations of coordinate d of slot k into CTA r
    auto push = [&](int k, int d, int r, float v) {
        const float h = __fsub_rn(__fadd_rn(v, sp.magic), sp.magic);  // nearest multiple of q
        const float lo = __fsub_rn(v, h);                              // exact
        float *q = reinterpret_cast<float *>(cluster.map_shared_rank(xi_s, r)) +
                   (((k >> 6) * D + d) * 32 + ((k >> 1) & 31)) * 4 + (k & 1);
        q[0] = h;
        q[2] = lo;
        cluster.map_shared_rank(xj_s, r)[k * D + d] = make_float2(-h, -lo);
    };
    cluster.sync();
    for (int it = 0; it < a.n_iter; ++it) {
        // ---- start: momenta, energies, half kick and drift
        {
            DF ke{}, xx{};
            for (int e = tid; e < nown; e += kThreads) {
                const int k = k0 + e / D;
                const int64_t g = (ra.perm ? static_cast<int64_t>(ra.perm[k]) : k) * D + e % D;
                float p;
                if (ta.momentum_src == 1) {
                    uint32_t c[4] = {static_cast<uint32_t>(g >> 2), static_cast<uint32_t>(iter0 + it), ta.chain, 0u};
                    philox10(c, ta.seed);
                    float z0, z1;
                    if (g & 2)
                        box_muller(c[2], c[3], z0, z1);
                    else
                        box_muller(c[0], c[1], z0, z1);
                    p = (g & 1) ? z1 : z0;
                } else if (ta.momentum_src == 2) {
                    p = static_cast<float>(ta.p_inj[(il0 + it) * n * D + g]);
                } else {
                    p = p_s[e];
                }
                const float x = x_s[e];
                df_add(ke, 0.5f * p * p);
                df_add(xx, x * x);
                const float tg = __fadd_rn(g0_s[e].x, g0_s[e].y) - lambda * x;
                p = p + half_eps * tg;
                const float xn = x + eps * p;
                x0_s[e] = x;
                p_s[e] = p;
                x_s[e] = xn;
                xmax = fmaxf(xmax, fabsf(xn));
            }
            warp_part(ke, part_s, kPartKe0);
            warp_part(xx, part_s, kPartXx0);
            __syncthreads();
            for (int e = tid; e < nown * kStCtas; e += kThreads) {
                const int i = e / kStCtas;
                push(k0 + i / D, i % D, e % kStCtas, x_s[i]);
            }
        }
        cluster.sync();
        for (int step = 0; step < a.n_steps; ++step) {
            const bool last = step + 1 == a.n_steps;
            // log u for the decision, by a warp that mostly has no unit (FP64: long)
            if (step == 0 && ac.metropolis && tid == kThreads - 32) {
                double u;
                if (ac.u_src == 2) {
                    u = ac.u_inj[il0 + it];
                } else {
                    uint32_t c[4] = {0u, static_cast<uint32_t>(iter0 + it), ac.chain, 1u};
                    philox10(c, ac.seed);
                    u = open_unit(c[0]);
                }
                logu_s = log(u);
            }
            // ---- the units of this CTA
            DF se{}, sm{}, sl{};
            for (int l = warp; rank + l * kStCtas < units_all; l += kWarps) {
                const short4 un = unit_s[l];
                const int I = un.x, J = un.y, h = un.z, w = un.w;
                const float4 *ys = reinterpret_cast<const float4 *>(y_s + l * kUnitElems);
                const float2 *xjs = xj_s + (J * kTile + w * kWarpCols) * D;
                const float4 *xis = xi_s + I * 32 * D;
                float *rp = rowp_s + l * kUnitRows * D, *cp = colp_s + l * kWarpCols * D;
                float2 racc[kNQ][D];
#pragma unroll
                for (int q = 0; q < kNQ; ++q)
#pragma unroll
                    for (int k = 0; k < D; ++k) racc[q][k] = f2(0.f, 0.f);
                float2 e2 = f2(0.f, 0.f), md = f2(0.f, 0.f), prod = f2(1.f, 1.f);
                const bool masked =
                    J == I || (ragged && J == nt - 1) || (pa.tile_ho && pa.tile_ho[tile_index(I, J, nt)]);
                const int row_rel = (I - J) * kTile + h * kUnitRows;
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
                xis += h * (kUnitRows / 2);
                if constexpr (kTall) {
                    if (masked)
                        tile_tall<D, true, true, kNQ>(pa, ys, xjs, xis, lane, ybe, ybo, row_rel, w * kWarpCols, ncv,
                                                      racc, cp, e2, md, prod, box_s[warp]);
                    else
                        tile_tall<D, false, false, kNQ>(pa, ys, xjs, xis, lane, ybe, ybo, row_rel, w * kWarpCols, ncv,
                                                        racc, cp, e2, md, prod, box_s[warp]);
                    flush_rows_tall<D, kNQ>(racc, lane, rp);
                } else {
                    if (masked)
                        tile_chunk<D, true, true, kNQ>(pa, ys, xjs, xis, lane, row_rel, w * kWarpCols, ncv, racc, cp,
                                                       e2, md, prod, box_s[warp]);
                    else
                        tile_chunk<D, false, false, kNQ>(pa, ys, xjs, xis, lane, row_rel, w * kWarpCols, ncv, racc,
                                                         cp, e2, md, prod, box_s[warp]);
                    flush_rows<D, kNQ>(racc, lane, rp);
                }
                if (last) {
                    df_add(se, e2.x + e2.y);
                    df_add(sm, md.x + md.y);
                    // one log2 for the unit's 16 values of 1/Phi (at most 2 each): as many as the pass takes
                    df_add(sl, lg2_approx(prod.x * prod.y));
                }
            }
            if (last) {
                warp_part(se, part_s, kPartE2);
                warp_part(sm, part_s, kPartMd);
                warp_part(sl, part_s, kPartLp);
            }
            cluster.sync();
            // ---- each item's sums, update, and the new locations to every CTA
            DF ke{}, xx{};
            for (int kb = k0; kb < k1; kb += kThreads / 16) {
                const int k = kb + grp;
                const bool in = k < k1;
                DF acc[D];
#pragma unroll
                for (int d = 0; d < D; ++d) acc[d] = DF{0.f, 0.f};
                if (in) {
                    // row partials: 4 quarters of each tile of the row block; column partials: both halves of each
                    // tile above
                    const int B = k >> 6, r = k & (kTile - 1);
                    const int t0 = static_cast<int>(tile_index(B, B, nt)), R = 4 * (nt - B), C = 2 * (B + 1);
#pragma unroll 4
                    for (int i = sub; i < R + C; i += 16) {
                        int u;
                        const float *src;
                        float sign;
                        if (i < R) {
                            u = 8 * (t0 + (i >> 2)) + 4 * (r >> 5) + (i & 3);
                            src = rowp_s + ((u >> 4) * kUnitRows + (r & 31)) * D;
                            sign = -1.f;
                        } else {
                            u = 8 * static_cast<int>(tile_index((i - R) >> 1, B, nt)) + 4 * ((i - R) & 1) + (r >> 4);
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
                    const int e = (k - k0) * D;
#pragma unroll
                    for (int d = 0; d < D; ++d) {
                        const DF v = df_mul(acc[d], ra.part_scale_df);
                        if (!isfinite(v.hi)) bits |= kErrNonfinite;
                        const float x = x_s[e + d];
                        const float tg = v.hi - lambda * x;
                        if (last) {
                            const float p = p_s[e + d] + half_eps * tg;
                            p_s[e + d] = p;
                            g1_s[e + d] = make_float2(v.hi, v.lo);
                            df_add(ke, 0.5f * p * p);
                            df_add(xx, x * x);
                        } else {
                            const float p = p_s[e + d] + eps * tg;
                            xn[d] = x + eps * p;
                            p_s[e + d] = p;
                            x_s[e + d] = xn[d];
                            xmax = fmaxf(xmax, fabsf(xn[d]));
                        }
                    }
                }
                if (!last) {
#pragma unroll
                    for (int d = 0; d < D; ++d) xn[d] = __shfl_sync(0xffffffffu, xn[d], lane & 16);
                    if (in) {
#pragma unroll
                        for (int d = 0; d < D; ++d) push(k, d, sub, xn[d]);
                    }
                }
            }
            if (last) {
                warp_part(ke, part_s, kPartKe1);
                warp_part(xx, part_s, kPartXx1);
                float m = xmax;
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                if (lane == 0) part_s[kPartXmax][warp] = DF{m, 0.f};
                __syncthreads();
                // this CTA's sums to every CTA: thread (part, CTA)
                if (tid < kStParts * kStCtas) {
                    const int i = tid / kStCtas, r = tid % kStCtas;
                    DF t = part_s[i][0];
#pragma unroll
                    for (int w = 1; w < kWarps; ++w) {
                        if (i == kPartXmax)
                            t.hi = fmaxf(t.hi, part_s[i][w].hi);
                        else
                            df_add(t, part_s[i][w]);
                    }
                    *cluster.map_shared_rank(&all_s[rank][i], r) = static_cast<double>(t.hi) + static_cast<double>(t.lo);
                }
            }
            cluster.sync();
        }
        // ---- end: the same sums in every CTA, so the same decision
        if (warp < kStParts) {
            double v = all_s[lane & 15][warp];
#pragma unroll
            for (int o = 8; o >= 1; o >>= 1) {
                const double w = __shfl_xor_sync(0xffffffffu, v, o);
                v = warp == kPartXmax ? fmax(v, w) : v + w;
            }
            if (lane == 0) sum_s[warp] = v;
        }
        __syncthreads();
        constexpr double kLn2 = 0.69314718055994530942, kSqrt2Pi = 2.50662827463100050242;
        const double isg = ra.inv_sigma, isg2 = isg * isg;
        // (the scalar terms of the reduction, see reduce_body)
        double r1 = 0.0, l1 = 0.0, d1 = 0.0, dh = 0.0;
        if (tid == 0) {
            r1 = 0.5 * sum_s[kPartE2] * isg2 - kLn2 * sum_s[kPartLp];
            l1 = -ra.m_pairs * ra.log_sigma - r1;
            const double h0 = -(ll - 0.5 * ra.lambda * sum_s[kPartXx0] + prior) + sum_s[kPartKe0];
            const double h1 = -(l1 - 0.5 * ra.lambda * sum_s[kPartXx1] + prior) + sum_s[kPartKe1];
            dh = h1 - h0;
            keep_s = !ac.metropolis || (isfinite(dh) && logu_s < -dh) ? 1 : 0;
        }
        __syncthreads();
        const int keep = keep_s;
        if (tid == 0) {
            if (!isfinite(l1) || !isfinite(dh)) bits |= kErrNonfinite;
            if (rank == 0) {
                d1 = -ra.m_pairs * isg + sum_s[kPartE2] * isg2 * isg + sum_s[kPartMd] / kSqrt2Pi * isg2;
                if (!isfinite(d1)) bits |= kErrNonfinite;
                if (keep) {
                    sum_r = r1;
                    ds = d1;
                }
                accepted += keep;
                ac.scal[kLastDH] = dh;
                const int64_t il = il0 + it;
                if (ac.acc_out || ac.dh_out) {
                    if (il >= 0 && il < ac.out_cap) {
                        if (ac.acc_out) ac.acc_out[il] = keep;
                        if (ac.dh_out) ac.dh_out[il] = dh;
                    } else {
                        bits |= kErrOverflow;
                    }
                }
            }
            if (keep) ll = l1;
        }
        for (int e = tid; e < nown; e += kThreads) {
            if (keep)
                g0_s[e] = g1_s[e];
            else
                x_s[e] = x0_s[e];
        }
        // the split quantum grows when the trajectory outgrew its bound (the same rule in every CTA)
        const float m = static_cast<float>(sum_s[kPartXmax]);
        if (m > sp.bound) {
            Split ns;
            if (choose_split(m, D, ns))
                sp = ns;
            else
                bits |= kErrRange;
        }
        __syncthreads();
    }
    // ---- the state back, from this CTA's items
    if (bits) atomicOr(ra.err, bits);
    for (int e = tid; e < nown; e += kThreads) {
        const int k = k0 + e / D, d = e % D;
        const int64_t g = (ra.perm ? static_cast<int64_t>(ra.perm[k]) : k) * D + d;
        reinterpret_cast<float *>(ra.xs.x)[g] = x_s[e];
        reinterpret_cast<float *>(ra.p)[g] = p_s[e];
        reinterpret_cast<float2 *>(ra.grad)[g] = g0_s[e];
        write_split_slot(ra.xs, sp, k, D, d, x_s[e]);
    }
    if (tid == 0 && rank == 0) {
        *ra.xs.split = sp;
        atomicMax(ra.xs.xmax_bits, __float_as_uint(static_cast<float>(sum_s[kPartXmax])));
        ac.scal[kLogLik] = ll;
        ac.scal[kLogLikEnd] = ll;
        ac.scal[kSumR] = sum_r;
        ac.scal[kDSigma] = ds;
        if (ac.metropolis) {
            ta.counters[kIter] = iter0 + a.n_iter;
            ta.counters[kIterLocal] = il0 + a.n_iter;
            ta.counters[kAccepted] += accepted;
        }
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
    cfg.blockDim = dim3(32 * st_warps<D>());
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
    cfg.blockDim = dim3(32 * st_warps<D>());
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

// The rule: up to the number of row blocks at which a trajectory here takes
// less time than one over the whole chip.  A step, us, here against there:
// D = 1, N = 400 4.6 / 5.2, N = 576 6.7 / 5.0; D = 2, N = 300 5.3 / 6.0,
// N = 400 6.9 / 5.9; D = 3, N = 300 6.8 / 7.0, N = 400 9.3 / 6.9; D = 4,
// N = 200 6.6 / 8.1, N = 300 8.9 / 7.8; D = 6, N = 200 8.0 / 9.7, N = 300
// 11.7 / 9.9; D = 8, N = 200 10.8 / 11.9, N = 300 15.5 / 12.3; start and end
// of a trajectory add about 5 here and 18 there.
bool small_traj_fits(int64_t nt, int d) {
    if (d < 1 || d > 8 || nt > (d == 1 ? 7 : d == 2 ? 6 : d == 3 ? 5 : 4)) return false;
    if (StLayout(static_cast<int>(nt), d).bytes > kStMaxSmem) return false;
    MDS_ST_SWITCH(d, resident_d, static_cast<int>(nt))
    return false;
}

cudaError_t launch_small_traj(const SmallTrajArgs &a, int d, cudaStream_t s) {
    MDS_ST_SWITCH(d, launch_small_d, a, s)
    return cudaErrorInvalidValue;
}

}  // namespace mds
