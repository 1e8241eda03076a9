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
// What crosses between CTAs travels as one vector per item (a lane's access to
// another CTA is a packet of its own whatever its width): single floats took
// 4.1 us a step at N = 200, D = 2 and 8.0 at D = 6.
// Measured (GB300, a step inside an HMC iteration, this kernel against pass
// and reduction): N = 200 at D = 1, 2, 3, 6: 3.1, 3.5, 4.2, 5.0 us against
// 5.1, 5.9, 7.0, 9.8; N = 50, D = 2: 2.6 against 6.1; start and end of an
// iteration: 9 against 18 us.  10 iterations of 10 steps at N = 200, D = 2,
// the whole call: 818 -> 473 us.
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

// Floats between items in the arrays that other CTAs read or write: a lane's
// access to another CTA is a packet of its own whatever its width, so an
// item's coordinates travel as one vector (two beyond D = 4).
__host__ __device__ constexpr int st_stride(int d) { return d <= 2 ? d : d <= 4 ? 4 : 8; }

template <int D>
struct alignas(D == 1 ? 4 : D == 2 ? 8 : 16) StVec {
    float v[st_stride(D)];
};

// What the CTAs exchange at a trajectory's end, a row per CTA.
enum StPart : int { kPartKe0 = 0, kPartXx0, kPartKe1, kPartXx1, kPartE2, kPartMd, kPartLp, kPartXmax, kStParts };

// Shared memory of a CTA: its units of Y, their row and column sums, all
// split locations, and the state of the items it updates.
struct StLayout {
    int units, slots, xi, xj, xr, y, rowp, colp, own, g0, g1, bytes;
    __host__ __device__ StLayout(int nt, int d) {
        units = (8 * nt * (nt + 1) / 2 + kStCtas - 1) / kStCtas;
        slots = (nt * kTile + kStCtas - 1) / kStCtas;
        xi = 0;                                    // [nt][d][32] float4
        xj = xi + nt * d * 32 * 16;                // [nt * 64][d] float2
        const int st = st_stride(d);
        xr = xj + nt * kTile * d * 8;              // locations as the CTAs hand them over: [nt * 64][st]
        y = xr + nt * kTile * st * 4;              // [units][512]
        rowp = y + units * kUnitElems * 4;         // [units][32][st]
        colp = rowp + units * kUnitRows * st * 4;  // [units][16][st]
        own = colp + units * kWarpCols * st * 4;   // x, p, x at the start: [3][slots * d]
        g0 = own + slots * 3 * d * 4;              // gradient at the start (hi, lo): [slots * d] float2
        g1 = g0 + slots * d * 8;                   // gradient at the end
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

// L, sum r and dL/dsigma from the sums over all pairs (as reduce_body forms them).
struct StScalars {
    double ll, sum_r, ds;
};
__device__ __forceinline__ StScalars st_scalars(const ReduceArgs &ra, double e2, double md, double lp) {
    constexpr double kLn2 = 0.69314718055994530942, kInvSqrt2Pi = 0.39894228040143267794;
    const double isg = ra.inv_sigma, isg2 = isg * isg;
    StScalars t;
    t.sum_r = 0.5 * e2 * isg2 - kLn2 * lp;
    t.ll = -ra.m_pairs * ra.log_sigma - t.sum_r;
    t.ds = -ra.m_pairs * isg + e2 * isg2 * isg + md * kInvSqrt2Pi * isg2;
    return t;
}

// A CTA's part of the problem: its units, the arrays in shared memory, and the
// two halves of an evaluation.
template <int D>
struct SmallCta {
    static constexpr bool kTall = D <= 2;
    static constexpr int kNQ = kTall ? 4 : 2;  // row pairs per lane of a unit
    static constexpr int kS = st_stride(D);
    static constexpr int kWarps = st_warps<D>(), kThreads = 32 * kWarps;

    const PairArgs &pa;
    int rank, tid, warp, lane, nt, n, units_all;
    int k0, k1;  // the slots this CTA updates
    float4 *xi_s;
    float2 *xj_s;
    StVec<D> *xr_s, *rowp_s, *colp_s;
    float *y_s;
    float (*box_s)[2 * D];
    short4 *unit_s;

    __device__ __forceinline__ SmallCta(const PairArgs &a, const StLayout &L, unsigned char *smem, int rank_,
                                        float (*box)[2 * D], short4 *unit)
        : pa(a), rank(rank_), tid(static_cast<int>(threadIdx.x)), warp(tid >> 5), lane(tid & 31), nt(a.nt),
          n(static_cast<int>(a.n)), units_all(8 * a.nt * (a.nt + 1) / 2), box_s(box), unit_s(unit) {
        xi_s = reinterpret_cast<float4 *>(smem + L.xi);
        xj_s = reinterpret_cast<float2 *>(smem + L.xj);
        y_s = reinterpret_cast<float *>(smem + L.y);
        xr_s = reinterpret_cast<StVec<D> *>(smem + L.xr);
        rowp_s = reinterpret_cast<StVec<D> *>(smem + L.rowp);
        colp_s = reinterpret_cast<StVec<D> *>(smem + L.colp);
        const int per = (n + kStCtas - 1) / kStCtas;
        k0 = min(n, rank * per);
        k1 = min(n, k0 + per);
    }

    // Item of element e (slot, coordinate) of this CTA's slots, as an index into [N][D].
    __device__ __forceinline__ int64_t element(const int32_t *perm, int e) const {
        const int k = k0 + e / D;
        return (perm ? static_cast<int64_t>(perm[k]) : k) * D + e % D;
    }

    // The table of units and their Y.  Unit u: tile u / 8, rows
    // 32 ((u / 4) % 2) on, quarter u % 4; local unit u / 16 of CTA u % 16.  Y
    // does not change: it may stream in while the kernel before drains.
    __device__ __forceinline__ void stage_y() {
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
    }

    __device__ __forceinline__ void load_x() {
        for (int i = tid; i < nt * D * 32; i += kThreads) xi_s[i] = __ldcg(pa.xrow + i);
        for (int i = tid; i < nt * kTile * D; i += kThreads) xj_s[i] = __ldcg(pa.xcol2 + i);
    }

    // The split locations from the locations that the CTAs handed over.
    __device__ __forceinline__ void split_x(const Split &sp) {
        for (int e = tid; e < n * D; e += kThreads) {
            const int k = e / D, d = e % D;
            const float v = xr_s[k].v[d];
            const float h = __fsub_rn(__fadd_rn(v, sp.magic), sp.magic);  // nearest multiple of q
            const float lo = __fsub_rn(v, h);                              // exact
            float *q = reinterpret_cast<float *>(xi_s) + (((k >> 6) * D + d) * 32 + ((k >> 1) & 31)) * 4 + (k & 1);
            q[0] = h;
            q[2] = lo;
            xj_s[e] = make_float2(-h, -lo);
        }
        __syncthreads();
    }

    // The units of this CTA: row and column sums, and (scalars) the sums of
    // e^2, m' delta and log2(1 / Phi).
    __device__ __forceinline__ void units(bool scalars, DF &se, DF &sm, DF &sl) {
        const int tla = lane & 3, tlb = lane >> 2;
        const int ybe = (tlb & 1) * 32 + 8 * (tlb >> 1) + (tla | ((tlb & 1) << 2));
        const int ybo = (tlb & 1) * 32 + 8 * (tlb >> 1) + (tla | ((~tlb & 1) << 2));
        const bool ragged = n % kTile != 0;
        for (int l = warp; rank + l * kStCtas < units_all; l += kWarps) {
            const short4 un = unit_s[l];
            const int I = un.x, J = un.y, h = un.z, w = un.w;
            const float4 *ys = reinterpret_cast<const float4 *>(y_s + l * kUnitElems);
            const float2 *xjs = xj_s + (J * kTile + w * kWarpCols) * D;
            const float4 *xis = xi_s + I * 32 * D;
            float *rp = rowp_s[l * kUnitRows].v, *cp = colp_s[l * kWarpCols].v;
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
                    tile_tall<D, true, true, kNQ, kS>(pa, ys, xjs, xis, lane, ybe, ybo, row_rel, w * kWarpCols, ncv,
                                                  racc, cp, e2, md, prod, box_s[warp]);
                else
                    tile_tall<D, false, false, kNQ, kS>(pa, ys, xjs, xis, lane, ybe, ybo, row_rel, w * kWarpCols, ncv,
                                                    racc, cp, e2, md, prod, box_s[warp]);
                flush_rows_tall<D, kNQ, kS>(racc, lane, rp);
            } else {
                if (masked)
                    tile_chunk<D, true, true, kNQ, kS>(pa, ys, xjs, xis, lane, row_rel, w * kWarpCols, ncv, racc, cp,
                                                   e2, md, prod, box_s[warp]);
                else
                    tile_chunk<D, false, false, kNQ, kS>(pa, ys, xjs, xis, lane, row_rel, w * kWarpCols, ncv, racc,
                                                     cp, e2, md, prod, box_s[warp]);
                flush_rows<D, kNQ, kS>(racc, lane, rp);
            }
            if (scalars) {
                df_add(se, e2.x + e2.y);
                df_add(sm, md.x + md.y);
                // one log2 for the unit's 16 values of 1/Phi (at most 2 each): as many as the pass takes
                df_add(sl, lg2_approx(prod.x * prod.y));
            }
        }
    }

    // Sum of the partials of slot k over its 16 lanes (lane 0 of them has it),
    // in units of -sigma^2; every lane of the warp calls it.
    __device__ __forceinline__ void gather(const cg::cluster_group &cluster, int k, bool in, DF (&acc)[D]) const {
        const int sub = lane & 15;
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
                const StVec<D> *src;
                float sign;
                if (i < R) {
                    u = 8 * (t0 + (i >> 2)) + 4 * (r >> 5) + (i & 3);
                    src = rowp_s + (u >> 4) * kUnitRows + (r & 31);
                    sign = -1.f;
                } else {
                    u = 8 * static_cast<int>(tile_index((i - R) >> 1, B, nt)) + 4 * ((i - R) & 1) + (r >> 4);
                    src = colp_s + (u >> 4) * kWarpCols + (r & 15);
                    sign = 1.f;
                }
                const StVec<D> rem = *cluster.map_shared_rank(src, u & 15);
#pragma unroll
                for (int d = 0; d < D; ++d) df_add(acc[d], sign * rem.v[d]);
            }
        }
#pragma unroll
        for (int o = 8; o >= 1; o >>= 1)
#pragma unroll
            for (int d = 0; d < D; ++d) df_add(acc[d], df_shfl_xor(acc[d], o));
    }
};

template <int D>
__global__ void __launch_bounds__(32 * st_warps<D>(), 1) small_traj_kernel(const __grid_constant__ SmallTrajArgs a) {
    constexpr int kWarps = st_warps<D>(), kThreads = 32 * kWarps;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float box_s[kWarps][2 * D];
    __shared__ short4 unit_s[kStMaxUnits];  // row block, column block, half, quarter of each local unit
    cg::cluster_group cluster = cg::this_cluster();
    const TrajArgs &ta = a.traj;
    const AcceptArgs &ac = a.accept;
    const ReduceArgs &ra = a.reduce;
    const StLayout L(a.pair.nt, D);
    SmallCta<D> c(a.pair, L, smem, static_cast<int>(cluster.block_rank()), box_s, unit_s);
    const int rank = c.rank, tid = c.tid, warp = c.warp, lane = c.lane, n = c.n, k0 = c.k0, k1 = c.k1;
    const int nown = (k1 - k0) * D;
    const int sd = L.slots * D;
    float *const x_s = reinterpret_cast<float *>(smem + L.own), *const p_s = x_s + sd, *const x0_s = p_s + sd;
    float2 *const g0_s = reinterpret_cast<float2 *>(smem + L.g0), *const g1_s = reinterpret_cast<float2 *>(smem + L.g1);
    __shared__ DF part_s[kStParts][kWarps];
    __shared__ double all_s[kStCtas][kStParts];  // every CTA's sums
    __shared__ double sum_s[kStParts];
    __shared__ double logu_s;
    __shared__ int keep_s;
    pdl_trigger();
    c.stage_y();
    pdl_wait();
    Split sp = *ra.xs.split;
    const int64_t iter0 = ta.counters[kIter], il0 = ta.counters[kIterLocal];
    double ll = ac.scal[kLogLik], sum_r = ac.scal[kSumR], ds = ac.scal[kDSigma];  // at the current x
    const double prior = ac.scal[kPriorLogp];
    c.load_x();
    const int sub = lane & 15, grp = tid >> 4;
    for (int e = tid; e < nown; e += kThreads) {
        const int64_t g = c.element(ra.perm, e);
        x_s[e] = __ldcg(reinterpret_cast<const float *>(ra.xs.x) + g);
        p_s[e] = __ldcg(reinterpret_cast<const float *>(ra.p) + g);
        g0_s[e] = __ldcg(reinterpret_cast<const float2 *>(ra.grad) + g);
    }
    const float eps = static_cast<float>(ra.eps), half_eps = static_cast<float>(0.5 * ra.eps);
    const float lambda = static_cast<float>(ra.lambda);
    float xmax = 0.f;
    unsigned bits = 0;  // error bits
    int64_t accepted = 0;
    // the locations of slot k (its x in lane-local x, or this CTA's x_s) into CTA r
    auto push = [&](int k, int r, const float *x) {
        StVec<D> v{};
#pragma unroll
        for (int d = 0; d < D; ++d) v.v[d] = x[d];
        *cluster.map_shared_rank(c.xr_s + k, r) = v;
    };
    cluster.sync();
    for (int it = 0; it < a.n_iter; ++it) {
        // ---- start: momenta, energies, half kick and drift
        {
            DF ke{}, xx{};
            for (int e = tid; e < nown; e += kThreads) {
                const int64_t g = c.element(ra.perm, e);
                float p;
                if (ta.momentum_src == 1) {
                    uint32_t ctr[4] = {static_cast<uint32_t>(g >> 2), static_cast<uint32_t>(iter0 + it), ta.chain, 0u};
                    philox10(ctr, ta.seed);
                    float z0, z1;
                    if (g & 2)
                        box_muller(ctr[2], ctr[3], z0, z1);
                    else
                        box_muller(ctr[0], ctr[1], z0, z1);
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
            for (int e = tid; e < (k1 - k0) * kStCtas; e += kThreads) {
                const int i = e / kStCtas;
                push(k0 + i, e % kStCtas, x_s + i * D);
            }
        }
        cluster.sync();
        c.split_x(sp);
        for (int step = 0; step < a.n_steps; ++step) {
            const bool last = step + 1 == a.n_steps;
            // log u for the decision, by a warp that mostly has no unit (FP64: long)
            if (step == 0 && ac.metropolis && tid == kThreads - 32) {
                double u;
                if (ac.u_src == 2) {
                    u = ac.u_inj[il0 + it];
                } else {
                    uint32_t ctr[4] = {0u, static_cast<uint32_t>(iter0 + it), ac.chain, 1u};
                    philox10(ctr, ac.seed);
                    u = open_unit(ctr[0]);
                }
                logu_s = log(u);
            }
            // ---- the units of this CTA
            DF se{}, sm{}, sl{};
            c.units(last, se, sm, sl);
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
                c.gather(cluster, k, in, acc);
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
                    if (in) push(k, sub, xn);
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
            if (!last) c.split_x(sp);
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
        double l1 = 0.0, dh = 0.0;
        StScalars t1{};
        if (tid == 0) {
            t1 = st_scalars(ra, sum_s[kPartE2], sum_s[kPartMd], sum_s[kPartLp]);
            l1 = t1.ll;
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
                if (!isfinite(t1.ds)) bits |= kErrNonfinite;
                if (keep) {
                    sum_r = t1.sum_r;
                    ds = t1.ds;
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
        // (but for an infinite maximum: a diverged trajectory, reported as non-finite)
        float m = static_cast<float>(sum_s[kPartXmax]);
        if (isinf(m)) m = xmax = sp.bound;
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
        const int64_t g = c.element(ra.perm, e);
        reinterpret_cast<float *>(ra.xs.x)[g] = x_s[e];
        reinterpret_cast<float *>(ra.p)[g] = p_s[e];
        reinterpret_cast<float2 *>(ra.grad)[g] = g0_s[e];
        write_split_slot(ra.xs, sp, k0 + e / D, D, e % D, x_s[e]);
    }
    if (tid == 0 && rank == 0) {
        *ra.xs.split = sp;
        const float m = static_cast<float>(sum_s[kPartXmax]);
        atomicMax(ra.xs.xmax_bits, __float_as_uint(isinf(m) ? sp.bound : m));
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

// One evaluation (gradient, L, sum r, dL/dsigma) at the current locations in
// one launch: the units, the gather, the scalar terms, and the hand-over that
// publish_kernel does behind a pass and its reduction.
enum StEvalPart : int { kEvE2 = 0, kEvMd, kEvLp, kEvBits, kEvParts };

template <int D>
__global__ void __launch_bounds__(32 * st_warps<D>(), 1) small_eval_kernel(const __grid_constant__ SmallEvalArgs a) {
    constexpr int kWarps = st_warps<D>(), kThreads = 32 * kWarps;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ float box_s[kWarps][2 * D];
    __shared__ short4 unit_s[kStMaxUnits];
    __shared__ DF part_s[kEvParts][kWarps];
    __shared__ double all_s[kStCtas][kEvParts];
    __shared__ double sum_s[kEvParts], scal_s[kScalars];
    __shared__ unsigned bits_s, err_s;
    cg::cluster_group cluster = cg::this_cluster();
    const ReduceArgs &ra = a.reduce;
    const StLayout L(a.pair.nt, D);
    SmallCta<D> c(a.pair, L, smem, static_cast<int>(cluster.block_rank()), box_s, unit_s);
    const int rank = c.rank, tid = c.tid, warp = c.warp, lane = c.lane, k0 = c.k0, k1 = c.k1, nown = (k1 - k0) * D;
    float2 *const g_s = reinterpret_cast<float2 *>(smem + L.g0);
    pdl_trigger();
    c.stage_y();
    if (tid == 0) bits_s = 0u;
    pdl_wait();
    c.load_x();
    if (tid == 0) err_s = __ldcg(ra.err);
    if (rank == 0 && tid < kScalars) scal_s[tid] = __ldcg(ra.scal + tid);
    __syncthreads();
    DF se{}, sm{}, sl{};
    c.units(true, se, sm, sl);
    warp_part(se, part_s, kEvE2);
    warp_part(sm, part_s, kEvMd);
    warp_part(sl, part_s, kEvLp);
    cluster.sync();
    unsigned bad = 0;
    for (int kb = k0; kb < k1; kb += kThreads / 16) {
        const int k = kb + (tid >> 4);
        const bool in = k < k1;
        DF acc[D];
        c.gather(cluster, k, in, acc);
        if (in && (lane & 15) == 0) {
#pragma unroll
            for (int d = 0; d < D; ++d) {
                const DF v = df_mul(acc[d], ra.part_scale_df);
                if (!isfinite(v.hi)) bad = kErrNonfinite;
                g_s[(k - k0) * D + d] = make_float2(v.hi, v.lo);
            }
        }
    }
    if (bad) atomicOr(&bits_s, bad);
    __syncthreads();
    if (tid < kEvParts * kStCtas) {
        const int i = tid / kStCtas, r = tid % kStCtas;
        double v;
        if (i == kEvBits) {
            v = bits_s;
        } else {
            DF t = part_s[i][0];
#pragma unroll
            for (int w = 1; w < kWarps; ++w) df_add(t, part_s[i][w]);
            v = static_cast<double>(t.hi) + static_cast<double>(t.lo);
        }
        *cluster.map_shared_rank(&all_s[rank][i], r) = v;
    }
    cluster.sync();
    if (warp < kEvParts) {
        double v = all_s[lane & 15][warp];
#pragma unroll
        for (int o = 8; o >= 1; o >>= 1) {
            const double w = __shfl_xor_sync(0xffffffffu, v, o);
            v = warp == kEvBits ? fmax(v, w) : v + w;
        }
        if (lane == 0) sum_s[warp] = v;
    }
    __syncthreads();
    if (tid == 0) {
        const StScalars t = st_scalars(ra, sum_s[kEvE2], sum_s[kEvMd], sum_s[kEvLp]);
        unsigned b = sum_s[kEvBits] > 0.0 ? kErrNonfinite : 0u;
        if (!isfinite(t.ll) || !isfinite(t.ds)) b |= kErrNonfinite;
        bits_s = b;
        scal_s[kLogLik] = t.ll;
        scal_s[kLogLikEnd] = t.ll;
        scal_s[kSumR] = t.sum_r;
        scal_s[kDSigma] = t.ds;
    }
    __syncthreads();
    const unsigned err = err_s | bits_s;  // the same in every CTA
    for (int e = tid; e < nown; e += kThreads) {
        const int64_t g = c.element(ra.perm, e);
        const float2 v = g_s[e];
        reinterpret_cast<float2 *>(ra.grad)[g] = v;
        if (a.dst && err == 0u) {
            const double w = static_cast<double>(v.x) + static_cast<double>(v.y);
            if (a.dst_f64)
                static_cast<double *>(a.dst)[g] = w;
            else
                static_cast<float *>(a.dst)[g] = static_cast<float>(w);
        }
    }
    if (rank == 0) {
        if (tid < kScalars) {
            ra.scal[tid] = scal_s[tid];
            if (a.pub) a.pub->scal[tid] = scal_s[tid];
        }
        if (tid == 0) {
            if (bits_s) atomicOr(ra.err, bits_s);
            if (a.pub) a.pub->err = err;
        }
    }
}

template <typename F>
cudaError_t prepare(F *kernel, int smem) {
    const void *fn = reinterpret_cast<const void *>(kernel);
    cudaError_t e = raise_dyn_smem(fn, smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

// One cluster, under programmatic dependent launch.
template <int D, typename A>
cudaError_t launch_cluster(void (*kernel)(A), const A &a, cudaStream_t s, int *clusters) {
    const int smem = StLayout(a.pair.nt, D).bytes;
    cudaError_t e = clusters ? prepare(kernel, smem) : cudaSuccess;
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
    cfg.numAttrs = clusters ? 1 : 2;
    // clusters: only set the kernel's attributes and ask how many can be resident (before any launch: the fits rules)
    if (clusters) return cudaOccupancyMaxActiveClusters(clusters, kernel, &cfg);
    e = cudaLaunchKernelEx(&cfg, kernel, a);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int D>
cudaError_t launch_traj_d(const SmallTrajArgs &a, cudaStream_t s) {
    return launch_cluster<D>(small_traj_kernel<D>, a, s, nullptr);
}
template <int D>
cudaError_t launch_eval_d(const SmallEvalArgs &a, cudaStream_t s) {
    return launch_cluster<D>(small_eval_kernel<D>, a, s, nullptr);
}

// Whether a cluster can be resident on this device (16 SMs of one GPC).
template <int D>
bool resident_d(int nt) {
    SmallTrajArgs t{};
    SmallEvalArgs v{};
    t.pair.nt = v.pair.nt = nt;
    int n_traj = 0, n_eval = 0;
    if (launch_cluster<D>(small_traj_kernel<D>, t, nullptr, &n_traj) != cudaSuccess ||
        launch_cluster<D>(small_eval_kernel<D>, v, nullptr, &n_eval) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return n_traj >= 1 && n_eval >= 1;
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

// The rules: up to the number of row blocks at which this is faster than the
// whole chip with its hand-overs.  Trajectories, us a step here against pass
// and reduction (start and end of a trajectory: 9 here, 18 there): D = 1,
// N = 512 5.2 / 5.0, N = 640 6.8 / 5.2; D = 2, N = 512 5.9 / 6.0, N = 640
// 7.9 / 6.2; D = 3, N = 448 6.2 / 6.9, N = 512 7.9 / 6.9; D = 4, N = 448
// 6.5 / 8.1, N = 512 8.3 / 8.1; D = 6, N = 384 8.5 / 9.8, N = 448 9.8 / 9.5;
// D = 8, N = 384 10.2 / 12.1, N = 448 11.7 / 11.9.
bool small_traj_fits(int64_t nt, int d) {
    if (d < 1 || d > 8 || nt > (d <= 2 ? kStMaxBlocks : d <= 4 ? 7 : 6)) return false;
    if (StLayout(static_cast<int>(nt), d).bytes > kStMaxSmem) return false;
    MDS_ST_SWITCH(d, resident_d, static_cast<int>(nt))
    return false;
}

// Evaluations, us a gradient call here against pass, reduction and hand-over:
// D = 2, N = 50 18.3 / 20.3, N = 200 19.5 / 19.6; D = 4, N = 320 20.3 / 21.9,
// N = 448 22.0 / 22.1; D = 6, N = 320 21.3 / 23.4, N = 384 24.6 / 23.4; D = 8,
// N = 320 23.1 / 25.8, N = 448 26.6 / 26.2 (the wait and the launches on the
// host are about 13 of them).
bool small_eval_fits(int64_t nt, int d) { return nt <= (d <= 2 ? 2 : 5) && small_traj_fits(nt, d); }

cudaError_t launch_small_traj(const SmallTrajArgs &a, int d, cudaStream_t s) {
    MDS_ST_SWITCH(d, launch_traj_d, a, s)
    return cudaErrorInvalidValue;
}

cudaError_t launch_small_eval(const SmallEvalArgs &a, int d, cudaStream_t s) {
    MDS_ST_SWITCH(d, launch_eval_d, a, s)
    return cudaErrorInvalidValue;
}

}  // namespace mds
