// Short rows of the compressors with a dense message (bit-wise, RTN) in one launch: a thread-block cluster per worker holds
// the row in the shared memory of its blocks; largest magnitude, level statistics, draw and message follow there, with a
// cluster barrier (about a microsecond) where the longer rows have a kernel boundary.
// The blocks exchange the largest magnitudes and, with adaptive probabilities, the sums of the levels.
#pragma once

#include <algorithm>

#include <cooperative_groups.h>

#include "bitplanes.cuh"

namespace mlmc {
namespace {

namespace cg = cooperative_groups;

constexpr int kDenseMost = 16;                 // blocks per cluster
constexpr int kDenseLevels = 8;
constexpr int kDenseSpread = 16;               // groups per block where there are SMs to spread them over,
constexpr int kDenseGroups = 28;               // at most
constexpr int kDenseBytes = kDenseGroups * 4096;

template <int WARPS, typename S>
struct DenseShared {
    uint32_t top[kDenseMost];                  // per block: its largest key
    S sum[kDenseMost][kDenseLevels];           // per block: its sums of the levels
    uint32_t warp_top[WARPS];
    S warp_sum[kDenseLevels][WARPS];
    double p;
    int level;
};

// Blocks per cluster, 0: the row is too long or the workers too many.  A group per warp if the clusters of all workers fit the
// GPU at a time (they are placed within a GPC: 16-block clusters leave SMs over), otherwise the largest clusters that do.
// With more than kDenseGroups groups per block the few warps of two workers' clusters take as long as kernels on the whole GPU.
// us per message, cluster / kernels, 16 blocks, groups per block 20, 28, 36, 48:
//   bit-wise, fp32, adaptive, 2 workers 14 / 19, 16 / 19, 19 / 19, 21 / 19;  7 workers 15 / 22, 17 / 25, 20 / 28, 23 / 33
//   RTN, fp32, adaptive, 2 workers 19 / 22, 25 / 23, 28 / 25, 35 / 26;       7 workers 20 / 27, 25 / 32, 28 / 34, 34 / 41
//   RTN, fp32, given p, 2 workers 10 / 10, 12 / 10, 13 / 11, 16 / 11;        7 workers 10 / 14, 12 / 14, 14 / 16, 16 / 17
inline int dense_cluster_blocks(const Workspace& ws, int64_t d, int M) {
    const int64_t groups = (d + 1023) / 1024;
    int best = 0;
    for (int i = 0; i < 5; ++i) {
        if (M > ws.limits.dense_fit[i]) break;
        best = 1 << i;
        if (groups <= (int64_t)kDenseSpread << i) break;
    }
    return best && (groups + best - 1) / best <= kDenseGroups ? best : 0;
}

// The block's groups g0 .. g0 + n - 1 into its slots (group i by warp i mod WARPS; the others may read them after the call); returns the row's largest key, the
// same in every block.  Entries past the row's end are zeros.
template <typename T, int WARPS, typename S>
__device__ __forceinline__ uint32_t dense_load(cg::cluster_group& cluster, const T* __restrict__ row, int64_t d, int64_t g0, int n,
                                               uint32_t* slots, DenseShared<WARPS, S>& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    cluster.barrier_arrive();
    for (int i = warp; i < n; i += WARPS) fetch_group<T>(row, d, g0 + i, g0 + n, slots + i * kGroupSlot<T>);
    cp_async_wait<0>();
    __syncwarp();
    uint32_t mx = 0;
    for (int i = warp; i < n; i += WARPS) {
        const uint4* q = reinterpret_cast<const uint4*>(slots + i * kGroupSlot<T>);
#pragma unroll
        for (int c = 0; c < kGroupChunks<T>; ++c) {
            const uint4 x = q[c * 32 + lane];
            if constexpr (sizeof(T) == 4) {
                mx = max(max(mx, x.x & 0x7FFFFFFFu), max(x.y & 0x7FFFFFFFu, max(x.z & 0x7FFFFFFFu, x.w & 0x7FFFFFFFu)));
            } else {
                const uint32_t a = __vmaxu2(__vmaxu2(x.x & 0x7FFF7FFFu, x.y & 0x7FFF7FFFu),
                                            __vmaxu2(x.z & 0x7FFF7FFFu, x.w & 0x7FFF7FFFu));
                mx = max(mx, max(a & 0xFFFFu, a >> 16));
            }
        }
    }
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    if (lane == 0) sh.warp_top[warp] = mx;
    __syncthreads();
    const int CL = (int)cluster.num_blocks();
    mx = __reduce_max_sync(0xFFFFFFFFu, sh.warp_top[lane % WARPS]);
    cluster.barrier_wait();  // every block of the cluster runs: its shared memory can be written
    if (threadIdx.x < CL) cluster.map_shared_rank(sh.top, threadIdx.x)[cluster.block_rank()] = mx;
    cluster.sync();
    mx = 0;
#pragma unroll
    for (int r = 0; r < kDenseMost; ++r) mx = max(mx, r < CL ? sh.top[r] : 0u);
    return mx;
}

// Sums over the row of what the threads have of every level (a thread's 32-bit sums stay below 2^32 / 32): lane l of warp 0
// returns level l, the same in every block.  Fixed order.
template <typename A, int WARPS, typename S>
__device__ __forceinline__ S dense_sums(cg::cluster_group& cluster, const A (&acc)[kDenseLevels], DenseShared<WARPS, S>& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, CL = (int)cluster.num_blocks();
    if constexpr (sizeof(A) == 4) {  // a level per lane, then a level per warp
        uint32_t mine = 0;
#pragma unroll
        for (int l = 0; l < kDenseLevels; ++l) {
            const uint32_t x = __reduce_add_sync(0xFFFFFFFFu, acc[l]);
            mine = lane == l ? x : mine;
        }
        if (lane < kDenseLevels) sh.warp_sum[lane][warp] = (S)mine;
        __syncthreads();
        static_assert(WARPS <= 32 && (sizeof(A) != 4 || WARPS >= kDenseLevels), "the warps' sums of a level fit a warp");
        if (warp < kDenseLevels) {
            const uint32_t x = lane < WARPS ? (uint32_t)sh.warp_sum[warp][lane] : 0u;
            const S s = (S)__reduce_add_sync(0xFFFFFFFFu, x & 0xFFFFu) + (S)__reduce_add_sync(0xFFFFFFFFu, x >> 16) * (S)65536;
            if (lane < CL) cluster.map_shared_rank(&sh.sum[0][0], lane)[cluster.block_rank() * kDenseLevels + warp] = s;
        }
    } else {
        // half of the levels go to the partner lane in each of the first three steps: lane l ends with level l / 4
        static_assert(kDenseLevels == 8, "three halvings");
        S x[4], y[2], z;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const S got = __shfl_xor_sync(0xFFFFFFFFu, (lane & 16) ? acc[i] : acc[i + 4], 16);
            x[i] = ((lane & 16) ? acc[i + 4] : acc[i]) + got;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const S got = __shfl_xor_sync(0xFFFFFFFFu, (lane & 8) ? x[i] : x[i + 2], 8);
            y[i] = ((lane & 8) ? x[i + 2] : x[i]) + got;
        }
        z = __shfl_xor_sync(0xFFFFFFFFu, (lane & 4) ? y[0] : y[1], 4) + ((lane & 4) ? y[1] : y[0]);
        z += __shfl_xor_sync(0xFFFFFFFFu, z, 2);
        z += __shfl_xor_sync(0xFFFFFFFFu, z, 1);
        if ((lane & 3) == 0) sh.warp_sum[lane >> 2][warp] = z;
        __syncthreads();
        for (int i = threadIdx.x; i < kDenseLevels * CL; i += WARPS * 32) {
            S s = 0;
#pragma unroll
            for (int w = 0; w < WARPS; ++w) s += sh.warp_sum[i % kDenseLevels][w];
            cluster.map_shared_rank(&sh.sum[0][0], i / kDenseLevels)[cluster.block_rank() * kDenseLevels + i % kDenseLevels] = s;
        }
    }
    cluster.sync();
    S total = 0;
    if (threadIdx.x < kDenseLevels)
#pragma unroll
        for (int r = 0; r < kDenseMost; ++r) total += r < CL ? sh.sum[r][threadIdx.x] : S(0);
    return total;
}

// The level of the message, by every block for itself; the first block of the cluster writes the header.  delta: the norm
// of level l in lane l of warp 0.
template <int WARPS, typename S>
__device__ __forceinline__ int dense_level(const DrawPlan& pl, const DrawnLevels& drawn, int adaptive, int m, bool first, double delta,
                                           float scale, DenseShared<WARPS, S>& sh, double* p_out, int* status, int* worker_err) {
    const int lane = threadIdx.x & 31;
    int level = drawn.level[m];
    double p_sel = drawn.p[level];
    if (adaptive) {
        if (threadIdx.x < 32) {
            double p;
            const int drawn_level = warp_draw(delta, pl.L, counter_uniform(pl.seed, pl.step, (uint64_t)m), &p);
            if (first && lane < pl.L) {
                pl.delta_all[m * kMaxLevels + lane] = delta;
                pl.p_all[m * kMaxLevels + lane] = p;
            }
            p_sel = __shfl_sync(0xFFFFFFFFu, p, drawn_level);
            if (lane == 0) {
                sh.level = drawn_level;
                sh.p = p_sel;
            }
        }
        __syncthreads();
        level = sh.level;
        p_sel = sh.p;
    }
    *p_out = p_sel;
    if (first && threadIdx.x == 0) write_header(pl, m, level, p_sel, scale, status, worker_err);
    return level;
}

template <typename K>
bool configure_dense_cluster(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDenseBytes) == cudaSuccess &&
           cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
}

}  // namespace
}  // namespace mlmc
