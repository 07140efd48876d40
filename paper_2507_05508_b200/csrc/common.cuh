// Shared declarations of the MLMC CUDA library: workspace layout, device helpers, launcher prototypes.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/mlmc.h"
#include "../../include/mlmc_instr.h"

namespace mlmc {

constexpr int kMaxLevels = MLMC_MAX_LEVELS;   // L <= 32, so at most 31 thresholds per worker
constexpr int kMaxQueries = kMaxLevels;
constexpr int kBins1 = 32768;                 // leading digit: key bits 30..16 (fp32) / the whole key (bf16)
constexpr int kBins23 = 256;                  // second and third digits: key bits 15..8 and 7..0
constexpr uint32_t kKeyNone = 0xFFFFFFFFu;    // threshold above every finite key: "nothing is inside"
constexpr uint32_t kNoSlot = 0xFFu;

constexpr int kSweepThreads = 512;            // histogram / masked / norm sweeps
constexpr int kEmitMaxWorkers = 1024;         // M of one call: the emit and averaging kernels keep per-worker offsets in shared memory
constexpr int kEmitRows = 16;                 // 32-bit words per lane that a warp of the emit kernels holds at a time
constexpr int kEmitTile = 4096;               // 32-bit words per emit tile (1 fp32 or 2 bf16 elements each); one warp per tile
constexpr int kEmitTileVecs = kEmitTile / 4;  // 16-byte vectors per tile, for both element types
constexpr int kEmitGroups = kEmitTile / (kEmitRows * 32);  // batches of kEmitRows * 32 words per tile: 8
constexpr int kEmitGroupVecs = kEmitTileVecs / kEmitGroups;  // 16-byte vectors per batch: 128
constexpr int kBatchKeys = kEmitGroupVecs * 4;  // fp32 entries of a batch
constexpr int kItemTiles = 4;                 // emit tiles per item of the band count: one batch per lane of a warp
constexpr int kSuperItems = 32;               // items per super-item, super-items per hyper-item: their counts are added up too
constexpr int kTileBits = 21;                 // of a listed tile: at most 2^20 tiles per worker (d < 2^32)
constexpr int kEnergyCells = 2 * kMaxLevels;  // (boundary bin, interval) pairs: at most 31 bins, each threshold adds one interval
constexpr int kAggTile = 4096;                // dense output elements per aggregation tile

// Per-worker selection query: the rank-k element of the total order.
struct Query {
    uint32_t k;        // target rank, 1 <= k < d for live queries
    uint32_t prefix;   // key bits fixed so far
    uint32_t rem;      // rank still to descend inside the current prefix set (1-based, from the top)
    uint32_t slot;     // histogram slot of the next digit pass (kNoSlot when resolved or trivial)
    uint32_t T;        // resolved threshold key
    uint32_t c;        // #{ key > T }
    uint32_t n;        // #{ key == T }
    uint32_t r;        // how many key == T elements, in index order, are inside Top-k  (k - c)
    uint32_t trivial;  // 1: k == 0 (nothing inside), 2: k >= d (everything inside), 0: live
    uint32_t slot2;    // histogram slot of the second digit pass = index of the boundary bin among the distinct ones
    uint32_t pad[2];
};

// Emit parameters of one worker, produced by the draw kernel.
struct EmitParams {
    uint32_t Ta, ra;   // Top-k_{l*-1}: inside iff key > Ta or (key == Ta and tie rank <= ra)
    uint32_t Tb, rb;   // Top-k_{l*}
    double inv_p;      // 1 / p_{l*}
    uint32_t expect;   // k_{l*} - k_{l*-1}
    int32_t enabled;   // 0: worker skipped (device error)
    int32_t level;
    int32_t pad;
};

// Kernel identifiers for launch accounting and per-kernel timing.
enum KernelId {
    K_BEGIN = 0, K_UNIFORMS, K_HIST1, K_RESOLVE1, K_SUMS_CAND, K_CAND2, K_CAND3, K_BAND_HEADER, K_COPY_PROBS, K_EMIT, K_AGG_OFFSETS,
    K_AGG_TOPK, K_ABSMAX, K_BIT_STATS, K_BIT_PACK, K_AGG_BIT, K_TILE_LIST, K_BAND_COUNT, K_FLOAT_PACK, K_AGG_FLOAT,
    K_RTN_STATS, K_RTN_EMIT, K_AGG_DENSE, K_SEG_RESOLVE, K_SEG_SWEEP, K_SEG_BUCKETS, K_SEG_NORMS, K_SEG_DRAW, K_CLUSTER_TOPK,
    K_BIT_CLUSTER, K_RTN_CLUSTER, K_SORT_ROWS, K_SAMPLE, K_BRACKET_SWEEP, K_CAND_HIST, K_MISSED_HIST, K_MISSED_SUMS, K_COUNT
};

// Level probabilities handed to a kernel by value.
struct ProbList {
    double p[kMaxLevels];
};
inline ProbList prob_list(const double* p, int L) {
    ProbList r = {};
    if (p)
        for (int l = 0; l < L; ++l) r.p[l] = p[l];
    return r;
}

// The levels of a call with given probabilities: they depend on seed, step and worker only, so the host draws them.
struct DrawnLevels {
    double p[kMaxLevels];
    uint8_t level[kEmitMaxWorkers];
};

constexpr int kTimingPool = 2048;  // event pairs kept between two reads

// Brackets of a worker's thresholds (topk_bracket.cu): runs of leading-digit bins, from the largest keys down.
struct BracketRuns {
    int n;
    int top[kMaxQueries], low[kMaxQueries];  // highest and lowest bin
    uint8_t code[kMaxQueries + 1];           // level interval of the keys above run i; [n]: below the last one
};
constexpr int kLeftOut = 2;  // Workspace::miss: the sample finds more keys in the brackets than the candidate list has room for
constexpr int64_t kBracketLeast = 1 << 21;  // entries of a row: at least twice as many as the largest sample

// What the device can place.
struct KernelLimits {
    // clusters of 1, 2, .. 16 blocks that run at a time
    int topk_fit[5];             // of the short-row Top-k kernel
    int dense_fit[5];            // of the short-row dense kernels
    int sample_fit;              // clusters of 16 blocks of the sample kernel
    // blocks per SM
    int band_count[2];           // fp32, bf16
    int aggregate_topk, aggregate_bitwise, aggregate_float;
    int rtn_stats[2][2];         // fp32, bf16; few levels, many
    int sort_rows;
};

struct Workspace {
    // per-kernel timing (off by default): one CUDA event pair around every kernel launch
    bool timing;
    int timing_used;
    cudaEvent_t* ev_start;
    cudaEvent_t* ev_stop;
    int* ev_id;
    int64_t launches_by_id[K_COUNT];
    int device;
    int64_t d_max;
    int M_max, L_max;
    int sm_count;
    int64_t launches;
    KernelLimits limits;
    bool long_sweeps;            // this call's sweeps are long enough to be launched without overlap (see launch_kernel)
    // device memory
    int* status;                 // sticky status word
    int* worker_err;             // [M] per-worker device error (0 = fine)
    uint32_t* hist1;             // [M][kBins1]  counts, then suffix sums in place
    uint8_t* table1;             // [M][kBins1]  leading-digit bin -> slot of pass 2
    uint32_t* hist2;             // [M][kMaxQueries][256], hist3 behind it
    uint8_t* map2;               // [M][kMaxQueries][256] (slot2, digit2) -> slot of pass 3, or 64 + energy cell
    uint32_t* hist3;             // [M][kMaxQueries][256]
    Query* queries;              // [M][kMaxQueries]
    uint32_t* done;              // [M] blocks of a worker that have finished (every kernel that counts leaves it at zero)
    double* sum_partial;         // [M][sum_ctas][kMaxLevels]  sweep 2: energy of the threshold-free bins
    int sum_ctas, cur_sum_ctas;
    unsigned long long* cand_S;  // [M][kEnergyCells][2 halves] integer energy sums of the boundary-bin keys outside the threshold sub-bins
    uint32_t* cand_keys;         // [M][cand_cap] keys of the boundary-bin elements
    int64_t cand_cap;
    uint32_t* cand_count;        // [M]
    int* cand_overflow;          // [M] 1: the candidates did not fit, full-sweep passes take over
    double* p_all;               // [M][kMaxLevels]
    double* delta_all;           // [M][kMaxLevels]
    double* u_dev;               // [M] (mlmc_read_u)
    EmitParams* emit;            // [M]
    uint4* tile_desc;            // [M][tiles per worker] {C, A, B, tie flag} of every emit tile
    uint4* level_desc;           // {C, A, B, batches} of every item [M][items], then super-item, then hyper-item
    uint2* tile_list;            // the tiles of all workers that can hold band entries, in any order: {worker << kTileBits | tile, batch mask}
    uint32_t* list_n;            // how many
    int64_t max_tiles;
    // [M][tiles per worker][kEmitGroups] largest magnitude key of every batch of every emit tile (first sweep of a message)
    uint32_t* tile_max;
    uint32_t* group_n;           // [M] how many batches the last emission had to read
    int64_t last_emit_tiles;     // tiles per row of the last emission (host side, for mlmc_read_listed_tiles)
    uint32_t* cand_floor;        // [M] smallest key that can be a candidate of sweep 2 (lower edge of the lowest boundary bin)
    uint32_t* agg_offsets;       // [M][agg_tiles_max + 1]
    // bit-wise
    uint32_t* gmax_bits;         // [2][M] largest key; after the first sweep of a long RTN message the smallest of the batches' largest ones
    uint32_t* acc_word;          // [2][M] running maxima (or error flag) of a sweep; its last block leaves them at zero
    unsigned long long* S_partial;  // [M][stat_ctas][kMaxLevels]
    int stat_ctas;
    int32_t* bit_level;          // [M] drawn level of a dense message (-1: void), read by the kernel that writes it
    // fixed-p Top-k: boundary bins of the previous call, per worker and level boundary, reused as brackets
    uint32_t* prev_bin;          // [M][kMaxLevels] leading-digit bin of threshold j at the last call that resolved it (kKeyNone: none)
    uint4* bracket;              // [M] {lo_a, width_a, lo_b, width_b}: bins collected as candidates by the first sweep
    int* bracket_hit;            // [M] 1: both boundary bins of the drawn band lie in their brackets
    // [3] workers with both brackets hit / a bracket missed / no bracket yet; from [4] on, sampled brackets: all held / missed / left out
    // (cumulative)
    unsigned long long* bracket_stats;
    int64_t sig_d, sig_ld;       // host: the problem the stored bins belong to
    int sig_M, sig_L, sig_dtype;
    int64_t sig_k[kMaxLevels];
    // adaptive Top-k with sampled brackets
    BracketRuns* runs;           // [M]
    int* miss;                   // [M] 1: a threshold lies outside its bracket, or the candidates did not fit; kLeftOut
    uint32_t* part_n;            // [M][parts] candidates that every warp of the sweep found
    int sweep_blocks, parts;     // host: blocks and warps of the sweep per worker,
    uint32_t part_cap;           //       room of each warp
    // s-Top-k with more levels than kMaxLevels
    int64_t big_cap;             // most levels
    void* seg_scratch;           // buffers of the segment norms (stopk_segments.cu), allocated at first use
    size_t seg_bytes;
    // RTN: per-block residual energies of every level
    double* rtn_partial;         // [M][rtn_ctas][kMaxLevels]
    int rtn_ctas;
};

// Level draw and message header of the dense compressors (bit planes, RTN).
struct DrawPlan {
    int L;
    int w_max;                  // planes of the message buffer; width[l] of them are needed (RTN: all 0)
    int width[kMaxLevels];
    uint64_t seed, step;
    int32_t* bit_level;
    double* p_all;
    double* delta_all;
    float* out_scale;           // null: no message (mlmc_level_probs)
    int32_t* out_level;
    double* out_p_sel;
};

// ---------------------------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void set_status(int* status, int code) { atomicCAS(status, 0, code); }

// Adds the three 16-bit limbs of x (below 2^48) to the shared-memory words at addr, addr + STRIDE and addr + 2 STRIDE bytes.
// (Under a predicate each of the three becomes a branch: 33 instead of 22 instructions per entry.)
template <uint32_t STRIDE>
__device__ __forceinline__ void shared_add_limbs(uint32_t addr, uint64_t x) {
    asm volatile("red.shared.add.u32 [%0], %1;\n\tred.shared.add.u32 [%0 + %4], %2;\n\tred.shared.add.u32 [%0 + %5], %3;" ::"r"(addr),
                 "r"((uint32_t)x & 0xFFFFu), "r"(__byte_perm((uint32_t)x, 0u, 0x4432)), "r"((uint32_t)(x >> 32)), "n"(STRIDE),
                 "n"(2 * STRIDE)
                 : "memory");
}

// Stores x at the shared-memory address `at` and moves on by `step` bytes, where `flag` is negative; no branch.
__device__ __forceinline__ void shared_push_if_negative(int flag, uint32_t& at, uint32_t x, uint32_t step) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %1, 0;\n\t@p st.shared.u32 [%0], %2;\n\t@p add.u32 %0, %0, %3;\n\t}"
                 : "+r"(at) : "r"(flag), "r"(x), "r"(step) : "memory");
}

// Two fp32 numbers in a 64-bit register: packed instructions take one issue slot for both (and the time of two), and round each like
// the single instruction.  The compiler (nvcc 12.9) merges a packed product into an addition that follows it, .rn or not: where
// both have to round, the addition is written as a multiply-add with a 1 that the compiler does not know.
__device__ __forceinline__ uint64_t pair(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ uint64_t mul_pair(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t add_pair(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma_pair(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t fma_pair_toward_zero(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rz.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// mant^2 of an fp32 entry (the implicit bit included, below the normal range none): the entry is mant 2^(max(e,1) - 150).
__device__ __forceinline__ uint64_t mantissa_squared(uint32_t bits) {
    const uint32_t mant = min(bits & 0x7FFFFFFFu, (bits & 0x7FFFFFu) | 0x800000u);  // the key itself where it lies below 2^23
    return (uint64_t)mant * mant;
}

// Every kernel of the library starts with pdl_enter().  The kernels are launched with programmatic stream
// serialization, so a kernel's blocks may become resident while the kernel before it in the stream is still running;
// nothing is read or written before the wait, which returns when that kernel has completed and its writes are visible.
// A chain of short kernels then pays about 1 us per launch instead of 3 to 4.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// True in every thread of the one block of `nblocks` that gets here last: what the other blocks wrote before is
// visible to it (read with __ldcg).  No block waits for another.  The counter is left at zero for the next kernel.
__device__ __forceinline__ bool last_block(uint32_t* counter, uint32_t nblocks) {
    __shared__ bool sh_last;
    __syncthreads();
    if (nblocks == 1u) return true;
    if (threadIdx.x == 0) {
        __threadfence();
        sh_last = atomicAdd(counter, 1u) == nblocks - 1u;
        if (sh_last) *counter = 0u;
        __threadfence();
    }
    __syncthreads();
    return sh_last;
}

__host__ __device__ __forceinline__ uint64_t splitmix_finalize(uint64_t z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// One uniform in [0,1) per (seed, step, worker): three chained SplitMix64 output rounds.
__host__ __device__ __forceinline__ double counter_uniform(uint64_t seed, uint64_t step, uint64_t worker) {
    const uint64_t golden = 0x9E3779B97F4A7C15ull;
    uint64_t h = splitmix_finalize(seed + golden);
    h = splitmix_finalize(h + step + golden);
    h = splitmix_finalize(h + worker + golden);
    return (double)(h >> 11) * 0x1.0p-53;
}

// cdf in ascending l; the last level with p > 0 and everything after it has cdf 1; l* = min{l : u < cdf_l}
// ("Sample l ~ p^l", Alg. 2 / Alg. 3).
__host__ __device__ __forceinline__ int draw_from_probs(const double* p, int L, double u) {
    int j_last = -1;
    for (int j = 0; j < L; ++j)
        if (p[j] > 0.0) j_last = j;
    double c = 0.0;
    for (int j = 0; j < L; ++j) {
        c += p[j];
        const double cdf = (j >= j_last) ? 1.0 : c;
        if (u < cdf) return j;
    }
    return 0;
}

// Header of one worker's dense message, by one thread.
__device__ __forceinline__ void write_header(const DrawPlan& pl, int m, int level, double p_sel, float scale, int* status,
                                             int* worker_err) {
    if (pl.out_level) {
        if (pl.width[level] > pl.w_max) {
            worker_err[m] = MLMC_ERR_CAPACITY;
            set_status(status, MLMC_ERR_CAPACITY);
            level = -1;
        }
        pl.out_level[m] = level;
        pl.out_p_sel[m] = level >= 0 ? p_sel : 0.0;
        pl.out_scale[m] = scale;
    }
    pl.bit_level[m] = level;
    if (level >= 0) pl.p_all[m * kMaxLevels + level] = p_sel;
}

__device__ __forceinline__ void void_header(const DrawPlan& pl, int m) {
    pl.bit_level[m] = -1;
    if (pl.out_level) {
        pl.out_level[m] = -1;
        pl.out_p_sel[m] = 0.0;
        pl.out_scale[m] = 0.0f;
    }
}

// p_l = delta_l / sum delta (Lemma 3.4; all weight on level 0 where every delta is 0) and the draw l* = min{ l : u < cdf_l },
// by one warp, a level per lane (delta = 0 from level L on).  The last level with p > 0 has cdf 1.  Both sums go over the levels in
// ascending order: the shuffles do not depend on one another, so a step costs one addition.  (A butterfly and a tree of 5
// steps each round otherwise and save nothing that could be measured: 3 x 700,001 entries, 15 levels, 55 to 59 us either way.)
__device__ __forceinline__ int warp_draw(double delta, int L, double u, double* p_out) {
    const int l = threadIdx.x & 31;
    double total = 0.0;
#pragma unroll 4
    for (int i = 0; i < L; ++i) total += __shfl_sync(0xFFFFFFFFu, delta, i);
    const double p = (total > 0.0) ? delta / total : (l == 0 ? 1.0 : 0.0);
    double cdf = 0.0;
#pragma unroll 4
    for (int i = 0; i < L; ++i) {
        const double y = __shfl_sync(0xFFFFFFFFu, p, i);
        if (i <= l) cdf += y;
    }
    const uint32_t positive = __ballot_sync(0xFFFFFFFFu, p > 0.0);  // never empty
    const uint32_t below = __ballot_sync(0xFFFFFFFFu, p > 0.0 && u < cdf);
    *p_out = p;
    return below ? __ffs(below) - 1 : 31 - __clz((int)positive);
}

// Probabilities from the residual norms sh_delta[L] of one worker, the draw and the header; by warp 0 of the block.
__device__ __forceinline__ void finish_levels(const DrawPlan& pl, int m, const double* sh_delta, float scale, int* status,
                                              int* worker_err) {
    if (threadIdx.x >= 32) return;
    const int l = threadIdx.x;
    const double delta = l < pl.L ? sh_delta[l] : 0.0;
    double p;
    const int level = warp_draw(delta, pl.L, counter_uniform(pl.seed, pl.step, (uint64_t)m), &p);
    if (l < pl.L) {
        pl.delta_all[m * kMaxLevels + l] = delta;
        pl.p_all[m * kMaxLevels + l] = p;
    }
    const double p_sel = __shfl_sync(0xFFFFFFFFu, p, level);
    if (l == 0) write_header(pl, m, level, p_sel, scale, status, worker_err);
}

inline DrawnLevels draw_levels(const double* p, int L, uint64_t seed, uint64_t step, int M) {
    DrawnLevels r = {};
    if (!p) return r;
    for (int l = 0; l < L; ++l) r.p[l] = p[l];
    for (int m = 0; m < M; ++m) r.level[m] = (uint8_t)draw_from_probs(p, L, counter_uniform(seed, step, (uint64_t)m));
    return r;
}

// Magnitude key: monotone in |g| for finite values.  fp32: 31 bits; bf16: 15 bits.
template <typename T>
struct ElemTraits;

template <>
struct ElemTraits<float> {
    static constexpr int kVec = 4;             // elements per 16-byte load
    static constexpr uint32_t kInfKey = 0x7F800000u;
    static constexpr int kShift1 = 16;         // key >> kShift1 = leading digit
    __device__ static __forceinline__ uint32_t key(uint32_t bits) { return bits & 0x7FFFFFFFu; }
    __device__ static __forceinline__ float value(uint32_t bits) { return __uint_as_float(bits); }
};

struct bf16_t {
    uint16_t x;
};

template <>
struct ElemTraits<bf16_t> {
    static constexpr int kVec = 8;
    static constexpr uint32_t kInfKey = 0x7F80u;
    static constexpr int kShift1 = 0;
    __device__ static __forceinline__ uint32_t key(uint32_t bits) { return bits & 0x7FFFu; }
    __device__ static __forceinline__ float value(uint32_t bits) { return __uint_as_float(bits << 16); }
};

// Loads the 16-byte vector v of a row and hands each element's raw bits to f(index_in_row, bits).
// Elements at or past d are skipped; a vector that straddles d is read element by element.
template <typename T, typename F>
__device__ __forceinline__ void for_each_in_vector(const T* row, int64_t v, int64_t d, F&& f) {
    constexpr int V = ElemTraits<T>::kVec;
    const int64_t base = v * V;
    if (base + V <= d) {
        const uint4 q = __ldg(reinterpret_cast<const uint4*>(row) + v);
        if constexpr (V == 4) {
            f(base + 0, q.x);
            f(base + 1, q.y);
            f(base + 2, q.z);
            f(base + 3, q.w);
        } else {
            f(base + 0, q.x & 0xFFFFu);
            f(base + 1, q.x >> 16);
            f(base + 2, q.y & 0xFFFFu);
            f(base + 3, q.y >> 16);
            f(base + 4, q.z & 0xFFFFu);
            f(base + 5, q.z >> 16);
            f(base + 6, q.w & 0xFFFFu);
            f(base + 7, q.w >> 16);
        }
    } else {
        for (int64_t i = base; i < d; ++i) {
            uint32_t bits;
            if constexpr (V == 4)
                bits = reinterpret_cast<const uint32_t*>(row)[i];
            else
                bits = reinterpret_cast<const uint16_t*>(row)[i];
            f(i, bits);
        }
    }
}

// A warp's 1024 histogram bins in coalesced vectors: lane l has the vectors i * 32 + l of the 256.
__device__ __forceinline__ void load_bins(const uint32_t* bins, uint4 (&x)[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = reinterpret_cast<const uint4*>(bins)[i * 32 + (threadIdx.x & 31)];
}
// Hands every lane the 32 bins from 32 * mine through shared memory (rows: 256 vectors per warp; vector j of bin group t at j ^ t, so that
// neither side meets in a bank).  Read directly, every load touches 32 lines (segment_resolve of 16 rows 23.6 us, 20.9 so).
__device__ __forceinline__ void hand_over_bins(const uint4 (&x)[8], uint4* rows, int mine, uint32_t (&cnt)[32]) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int owner = i * 4 + (lane >> 3);
        rows[owner * 8 + ((lane ^ owner) & 7)] = x[i];
    }
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint4 y = rows[mine * 8 + ((i ^ mine) & 7)];
        cnt[4 * i] = y.x; cnt[4 * i + 1] = y.y; cnt[4 * i + 2] = y.z; cnt[4 * i + 3] = y.w;
    }
}

constexpr size_t kBinRowsSmem = (size_t)kBins1 * sizeof(uint32_t);  // rows of 32 warps

// Asks for the 128-byte line at p as far as L2.
__device__ __forceinline__ void prefetch_line(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// 16-byte asynchronous copy from global to shared memory (cp.async), grouped by commit / wait.
__device__ __forceinline__ void cp_async_16(void* smem_dst, const void* gmem_src) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// A block's threads stream the 16-byte vectors of `src`, VECS per thread and trip: trips first, first + step, ... below `end`.
// Three trips are in flight while one is used; a thread copies and reads only its own vectors, so there is no barrier.
// ring: [4][VECS][THREADS] vectors of shared memory.  (The loop is not unrolled over the slots: the bodies are long, and
// four copies of one miss the instruction cache.)
template <int VECS, int THREADS, typename F>
__device__ __forceinline__ void stream_trips(const uint4* __restrict__ src, int64_t first, int64_t step, int64_t end, uint4* ring, F&& f) {
    if (first >= end) return;
    uint4* mine = ring + threadIdx.x;
    const uint4* from = src + first * (VECS * THREADS) + threadIdx.x;
    const int64_t ahead = step * (VECS * THREADS);
    int left = (int)((end - first + step - 1) / step), unasked = left;  // trips to use, trips to ask for
    auto fetch = [&](int at) {
        if (unasked > 0) {
#pragma unroll
            for (int j = 0; j < VECS; ++j) cp_async_16(mine + at + j * THREADS, from + j * THREADS);
            from += ahead;
            --unasked;
        }
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < 3; ++i) fetch(i * VECS * THREADS);
    int at = 0, to = 3 * VECS * THREADS;  // slot in use, slot to fill
#pragma unroll 1
    do {
        fetch(to);
        cp_async_wait<3>();
        uint4 q[VECS];
#pragma unroll
        for (int j = 0; j < VECS; ++j) q[j] = mine[at + j * THREADS];
        f(q);
        to = at;
        at = at + VECS * THREADS < 4 * VECS * THREADS ? at + VECS * THREADS : 0;
    } while (--left);
    cp_async_wait<0>();
}

// Emit tiles of one row: kEmitTile 32-bit words each (one fp32 or two bf16 elements per word).
inline int emit_tiles_per_worker(int64_t d, int dtype) {
    const int per_word = (dtype == MLMC_BF16) ? 2 : 1;
    const int64_t words = (d + per_word - 1) / per_word;
    return (int)((words + kEmitTile - 1) / kEmitTile);
}

struct EmitCounts {
    int items, supers, hypers;  // per worker
    int total() const { return items + supers + hypers; }
};
inline EmitCounts emit_counts(int tiles) {
    EmitCounts n;
    n.items = (tiles + kItemTiles - 1) / kItemTiles;
    n.supers = (n.items + kSuperItems - 1) / kSuperItems;
    n.hypers = (n.supers + kSuperItems - 1) / kSuperItems;
    return n;
}

// Resident blocks per SM, at least 1.
template <typename K>
int resident_blocks(K kernel, int threads, size_t smem) {
    int n = 0;
    const bool ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kernel, threads, smem) == cudaSuccess;
    return ok && n >= 1 ? n : 1;
}

// Clusters of 2^i blocks that run at a time (a block takes an SM).
template <typename K>
void clusters_that_fit(K kernel, int threads, size_t smem, int (&fit)[5]) {
    for (int i = 0; i < 5; ++i) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(1 << i);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = 1 << i;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        fit[i] = 0;
        if (cudaOccupancyMaxActiveClusters(&fit[i], kernel, &cfg) != cudaSuccess) {
            cudaGetLastError();
            fit[i] = 0;
        }
    }
}

// Brackets one kernel launch: counts it and, when timing is on, records an event pair on the stream.
struct LaunchScope {
    Workspace& ws;
    cudaStream_t s;
    int slot;
    LaunchScope(Workspace& w, int id, cudaStream_t st) : ws(w), s(st), slot(-1) {
        ws.launches++;
        ws.launches_by_id[id]++;
        if (ws.timing && ws.timing_used < kTimingPool) {
            slot = ws.timing_used++;
            ws.ev_id[slot] = id;
            cudaEventRecord(ws.ev_start[slot], s);
        }
    }
    ~LaunchScope() {
        if (slot >= 0) cudaEventRecord(ws.ev_stop[slot], s);
    }
};

// Kernels that stream the gradients or the messages.
inline bool is_sweep(int id) {
    switch (id) {
        case K_HIST1: case K_SUMS_CAND: case K_BAND_COUNT: case K_EMIT: case K_AGG_TOPK: case K_ABSMAX: case K_BIT_STATS:
        case K_BIT_PACK: case K_AGG_BIT: case K_FLOAT_PACK: case K_AGG_FLOAT: case K_RTN_STATS:
        case K_RTN_EMIT: case K_AGG_DENSE: case K_SEG_SWEEP: case K_BRACKET_SWEEP:
            return true;
        default:
            return false;
    }
}

// Enqueues one kernel, with programmatic stream serialization (see pdl_enter) unless it is a long sweep.  Blocks that
// become resident beside the last blocks of the kernel before them inherit its split of L1 and shared memory, and a
// sweep with a small L1 keeps fewer loads in flight: on 4 GB that cost 5 to 10 % of the sweep (bit-wise step 3.00 ->
// 3.27 ms, Top-k step 2.33 -> 2.49 ms), where the overlap gains 2 us a launch; the two meet at about 100 MB.
constexpr int64_t kLongSweepBytes = 100 << 20;
inline void set_call_size(Workspace& ws, int64_t d, int M, int elem_size) { ws.long_sweeps = d * M * elem_size > kLongSweepBytes; }

template <typename... P, typename... A>
inline void launch_kernel_cluster(Workspace& ws, int id, int cluster, void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                                  cudaStream_t s, A&&... args) {
    LaunchScope t(ws, id, s);
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = attr;
    if (cluster > 1) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = (unsigned)cluster;
        attr[cfg.numAttrs].val.clusterDim.y = attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    if (!(ws.long_sweeps && is_sweep(id))) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        ++cfg.numAttrs;
    }
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename... P, typename... A>
inline void launch_kernel(Workspace& ws, int id, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                          A&&... args) {
    launch_kernel_cluster(ws, id, 1, kernel, grid, threads, smem, s, args...);
}

// Enqueues one kernel whose blocks all run at a time (they meet at grid barriers).
template <typename... P, typename... A>
inline void launch_kernel_grid(Workspace& ws, int id, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
    LaunchScope t(ws, id, s);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

// ---------------------------------------------------------------------------------------------
// launchers (each enqueues on `s` and bumps ws.launches)
// ---------------------------------------------------------------------------------------------
// topk_select.cu
int configure_select_kernels();
// One worker of a call whose level is drawn on the host (given p): the level, its probability and the two ranks that
// bound its band.
struct DrawnBand {
    double p;
    int32_t level;
    uint32_t k_lo, k_hi;
};
void launch_begin_adaptive(Workspace& ws, int dtype, int64_t d, int M, const int64_t* k, int L, cudaStream_t s);
void launch_begin_drawn(Workspace& ws, int dtype, int64_t d, int M, const DrawnBand* bands, int L, bool brackets, cudaStream_t s);
void launch_uniforms(Workspace& ws, int M, uint64_t seed, uint64_t step, cudaStream_t s);
void launch_hist1(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, bool brackets, const int* only, cudaStream_t s);
// What the last kernel of a selection does with its thresholds.
struct FinishPlan {
    int L;              // levels; queries are the L - 1 boundaries (adaptive) or the two of the drawn band
    int nq;
    int adaptive;       // energies, probabilities and the draw
    int want_emit;      // message header and emit parameters
    int64_t d;
    uint64_t seed, step;
    uint32_t k[kMaxLevels];
    int64_t* out_count;
    int32_t* out_level;
    double* out_p_sel;
    int64_t capacity;
};
void launch_resolve1(Workspace& ws, int dtype, int M, const FinishPlan& plan, bool brackets, bool sampled, int* miss, cudaStream_t s);
void launch_sums_candidates(Workspace& ws, const void* g, int64_t d, int M, int64_t ld, const FinishPlan& plan, bool brackets,
                            const int* only, cudaStream_t s);
void launch_digit_passes(Workspace& ws, const void* g, int64_t d, int M, int64_t ld, const FinishPlan& plan, bool sampled, cudaStream_t s);
void launch_band_header(Workspace& ws, int M, const FinishPlan& plan, cudaStream_t s);
void launch_copy_probs(Workspace& ws, int M, int L, const double* p_fixed, double* p_out, double* delta_out,
                       cudaStream_t s);
// topk_bracket.cu: adaptive Top-k of long fp32 rows, one sweep
int configure_bracket_kernels();
void bracket_limits(KernelLimits* limits);
bool use_brackets(const Workspace& ws, int dtype, int64_t d, int M, const int64_t* k, int L);
void launch_bracket_sweep(Workspace& ws, const float* g, int64_t d, int M, int64_t ld, const int64_t* k, const FinishPlan& plan,
                          cudaStream_t s);
// topk_emit.cu
int configure_emit_kernels();
void emit_limits(KernelLimits* limits);
void launch_emit(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const mlmc_topk_msgs& out,
                 cudaStream_t s);
void launch_aggregate_topk(Workspace& ws, const mlmc_topk_msgs& msgs, int M, int64_t d, float* out, cudaStream_t s);
// bitwise.cu
int configure_bit_kernels();
void bit_limits(KernelLimits* limits);
// Largest keys of the batches where the message kernels skip the batches that round to 0: in long sweeps (above 100 MB).  us per step,
// given p, everything read / with the look, rows in layers: bit planes 106 MB 60 / 56, 400 MB 180 / 147, 4 GB 1484 / 1161; RTN
// 84 / 78, 271 / 237, 2478 / 2046.  Entries of one scale, where nothing is skipped: bit planes 71 / 70, 205 / 205, 1724 / 1739.
// Shorter calls lie in L2, and to look first costs more than to read (8 x 1M entries, bit planes: 32.2 us per step, 33.4 with the look).
inline const uint32_t* zero_batches(const Workspace& ws) { return ws.long_sweeps ? ws.tile_max : nullptr; }
// Largest magnitude of every worker, in long sweeps of its batches too, and the NaN / Inf check; with `p` (given probabilities) also
// the draw and the header; with `signs` (a bit-plane message, long sweeps) its sign planes, but for the ragged end of a row.
void launch_absmax(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const DrawPlan& plan, const double* p,
                   const mlmc_bit_msgs* signs, cudaStream_t s);
DrawPlan bit_draw_plan(Workspace& ws, const int32_t* b, int L, uint64_t seed, uint64_t step, const mlmc_bit_msgs* out);
// Adaptive: field energies of every level, probabilities, draw and header.
void launch_bit_stats(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b, int L,
                      const DrawPlan& plan, cudaStream_t s);
bool launch_bit_cluster(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b, int L,
                        const DrawPlan& plan, const double* p, const mlmc_bit_msgs& out, cudaStream_t s);
void launch_bit_pack(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b, int L,
                     const mlmc_bit_msgs& out, cudaStream_t s);
void launch_aggregate_bitwise(Workspace& ws, const mlmc_bit_msgs& msgs, const int32_t* b, int L, int M, int64_t d,
                              float* out, cudaStream_t s);

// floatbits.cu
int configure_float_kernels();
void float_limits(KernelLimits* limits);
void launch_compress_floatbits(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* mb,
                               int L, const double* p, uint64_t seed, uint64_t step, const mlmc_float_msgs& out, cudaStream_t s);
void launch_aggregate_floatbits(Workspace& ws, const mlmc_float_msgs& msgs, const int32_t* mb, int L, int M, int64_t d,
                                float* out, cudaStream_t s);
// rtn.cu
DrawPlan rtn_draw_plan(Workspace& ws, int L, uint64_t seed, uint64_t step, const mlmc_rtn_msgs* out);
// Adaptive: residual energies of every level, probabilities, draw and header.
void launch_rtn_stats(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                      const DrawPlan& plan, cudaStream_t s);
int configure_rtn_kernels();
void rtn_limits(KernelLimits* limits);
bool launch_rtn_cluster(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                        const DrawPlan& plan, const double* p, const mlmc_rtn_msgs& out, cudaStream_t s);
void launch_rtn_emit(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                     const mlmc_rtn_msgs& out, cudaStream_t s);
void launch_aggregate_dense(Workspace& ws, const float* val, const int32_t* level, int M, int64_t d, int64_t ldv,
                            float* out, cudaStream_t s);
// topk_cluster.cu: Top-k messages of short rows in one launch
int configure_cluster_kernels();
void cluster_limits(KernelLimits* limits);
int cluster_blocks(const Workspace& ws, int dtype, int64_t d, int M, bool given);
void launch_cluster_topk(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const FinishPlan& plan,
                         const DrawnBand* bands, const mlmc_topk_msgs* out, cudaStream_t s);
// stopk_segments.cu: s-Top-k with adaptive p and many segments
int configure_segment_kernels();
int reserve_segments(Workspace& ws);
void launch_segments(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, int64_t s_len, int64_t L,
                     uint64_t seed, uint64_t step, cudaStream_t s);

}  // namespace mlmc
