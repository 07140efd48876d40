// Adaptive Top-k of long fp32 rows in one sweep: brackets around the level thresholds from a sample of the row.
//
// The thresholds of the levels (ranks k_0 .. k_{L-2} of the magnitude order) and the energies of the bands between them
// (Lemma 3.4) need the whole row.  With the leading-digit histogram (topk_select.cu) they take two reads of it: one to
// find the digit bins of the thresholds, one to add up the energies and to collect the keys that share a bin with a
// threshold.  Here a sample says where the thresholds lie, within a bracket of a few bins each, and one read does the
// rest:
//   sample         clears what the selection accumulates into; a cluster per worker counts a stratified sample of the
//                  row and turns every rank into a bracket of bins; brackets that touch form one run.  A worker whose
//                  runs hold too many keys (exact zeros, equal magnitudes around a threshold) takes the call out of the sweep;
//   bracket_sweep  energy and count of the keys between the runs, the keys inside the runs as candidates, the largest
//                  key of every batch for the emission;
//   candidate_hist leading-digit counts of the candidates; with the counts between the runs they stand in for the
//                  histogram of the row.
// The rest is topk_select.cu: resolve1 finds the bin of every threshold (in a run, or the worker is sent through the
// histogram path), the digit passes end the selection.  Thresholds and bands never depend on the sample; the energies are the same
// sums of squares in fp64, added up in an order that follows the runs, so that norms and probabilities agree to rounding.
#include <cooperative_groups.h>

#include <algorithm>

#include "topk_finish.cuh"

namespace cg = cooperative_groups;

namespace mlmc {

namespace {

constexpr int kSampleThreads = 1024;
constexpr int kSampleTrips = 16;                 // 16-byte vectors per thread: 65,536 keys per block
constexpr int kSectorKeys = 8;                   // keys that are sampled together (32 bytes: two threads)
constexpr int kBlockSectors = kSampleThreads * kSampleTrips * 4 / kSectorKeys;

struct SampleRanks {
    uint32_t k[kMaxQueries];
    int nq;
    uint32_t most;  // sampled keys that the runs may hold
};

// The half width of a bracket is kSampleSigmas standard deviations of the sample rank of independent keys from one
// distribution.  Keys that are sampled together may say the same (up to sqrt(8) times the deviation); strata that differ
// from one another lower it (the ranks then vary within the strata only).
constexpr double kSampleSigmas = 5.0;
__host__ __device__ inline double bracket_half(double r, double n) {  // of sample rank r among n sampled keys
    const double v = r * (1.0 - r / n);
    return kSampleSigmas * sqrt(v > 0.0 ? v : 0.0) + 1.0;
}

// Share of the candidate list that the runs may fill, by the sample.  The keys are spread over the parts of the list by batches, and one
// full part sends the worker through the two other sweeps after this one.  8 x 2^25 entries, a threshold among equal magnitudes: at
// 0.94 of the list 1022 us (two sweeps 1319), at 0.96 1651 (1330), left out 1366 (1363).
constexpr double kMostRoom = 0.93;

template <int C>
__global__ void __launch_bounds__(kSampleThreads, 1)
sample_kernel(ZeroList z, SampleRanks ranks, Query* queries, const float* __restrict__ g, int64_t d, int64_t ld, BracketRuns* runs,
              uint8_t* table, int* miss) {
    extern __shared__ uint32_t sh_hist[];  // [kBins1]
    __shared__ uint32_t sh_warp[32], sh_total;
    __shared__ uint32_t sh_at[2][kMaxQueries];
    // the bracket's edges: {bin, sampled keys above the upper edge's bin, or those down to the lower edge's}
    __shared__ uint2 sh_edge[2][kMaxQueries];
    __shared__ BracketRuns sh_runs;
    __shared__ uint32_t sh_inside;  // sampled keys in the runs
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = C > 1 ? (int)cluster.block_rank() : 0, m = blockIdx.x / C;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nq = ranks.nq;
    for (int b = threadIdx.x; b < kBins1; b += kSampleThreads) sh_hist[b] = 0;
    pdl_enter();
    clear_all(z);
    if (rank == 0 && threadIdx.x < nq) queries[m * kMaxQueries + threadIdx.x] = make_query(ranks.k[threadIdx.x], d);
    __syncthreads();
    constexpr uint32_t kStrata = kBlockSectors * C, n = kStrata * kSectorKeys;  // sampled keys
    if (threadIdx.x < nq) {  // bracket of query j: from the bin of sample rank r_j - half to the bin of sample rank r_j + half
        const double r = (double)ranks.k[threadIdx.x] / (double)d * n, half = bracket_half(r, n);
        sh_at[0][threadIdx.x] = (uint32_t)fmax(floor(r - half), 0.0);          // 0: up to the largest key
        sh_at[1][threadIdx.x] = (uint32_t)fmin(ceil(r + half), (double)n + 1.0);  // n + 1: down to the smallest
    }
    // Stratum i is a range of consecutive sectors, of which one is sampled; the blocks of the cluster take turns.
    const uint4* row = reinterpret_cast<const uint4*>(g + (int64_t)m * ld);
    const uint64_t sectors = (uint64_t)d / kSectorKeys;
#pragma unroll 1
    for (int t = 0; t < kSampleTrips; t += 8) {
        uint4 q[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint32_t i = (((t + j) * kSampleThreads + threadIdx.x) / 2) * C + rank;
            const uint64_t first = i * sectors / kStrata, end = (i + 1) * sectors / kStrata;  // a power of two
            const uint64_t at = first + __umulhi(i * 0x9E3779B1u, (uint32_t)(end - first));
            q[j] = __ldg(row + at * 2 + (threadIdx.x & 1));
        }
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            atomicAdd(&sh_hist[(q[j].x & 0x7FFFFFFFu) >> 16], 1u);
            atomicAdd(&sh_hist[(q[j].y & 0x7FFFFFFFu) >> 16], 1u);
            atomicAdd(&sh_hist[(q[j].z & 0x7FFFFFFFu) >> 16], 1u);
            atomicAdd(&sh_hist[(q[j].w & 0x7FFFFFFFu) >> 16], 1u);
        }
    }
    // Block r sums the cluster's counts of the bins [r kBins1 / C, (r + 1) kBins1 / C); a thread owns kBins1 / C / 1024 of them.
    constexpr int per = kBins1 / C / kSampleThreads;
    const int b0 = rank * (kBins1 / C) + threadIdx.x * per;
    uint32_t cnt[per];
    if (C > 1) cluster.sync(); else __syncthreads();
#pragma unroll
    for (int i = 0; i < per; ++i) cnt[i] = 0u;
#pragma unroll
    for (int r = 0; r < C; ++r) {
        const uint32_t* h = C > 1 ? cluster.map_shared_rank(sh_hist, (rank + r) % C) : sh_hist;
#pragma unroll
        for (int i = 0; i < per; i += 2) {
            const uint2 x = *reinterpret_cast<const uint2*>(h + b0 + i);
            cnt[i] += x.x;
            cnt[i + 1] += x.y;
        }
    }
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < per; ++i) sum += cnt[i];
    uint32_t suffix = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(0xFFFFFFFFu, suffix, o);
        if (lane + o < 32) suffix += y;
    }
    if (lane == 0) sh_warp[warp] = suffix;
    __syncthreads();
    const uint32_t w = sh_warp[lane];
    uint32_t above = suffix - sum + __reduce_add_sync(0xFFFFFFFFu, lane > warp ? w : 0u);
    if (C > 1) {
        if (threadIdx.x == 0) sh_total = above + sum;  // thread 0 owns the block's lowest bins
        cluster.sync();
        for (int r = rank + 1; r < C; ++r) above += *cluster.map_shared_rank(&sh_total, r);
    }
    for (int j = 0; j < nq; ++j) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t at = sh_at[e][j];
            int bin = -1;
            uint32_t count = 0;
            if (at == 0u) {
                if (b0 == 0) bin = kBins1 - 1;
            } else if (at > n) {
                if (b0 == 0) { bin = 0; count = n; }
            } else if (above < at && at <= above + sum) {
                uint32_t run = above;
#pragma unroll
                for (int i = per - 1; i >= 0; --i) {
                    if (run < at) { bin = b0 + i; count = e ? run + cnt[i] : run; }
                    run += cnt[i];
                }
            }
            if (bin >= 0) {
                for (int q = 0; q < C; ++q)
                    *(C > 1 ? cluster.map_shared_rank(&sh_edge[e][j], q) : &sh_edge[e][j]) = make_uint2((uint32_t)bin, count);
            }
        }
    }
    if (C > 1) cluster.sync(); else __syncthreads();
    if (threadIdx.x == 0) {  // runs from the largest keys down; at least one bin lies between two of them
        int R = 0, next = 0, top = 0, low = 0;
        uint32_t inside = 0, from = 0, to = 0;
        for (int j = 0; j < nq; ++j) {
            if (ranks.k[j] == 0u) next = j + 1;
            if (ranks.k[j] == 0u || (int64_t)ranks.k[j] >= d) continue;
            const uint2 upper = sh_edge[0][j], lower = sh_edge[1][j];
            const int hi = (int)upper.x, lo = (int)lower.x;
            if (R && hi >= low - 1) {
                low = min(low, lo);
                to = max(to, lower.y);
            } else {
                if (R) { sh_runs.top[R - 1] = top; sh_runs.low[R - 1] = low; }
                sh_runs.code[R] = (uint8_t)j;
                inside += to - from;
                from = upper.y;
                to = lower.y;
                top = hi;
                low = min(lo, hi);
                ++R;
            }
            next = j + 1;
        }
        inside += to - from;
        if (R) { sh_runs.top[R - 1] = top; sh_runs.low[R - 1] = low; }
        sh_runs.code[R] = (uint8_t)next;
        sh_runs.n = R;
        sh_inside = inside;
        if (rank == 0) {
            runs[m] = sh_runs;
            miss[m] = inside > ranks.most ? kLeftOut : 0;
        }
    }
    __syncthreads();
    if (sh_inside > ranks.most) return;  // nobody looks at the table
    const int R = sh_runs.n;
    // What the sweep looks up: the interval of a bin, or nq + 1 where it lies in a run.
    constexpr int kWords = kBins1 / 4 / C;
    for (int i = rank * kWords + threadIdx.x; i < (rank + 1) * kWords; i += kSampleThreads) {
        uint32_t word = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int bin = i * 4 + j;
            uint32_t code = 0;
            while (code < (uint32_t)R && sh_runs.low[code] > bin) ++code;
            if (code < (uint32_t)R && sh_runs.top[code] >= bin) code = (uint32_t)nq + 1u;
            word |= code << (8 * j);
        }
        reinterpret_cast<uint32_t*>(table + (int64_t)m * kBins1)[i] = word;
    }
}

// -------------------------------------------------------------------------------------------
// the sweep
// -------------------------------------------------------------------------------------------
// Interval i is the keys between run i - 1 (above) and run i (below).  A warp takes one batch of the emit tiles at a time (four
// 16-byte vectors per lane) and goes one of four ways, by what the batch holds:
//   - nothing reaches the lowest run: one fused multiply-add per key;
//   - nearly all keys lie in the two, or in the three, lowest intervals (of a schedule whose ranks double these hold 60 and 80 %
//     of a row): they are told apart by comparisons with the edges of the runs and added up in registers.  The other keys are set
//     aside in slots of the thread's own;
//   - every key is looked up: a byte per bin.
// A looked-up key is added to a column of shared memory per interval and thread (a key of a run to a column that nobody reads).
// Keys of runs and keys set aside wait in the slots until some lane has many; then every lane's last key is looked up, and
// the keys of runs go to the warp's own part of the candidate list.  All of this is in a fixed order: the sums, here and over
// the list, do not change from call to call.  Counts are exact integers, energies fp64 sums.
//
// Bound by issue (2.9 instructions per clock and SM, 25 per warp and key) with shared memory (62 %) and the integer pipe (57 %)
// behind it; the look-ups load the one, the comparisons the other.  8 x 124M entries, 15 levels: 950 us, where the histogram sweep
// and the sweep for energies and candidates took 605 + 996.  On the way there: three intervals compared wherever a quarter of the
// keys or less lies above them 973 us, two intervals or look-ups only 961; 21 warps instead of 24 (one scheduler has
// six and the others five) 1053; the warps of a block in step, so that all look up or all compare, 1044.
constexpr int kSlots = 16;                        // keys per thread; half a batch adds at most 8
constexpr int kSweepSmemMost = 226 * 1024;
constexpr int kFewAbove = 2, kSomeAbove = 1;      // of 32 keys: above the two, the three lowest intervals
constexpr int kSweepThreads24 = 768;              // 24 warps, six per scheduler

// One key against the edges of the lowest runs: x < lo_a: interval R (e0); hi_a <= x < lo_b: R - 1 (e1, c1); with three intervals
// hi_b <= x < lo_c: R - 2 (e2, c2); otherwise it is set aside.  No branch and no selection between sums: the square is multiplied by
// 1 or 0, of which only the high word is ever set (m0, m1, m2 are 0 or 1).  Counters as floats and the address by a multiplication,
// one = 1: the integer pipe has the comparisons to do.
__device__ __forceinline__ void window_add_two(uint32_t bits, float lo_a, float hi_a, float lo_b, double& e0, double& e1, double& m0,
                                               double& m1, float& c1, uint32_t& at, uint32_t step, uint32_t one) {
    asm volatile(
        "{\n\t.reg .pred p, q, s;\n\t.reg .f64 v;\n\t.reg .f32 x;\n\t.reg .b32 l, h;\n\t"
        "mov.b32 x, %6;\n\t"
        "abs.f32 x, x;\n\t"
        "cvt.f64.f32 v, x;\n\t"
        "mul.rn.f64 v, v, v;\n\t"
        "setp.lt.f32 p, x, %7;\n\t"
        "setp.ge.f32 q, x, %8;\n\t"
        "setp.lt.and.f32 q, x, %9, q;\n\t"
        "mov.b64 {l, h}, %2;\n\tselp.b32 h, 0x3FF00000, 0, p;\n\tmov.b64 %2, {l, h};\n\t"
        "mov.b64 {l, h}, %3;\n\tselp.b32 h, 0x3FF00000, 0, q;\n\tmov.b64 %3, {l, h};\n\t"
        "fma.rn.f64 %0, v, %2, %0;\n\t"
        "fma.rn.f64 %1, v, %3, %1;\n\t"
        "@q add.f32 %4, %4, 0f3F800000;\n\t"
        "or.pred s, p, q;\n\t"
        "@!s st.shared.u32 [%5], %6;\n\t"
        "@!s mad.lo.u32 %5, %10, %11, %5;\n\t}"
        : "+d"(e0), "+d"(e1), "+d"(m0), "+d"(m1), "+f"(c1), "+r"(at)
        : "r"(bits), "f"(lo_a), "f"(hi_a), "f"(lo_b), "r"(step), "r"(one)
        : "memory");
}
__device__ __forceinline__ void window_add_three(uint32_t bits, float lo_a, float hi_a, float lo_b, float hi_b, float lo_c, double& e0,
                                                 double& e1, double& e2, double& m0, double& m1, double& m2, float& c1, float& c2,
                                                 uint32_t& at, uint32_t step, uint32_t one) {
    asm volatile(
        "{\n\t.reg .pred p, q, r, s;\n\t.reg .f64 v;\n\t.reg .f32 x;\n\t.reg .b32 l, h;\n\t"
        "mov.b32 x, %9;\n\t"
        "abs.f32 x, x;\n\t"
        "cvt.f64.f32 v, x;\n\t"
        "mul.rn.f64 v, v, v;\n\t"
        "setp.lt.f32 p, x, %10;\n\t"
        "setp.ge.f32 q, x, %11;\n\t"
        "setp.lt.and.f32 q, x, %12, q;\n\t"
        "setp.ge.f32 r, x, %13;\n\t"
        "setp.lt.and.f32 r, x, %14, r;\n\t"
        "mov.b64 {l, h}, %3;\n\tselp.b32 h, 0x3FF00000, 0, p;\n\tmov.b64 %3, {l, h};\n\t"
        "mov.b64 {l, h}, %4;\n\tselp.b32 h, 0x3FF00000, 0, q;\n\tmov.b64 %4, {l, h};\n\t"
        "mov.b64 {l, h}, %5;\n\tselp.b32 h, 0x3FF00000, 0, r;\n\tmov.b64 %5, {l, h};\n\t"
        "fma.rn.f64 %0, v, %3, %0;\n\t"
        "fma.rn.f64 %1, v, %4, %1;\n\t"
        "fma.rn.f64 %2, v, %5, %2;\n\t"
        "@q add.f32 %6, %6, 0f3F800000;\n\t"
        "@r add.f32 %7, %7, 0f3F800000;\n\t"
        "or.pred s, p, q;\n\t"
        "or.pred s, s, r;\n\t"
        "@!s st.shared.u32 [%8], %9;\n\t"
        "@!s mad.lo.u32 %8, %15, %16, %8;\n\t}"
        : "+d"(e0), "+d"(e1), "+d"(e2), "+d"(m0), "+d"(m1), "+d"(m2), "+f"(c1), "+f"(c2), "+r"(at)
        : "r"(bits), "f"(lo_a), "f"(hi_a), "f"(lo_b), "f"(hi_b), "f"(lo_c), "r"(step), "r"(one)
        : "memory");
}

// The key's square to column n of the thread's energies and 1 to its counts (shared-memory addresses of column 0).
template <int THREADS>
__device__ __forceinline__ void column_add(uint32_t n, uint32_t bits, uint32_t energy, uint32_t count) {
    const double v = (double)__uint_as_float(bits);
    asm volatile(
        "{\n\t.reg .b32 a, c;\n\t.reg .f64 e;\n\t"
        "mad.lo.u32 a, %0, %4, %2;\n\t"
        "mad.lo.u32 c, %0, %5, %3;\n\t"
        "ld.shared.f64 e, [a];\n\t"
        "red.shared.add.u32 [c], 1;\n\t"
        "fma.rn.f64 e, %1, %1, e;\n\t"
        "st.shared.f64 [a], e;\n\t}" ::"r"(n), "d"(v), "r"(energy), "r"(count), "n"(THREADS * 8), "n"(THREADS * 4)
        : "memory");
}
// Stores x at the shared-memory address `at` and moves on by STEP bytes where a == b; no branch.
template <int STEP>
__device__ __forceinline__ void push_if_equal(uint32_t a, uint32_t b, uint32_t& at, uint32_t x, uint32_t one) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.eq.u32 p, %1, %2;\n\t@p st.shared.u32 [%0], %3;\n\t@p mad.lo.u32 %0, %4, %5, %0;\n\t}"
                 : "+r"(at) : "r"(a), "r"(b), "r"(x), "r"(one), "n"(STEP) : "memory");
}

// one = 1, zero = 0: arguments, so that the compiler does not fold them.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1)
bracket_sweep_kernel(const float* __restrict__ g, int64_t d, int64_t ld, int L, const BracketRuns* runs, const uint8_t* table,
                     uint32_t* __restrict__ tile_max, int tiles_per_worker, uint32_t* hist1, double* __restrict__ sum_partial,
                     int sum_ctas, uint32_t* __restrict__ cand_keys, int64_t cand_cap, uint32_t part_cap, uint32_t* part_n, int* miss, int M,
                     int* status, int* worker_err, uint32_t one, double zero) {
    extern __shared__ __align__(16) uint8_t sh_raw[];
    __shared__ BracketRuns sh_runs;
    constexpr int kWarps = THREADS / 32;
    constexpr uint32_t kStep = THREADS * 4;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int columns = L + 1;                                                   // intervals 0 .. L - 1, and one nobody reads
    uint8_t* code_of = sh_raw;                                                   // [kBins1]
    double* energy = reinterpret_cast<double*>(sh_raw + kBins1);                 // [columns][THREADS]
    uint32_t* counts = reinterpret_cast<uint32_t*>(energy + columns * THREADS);  // [columns][THREADS]
    uint32_t* slots = counts + columns * THREADS + threadIdx.x;                  // [kSlots][THREADS]
    pdl_enter();
    const int m = blockIdx.y;
    bool left_out = false;
    for (int i = threadIdx.x; i < M; i += THREADS) left_out |= miss[i] == kLeftOut;
    if (threadIdx.x == 0) sh_runs = runs[m];
    for (int i = threadIdx.x; i < kBins1 / 16; i += THREADS)
        reinterpret_cast<uint4*>(code_of)[i] = reinterpret_cast<const uint4*>(table + (int64_t)m * kBins1)[i];
    for (int l = 0; l < columns; ++l) {
        energy[l * THREADS + threadIdx.x] = 0.0;
        counts[l * THREADS + threadIdx.x] = 0u;
    }
    // Where one worker is left out all of them are: its two other sweeps take as long as those of all workers (the blocks are dealt
    // to the workers).  All blocks see the sample's mark of that worker, whoever else has been marked meanwhile.
    if (__syncthreads_or(left_out)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) miss[m] = kLeftOut;
        return;
    }
    const int R = sh_runs.n;
    // Edges of the three lowest runs as floats (the order of non-negative floats is that of their bits); a run that is not there
    // lies above every key.
    auto low_edge = [&](int i) { return i >= 0 ? __uint_as_float((uint32_t)sh_runs.low[i] << 16) : INFINITY; };
    auto high_edge = [&](int i) { return i >= 0 ? __uint_as_float(min(((uint32_t)sh_runs.top[i] + 1u) << 16, 0x7F800000u)) : INFINITY; };
    const float lo_a = low_edge(R - 1), hi_a = high_edge(R - 1), lo_b = low_edge(R - 2), hi_b = high_edge(R - 2), lo_c = low_edge(R - 3);
    const uint32_t floor_key = R ? (uint32_t)sh_runs.low[R - 1] << 16 : 0xFFFFFFFFu;
    const float* row = g + (int64_t)m * ld;
    uint32_t* tmax = tile_max + (int64_t)m * tiles_per_worker * kEmitGroups;
    uint32_t* part = cand_keys + (int64_t)m * cand_cap + (int64_t)(blockIdx.x * kWarps + warp) * part_cap;
    uint32_t part_at = 0;  // keys of this warp so far (warp-uniform)

    double e0 = 0.0, e1 = 0.0, e2 = 0.0, m0 = zero, m1 = zero, m2 = zero;  // intervals R, R - 1, R - 2
    float c1 = 0.0f, c2 = 0.0f;  // how many: exact, a thread sees fewer than 2^24 keys
    const uint32_t slots0 = (uint32_t)__cvta_generic_to_shared(slots);
    const uint32_t my_energy = (uint32_t)__cvta_generic_to_shared(energy + threadIdx.x),
                   my_count = (uint32_t)__cvta_generic_to_shared(counts + threadIdx.x);
    uint32_t at = slots0;
    auto look_up = [&](uint32_t bits) -> uint32_t { return code_of[(bits << 1) >> 17]; };
    // One key of every lane that has one, round by round, until no lane has more than `most`.  (Emptied whenever one lane's slots
    // were full, the others had few keys left and most lanes idled.)  Called by the whole warp.
    auto drain = [&](uint32_t most) {
        uint32_t n = (at - slots0) / kStep;
        for (int rounds = (int)__reduce_max_sync(0xFFFFFFFFu, n) - (int)most; rounds > 0; --rounds) {
            uint32_t bits = 0, code = 0;
            if (n) {
                bits = slots[--n * THREADS];
                code = look_up(bits);
                column_add<THREADS>(code, bits, my_energy, my_count);
            }
            const uint32_t mask = __ballot_sync(0xFFFFFFFFu, code == (uint32_t)L);
            if (mask) {
                const uint32_t to = part_at + (uint32_t)__popc(mask & ((1u << lane) - 1u));
                if (code == (uint32_t)L && to < part_cap) part[to] = bits & 0x7FFFFFFFu;
                part_at += (uint32_t)__popc(mask);
            }
        }
        at = slots0 + n * kStep;
    };
    auto make_room = [&]() {  // for half a batch
        if (__any_sync(0xFFFFFFFFu, at > slots0 + (kSlots - 8) * kStep)) drain(kSlots - 8);
    };

    const int nbatch = tiles_per_worker * kEmitGroups, stride = gridDim.x * kWarps;
    const int whole = (int)(d / kBatchKeys);  // batches that lie wholly inside the row
    bool bad = false;
    int b = blockIdx.x * kWarps + warp;
    // Every warp has every stride-th batch; the warps of a block start at different places of their lists, so that at any
    // time some look up (shared memory) while others compare (integer pipe): the batches of a layer go the same way.
    const int mine = b < whole ? (whole - b + stride - 1) / stride : 0;
    const uint4* const first = reinterpret_cast<const uint4*>(row) + (int64_t)b * kEmitGroupVecs + lane;
    int at_batch = (int)((int64_t)mine * warp / kWarps);
#pragma unroll 1
    for (int left = mine; left > 0; --left) {
        // The next batch comes as far as L2 meanwhile (16 lines of 128 bytes, one per lane): a second set of registers costs more.
        uint4 cur[4];
        const uint4* from = first + (int64_t)at_batch * stride * kEmitGroupVecs;
#pragma unroll
        for (int j = 0; j < 4; ++j) cur[j] = __ldg(from + j * 32);
        const int next = at_batch + 1 == mine ? 0 : at_batch + 1;
        if (lane < 16) prefetch_line(first + (int64_t)next * stride * kEmitGroupVecs + lane * 7);
        // largest key: the largest of the negative entries and of the others, each in its own order
        uint32_t un = 0;
        int sn = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            un = max(max(un, cur[j].x), cur[j].y);
            un = max(max(un, cur[j].z), cur[j].w);
            sn = max(max(sn, (int)cur[j].x), (int)cur[j].y);
            sn = max(max(sn, (int)cur[j].z), (int)cur[j].w);
        }
        const uint32_t wm = __reduce_max_sync(0xFFFFFFFFu, max(un & 0x7FFFFFFFu, (uint32_t)sn));
        bad |= wm >= 0x7F800000u;  // a non-finite entry shows in the largest key of its batch
        if (lane == 0) tmax[b + at_batch * stride] = wm;
        at_batch = next;
        if (wm < floor_key) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const double x0 = (double)__uint_as_float(cur[j].x), x1 = (double)__uint_as_float(cur[j].y),
                             x2 = (double)__uint_as_float(cur[j].z), x3 = (double)__uint_as_float(cur[j].w);
                e0 = fma(x0, x0, e0);
                e0 = fma(x1, x1, e0);
                e0 = fma(x2, x2, e0);
                e0 = fma(x3, x3, e0);
            }
            continue;
        }
        // one of a lane's keys says which way the batch goes
        const float probe = fabsf(__uint_as_float(cur[0].x));
        if (__popc(__ballot_sync(0xFFFFFFFFu, probe >= lo_b)) <= kFewAbove) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j == 2) make_room();
                window_add_two(cur[j].x, lo_a, hi_a, lo_b, e0, e1, m0, m1, c1, at, kStep, one);
                window_add_two(cur[j].y, lo_a, hi_a, lo_b, e0, e1, m0, m1, c1, at, kStep, one);
                window_add_two(cur[j].z, lo_a, hi_a, lo_b, e0, e1, m0, m1, c1, at, kStep, one);
                window_add_two(cur[j].w, lo_a, hi_a, lo_b, e0, e1, m0, m1, c1, at, kStep, one);
            }
        } else if (__popc(__ballot_sync(0xFFFFFFFFu, probe >= lo_c)) <= kSomeAbove) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j == 2) make_room();
                window_add_three(cur[j].x, lo_a, hi_a, lo_b, hi_b, lo_c, e0, e1, e2, m0, m1, m2, c1, c2, at, kStep, one);
                window_add_three(cur[j].y, lo_a, hi_a, lo_b, hi_b, lo_c, e0, e1, e2, m0, m1, m2, c1, c2, at, kStep, one);
                window_add_three(cur[j].z, lo_a, hi_a, lo_b, hi_b, lo_c, e0, e1, e2, m0, m1, m2, c1, c2, at, kStep, one);
                window_add_three(cur[j].w, lo_a, hi_a, lo_b, hi_b, lo_c, e0, e1, e2, m0, m1, m2, c1, c2, at, kStep, one);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                if (j == 2) make_room();
                const uint32_t n0 = look_up(cur[j].x), n1 = look_up(cur[j].y), n2 = look_up(cur[j].z), n3 = look_up(cur[j].w);
                column_add<THREADS>(n0, cur[j].x, my_energy, my_count);
                column_add<THREADS>(n1, cur[j].y, my_energy, my_count);
                column_add<THREADS>(n2, cur[j].z, my_energy, my_count);
                column_add<THREADS>(n3, cur[j].w, my_energy, my_count);
                push_if_equal<kStep>(n0, L, at, cur[j].x, one);  // a key of a run
                push_if_equal<kStep>(n1, L, at, cur[j].y, one);
                push_if_equal<kStep>(n2, L, at, cur[j].z, one);
                push_if_equal<kStep>(n3, L, at, cur[j].w, one);
            }
        }
        make_room();
    }
    for (b += mine * stride; b < nbatch; b += stride) {  // the row's end; batches past it have the largest key 0
        uint32_t most = 0;
        for (int64_t e = (int64_t)b * kBatchKeys + lane; e - lane < d; e += 32) {
            drain(kSlots - 8);
            if (e < d) {
                const uint32_t bits = reinterpret_cast<const uint32_t*>(row)[e];
                most = max(most, bits & 0x7FFFFFFFu);
                shared_push_if_negative(-1, at, bits, kStep);
            }
        }
        most = __reduce_max_sync(0xFFFFFFFFu, most);
        bad |= most >= 0x7F800000u;
        if (lane == 0) tmax[b] = most;
    }
    drain(0);
    if (lane == 0) {
        part_n[(int64_t)m * stride + blockIdx.x * kWarps + warp] = min(part_at, part_cap);
        if (part_at > part_cap) miss[m] = 1;
        if (bad) {
            worker_err[m] = MLMC_ERR_NONFINITE;
            set_status(status, MLMC_ERR_NONFINITE);
        }
    }
    energy[R * THREADS + threadIdx.x] += e0;
    if (R >= 1) {
        energy[(R - 1) * THREADS + threadIdx.x] += e1;
        counts[(R - 1) * THREADS + threadIdx.x] += (uint32_t)c1;
    }
    if (R >= 2) {
        energy[(R - 2) * THREADS + threadIdx.x] += e2;
        counts[(R - 2) * THREADS + threadIdx.x] += (uint32_t)c2;
    }
    double* out = sum_partial + ((int64_t)m * sum_ctas + blockIdx.x) * kMaxLevels;
    if (threadIdx.x < L) out[threadIdx.x] = 0.0;
    __syncthreads();
    for (int c = warp; c <= R; c += kWarps) {  // in a fixed order
        double e = 0.0;
        uint32_t n = 0;
        for (int i = lane; i < THREADS; i += 32) {
            e += energy[c * THREADS + i];
            n += counts[c * THREADS + i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
        n = __reduce_add_sync(0xFFFFFFFFu, n);
        if (lane == 0) {
            out[sh_runs.code[c]] = e;
            // the keys of interval c count in the bin above run c: it lies in no run
            if (c < R && n) atomicAdd(&hist1[(int64_t)m * kBins1 + sh_runs.top[c] + 1], n);
        }
    }
}

// Leading-digit counts of the candidates.
constexpr int kCandHistThreads = 1024;
__global__ void __launch_bounds__(kCandHistThreads, 1)
candidate_hist_kernel(const uint32_t* __restrict__ cand_keys, int64_t cand_cap, uint32_t part_cap, const uint32_t* part_n, int parts,
                      uint32_t* hist1, const int* miss, const int* worker_err) {
    extern __shared__ uint32_t sh_hist[];
    for (int b = threadIdx.x; b < kBins1; b += kCandHistThreads) sh_hist[b] = 0;
    pdl_enter();
    const int m = blockIdx.y, lane = threadIdx.x & 31;
    if (miss[m] || worker_err[m]) return;
    __syncthreads();
    for (int p = blockIdx.x * (kCandHistThreads / 32) + (threadIdx.x >> 5); p < parts; p += gridDim.x * (kCandHistThreads / 32)) {
        const uint32_t n = part_n[(int64_t)m * parts + p];
        const uint32_t* keys = cand_keys + (int64_t)m * cand_cap + (int64_t)p * part_cap;
        uint32_t i = 0;
        for (; i + 512u <= n; i += 512u) {
            uint4 q[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) q[j] = reinterpret_cast<const uint4*>(keys + i)[j * 32 + lane];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                atomicAdd(&sh_hist[q[j].x >> 16], 1u);
                atomicAdd(&sh_hist[q[j].y >> 16], 1u);
                atomicAdd(&sh_hist[q[j].z >> 16], 1u);
                atomicAdd(&sh_hist[q[j].w >> 16], 1u);
            }
        }
        for (i += lane; i < n; i += 32u) atomicAdd(&sh_hist[keys[i] >> 16], 1u);
    }
    __syncthreads();
    uint32_t* out = hist1 + (int64_t)m * kBins1;
    for (int b = threadIdx.x; b < kBins1; b += kCandHistThreads) {
        const uint32_t c = sh_hist[b];
        if (c) atomicAdd(&out[b], c);
    }
}

size_t sweep_smem(int L, int threads) {
    return (size_t)kBins1 + (size_t)(L + 1) * threads * 12 + (size_t)kSlots * threads * 4;
}

int cluster_of(const Workspace& ws, int M) { return M <= ws.limits.sample_fit ? 16 : M * 8 <= ws.sm_count ? 8 : M * 4 <= ws.sm_count ? 4 : M * 2 <= ws.sm_count ? 2 : 1; }

int sweep_blocks_of(const Workspace& ws, int M) { return std::max(1, std::min(ws.sm_count / M, ws.sum_ctas / 2)); }

}  // namespace

// One sweep instead of two: 45 us more for the sample, the candidate histogram and the launches, and up to 0.55 us less per million
// entries, the less the more keys lie in the brackets and around them.  That share is taken as the widths of the brackets plus
// kThresholdShare per threshold in the middle of the row (less towards its ends, where few keys share its bins); what it stands for
// is fitted to the times below.  us per step, adaptive p, two sweeps / one, entries of one scale and in layers of several:
//   share 3.7 %    8 x 2^25 five ranks 1155 / 1086, 1038 / 921;  ranks that double 1119 / 1071, 672 / 545
//   share 6.2 %    32 x 8.4M, ranks that double 1178 / 1187, 789 / 711;  32 x 25M 3174 / 3078, 2050 / 1718
//   share 9 %      16 x 16.8M ten ranks 1150 / 1166, 950 / 954;  128 x 2^21 five ranks 1251 / 1245, 1379 / 1336
//   share 11.5 %   32 x 8.4M ten ranks 1188 / 1249, 1020 / 1055;  32 x 25M 3375 / 3385, 2509 / 2491
//   share 14 %     16 x 16.8M 15 ranks 1144 / 1193, 917 / 971;  64 x 4.3M ten ranks 1229 / 1287, 1053 / 1111
//   share 29 %     128 x 2^21 15 ranks 1228 / 1432, 1111 / 1317
// Below 2^28 entries: 8 x 8M 245 / 249 (ranks that double) and 379 / 387 (five ranks), 16 x 4M 245 / 287.
// The sweep is bound by issue and takes a block per SM: with 75 to 98 workers, of one block each, a third of the SMs or more idle
// (80 x 3.4M, ranks that double: 1405 / 1513, 1023 / 1024).
// More levels than the columns of 24 warps have room for were not measured.
constexpr int64_t kBracketEntries = int64_t(1) << 28;
constexpr double kThresholdShare = 0.008;
bool use_brackets(const Workspace& ws, int dtype, int64_t d, int M, const int64_t* k, int L) {
    if (dtype != MLMC_F32 || d < kBracketLeast || d * M < kBracketEntries || sweep_smem(L, kSweepThreads24) > (size_t)kSweepSmemMost)
        return false;
    if (3 * sweep_blocks_of(ws, M) * M < 2 * ws.sm_count) return false;
    const double n = (double)cluster_of(ws, M) * kBlockSectors * kSectorKeys;
    double share = 0.0;
    for (int l = 0; l + 1 < L; ++l) {
        const double q = (double)k[l] / (double)d;
        if (k[l] > 0 && k[l] < d) share += 2.0 * bracket_half(q * n, n) / n + 2.0 * std::min(q, 1.0 - q) * kThresholdShare;
    }
    return share <= 0.12 - 0.02 * (double)kBracketEntries / ((double)d * M);
}

void launch_bracket_sweep(Workspace& ws, const float* g, int64_t d, int M, int64_t ld, const int64_t* k, const FinishPlan& plan,
                          cudaStream_t s) {
    const int C = cluster_of(ws, M);
    SampleRanks r = {};
    r.nq = plan.nq;
    for (int j = 0; j < r.nq; ++j) r.k[j] = (uint32_t)k[j];
    r.most = (uint32_t)(std::min(kMostRoom * (double)ws.cand_cap / (double)d, 1.0) * (C * kBlockSectors * kSectorKeys));
    const ZeroList z = selection_state(ws, MLMC_F32, d, M, r.nq, true);
    auto sample = [&](auto kernel) {
        launch_kernel_cluster(ws, K_SAMPLE, C, kernel, dim3(M * C), kSampleThreads, kBins1 * sizeof(uint32_t), s, z, r, ws.queries, g, d, ld,
                              ws.runs, ws.table1, ws.miss);
    };
    if (C == 16) sample(sample_kernel<16>);
    else if (C == 8) sample(sample_kernel<8>);
    else if (C == 4) sample(sample_kernel<4>);
    else if (C == 2) sample(sample_kernel<2>);
    else sample(sample_kernel<1>);
    constexpr int threads = kSweepThreads24;
    const int nb = sweep_blocks_of(ws, M), tpw = emit_tiles_per_worker(d, MLMC_F32);
    ws.sweep_blocks = nb;
    ws.parts = nb * (threads / 32);
    ws.part_cap = (uint32_t)(ws.cand_cap / ws.parts) & ~3u;  // parts start on 16 bytes
    launch_kernel(ws, K_BRACKET_SWEEP, bracket_sweep_kernel<threads>, dim3(nb, M), threads, sweep_smem(plan.L, threads), s, g, d, ld, plan.L,
                  ws.runs, ws.table1, ws.tile_max, tpw, ws.hist1, ws.sum_partial, ws.sum_ctas, ws.cand_keys, ws.cand_cap, ws.part_cap,
                  ws.part_n, ws.miss, M, ws.status, ws.worker_err, 1u, 0.0);
    launch_kernel(ws, K_CAND_HIST, candidate_hist_kernel, dim3(nb, M), kCandHistThreads, kBins1 * sizeof(uint32_t), s, ws.cand_keys,
                  ws.cand_cap, ws.part_cap, ws.part_n, ws.parts, ws.hist1, ws.miss, ws.worker_err);
}

void bracket_limits(KernelLimits* limits) {
    int fit[5];
    clusters_that_fit(sample_kernel<16>, kSampleThreads, kBins1 * sizeof(uint32_t), fit);
    limits->sample_fit = fit[4];
}

int configure_bracket_kernels() {
    const int hist = (int)(kBins1 * sizeof(uint32_t));
    auto set = [](auto kernel, int bytes) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    };
    return set(sample_kernel<16>, hist) && cudaFuncSetAttribute(sample_kernel<16>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                   set(sample_kernel<8>, hist) && set(sample_kernel<4>, hist) && set(sample_kernel<2>, hist) && set(sample_kernel<1>, hist) &&
                   set(bracket_sweep_kernel<kSweepThreads24>, kSweepSmemMost) && set(candidate_hist_kernel, hist)
               ? MLMC_OK
               : MLMC_ERR_CUDA;
}

}  // namespace mlmc
