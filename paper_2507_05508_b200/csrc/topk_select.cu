// Threshold selection, band norms, level probabilities and the level draw for MLMC-Top-k.
//
// The residual C^l(g) - C^{l-1}(g) of Top-k is the band of ranks (k_{l-1}, k_l] of the total order
// (|g| descending, index ascending) (Sec. 3.2).  A band is described by two thresholds: for rank k,
// T = key of the rank-k element, c = #{key > T}, n = #{key == T}, r = k - c = how many of the
// equal-key elements (in index order) are inside Top-k.  Thresholds come from an MSD radix select
// on the magnitude key: a 2^15-bin histogram of the leading digit for all queries at once, then two
// 8-bit digit passes restricted to the boundary bins (fp32 only; a bf16 key is its leading digit).
//
// Adaptive p (Lemma 3.4) makes every level boundary k_0 .. k_{L-2} a query.  With given p the level does not depend on
// the data: the host draws it before anything is launched, and only the two boundaries of the drawn band are queries.
// The boundary bins found by one such call are the next call's brackets, so that the first sweep can collect the
// boundary-bin keys itself.
//
// Launches of a selection: begin, hist1, resolve1 and, for fp32, sums_candidates and two digit passes.  The step that
// needs the whole result of a kernel runs in the block of each worker that finishes last.
#include <algorithm>

#include "topk_finish.cuh"

namespace mlmc {

namespace {

constexpr int kHistThreads = 1024;
constexpr int kResolveThreads = 1024;
constexpr int kDigitThreads = 512;

// -------------------------------------------------------------------------------------------
// begin: everything a selection accumulates into is cleared, and the queries are set up
// -------------------------------------------------------------------------------------------
struct RankList {
    uint32_t k[kMaxQueries];
    int nq;
};

__global__ void __launch_bounds__(512)
begin_adaptive_kernel(ZeroList z, RankList ranks, Query* queries, int64_t d, int M) {
    pdl_enter();
    clear_all(z);
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < M * kMaxQueries; i += gridDim.x * blockDim.x) {
        const int j = i % kMaxQueries;
        if (j < ranks.nq) queries[i] = make_query(ranks.k[j], d);
    }
}

template <int CAP>
__global__ void __launch_bounds__(512)
begin_drawn_kernel(ZeroList z, const __grid_constant__ DrawnList<CAP> drawn, Query* queries, EmitParams* emit, double* p_all,
                   int64_t d, int M, int L, const uint32_t* prev_bin, uint4* bracket) {
    pdl_enter();
    clear_all(z);
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    const DrawnBand b = drawn.band[m];
    emit[m].level = b.level;
    p_all[m * kMaxLevels] = b.p;
    queries[m * kMaxQueries] = make_query(b.k_lo, d);
    queries[m * kMaxQueries + 1] = make_query(b.k_hi, d);
    if (bracket) {
        // brackets of the first sweep: the bin where each boundary of the drawn band was found last time, and its
        // two neighbours (an empty bracket is {lo = all ones, width = 0}: bin - lo wraps to bin + 1 > 0)
        uint4 br = make_uint4(0xFFFFFFFFu, 0u, 0xFFFFFFFFu, 0u);
        if (b.level >= 1) {
            const uint32_t pb = prev_bin[m * kMaxLevels + b.level - 1];
            if (pb != kKeyNone) { br.x = pb ? pb - 1u : 0u; br.y = pb ? 2u : 1u; }
        }
        if (b.level < L - 1) {
            const uint32_t pb = prev_bin[m * kMaxLevels + b.level];
            if (pb != kKeyNone) { br.z = pb ? pb - 1u : 0u; br.w = pb ? 2u : 1u; }
        }
        bracket[m] = br;
    }
}

__global__ void uniforms_kernel(double* u_dev, int M, uint64_t seed, uint64_t step) {
    pdl_enter();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < M) u_dev[m] = counter_uniform(seed, step, (uint64_t)m);
}

// -------------------------------------------------------------------------------------------
// sweep 1: leading-digit histogram of every worker (shared-memory counts, flushed with atomics)
// -------------------------------------------------------------------------------------------
// A warp takes one batch of the emit tiles at a time (kEmitGroupVecs consecutive 16-byte vectors, four per lane, all in
// flight before the first is used) and stores the batch's largest key: the emission reads only the batches whose
// largest key reaches the lower threshold of the drawn band.
// BR (fixed p): the keys whose leading digit lies in one of the worker's two brackets (the bins around last
// call's boundary bins) are collected as candidates in the same sweep.  A batch whose largest key lies below both
// brackets is not tested (in a gradient with per-layer scales that is most batches).  Every warp stages its keys in a
// private shared-memory buffer and moves the buffer to the candidate list when it fills up (one global counter update
// per move).
// The stage is small so that the block leaves an L1 cache to the streamed vectors (with 96 KB of stages beside the 128 KB of
// counts the sweep of 16 x 11.7M keys took 170 us instead of 146).
constexpr int kWarpStage = 319;  // keys per warp stage (half a batch adds at most 256), plus one word for its count: 40 KB per block

// The key of element `at` of two vectors.
__device__ __forceinline__ uint32_t nth_key(const uint4& lo, const uint4& hi, int at) {
    const uint32_t x = (at & 4) ? hi.x : lo.x, y = (at & 4) ? hi.y : lo.y, z = (at & 4) ? hi.z : lo.z, w = (at & 4) ? hi.w : lo.w;
    const uint32_t xz = (at & 2) ? z : x, yw = (at & 2) ? w : y;
    return ((at & 1) ? yw : xz) & 0x7FFFFFFFu;
}

template <bool BR>
__global__ void __launch_bounds__(kHistThreads, 1)
hist1_kernel(const float* __restrict__ g, int64_t d, int64_t ld, uint32_t* __restrict__ hist1,
             uint32_t* __restrict__ tile_max, int tiles_per_worker, int* status, int* worker_err,
             const uint4* bracket, uint32_t* __restrict__ cand_keys, int64_t cand_cap,
             uint32_t* cand_count, int* cand_overflow, const int* only) {
    extern __shared__ uint32_t sh_hist[];
    using Tr = ElemTraits<float>;
    for (int b = threadIdx.x; b < kBins1; b += blockDim.x) sh_hist[b] = 0;
    pdl_enter();
    const int m = blockIdx.y;
    if (only && !only[m]) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // BR only: the warp's stage, its fill count in the word before it
    uint32_t* wcount = sh_hist + kBins1 + warp * (kWarpStage + 1);
    uint32_t* wstage = wcount + 1;
    uint32_t lo_a = 0xFFFFFFFFu, span_a = 0u, lo_b = 0xFFFFFFFFu, span_b = 0u;  // key ranges of the two brackets
    if (BR) {
        const uint4 br = bracket[m];
        if (br.x != 0xFFFFFFFFu) { lo_a = br.x << 16; span_a = ((br.y + 1u) << 16) - 1u; }
        if (br.z != 0xFFFFFFFFu) { lo_b = br.z << 16; span_b = ((br.w + 1u) << 16) - 1u; }
        if (lane == 0) *wcount = 0u;
    }
    uint32_t lo_min = min(lo_a, lo_b);  // no key reaches it once the list is full: the warp collects no more
    auto in_bracket = [&](uint32_t bits) -> bool {
        const uint32_t key = bits & 0x7FFFFFFFu;
        return (key - lo_a) <= span_a || (key - lo_b) <= span_b;  // an empty bracket: key - lo wraps to key + 1 > 0
    };
    auto flush_stage = [&]() {  // called by the whole warp, after a __syncwarp
        const uint32_t wfill = *wcount;
        if (wfill) {
            uint32_t base = 0;
            if (lane == 0) base = atomicAdd(&cand_count[m], wfill);
            base = __shfl_sync(0xFFFFFFFFu, base, 0);
            if ((int64_t)base + wfill <= cand_cap) {
                uint32_t* dst = cand_keys + (int64_t)m * cand_cap + base;
                for (uint32_t i = lane; i < wfill; i += 32) dst[i] = wstage[i];
            } else {
                if (lane == 0) cand_overflow[m] = 1;
                lo_min = 0xFFFFFFFFu;
            }
            __syncwarp();
            if (lane == 0) *wcount = 0u;
            __syncwarp();
        }
    };
    __syncthreads();
    const float* row = g + (int64_t)m * ld;
    uint32_t* tmax = tile_max + (int64_t)m * tiles_per_worker * kEmitGroups;
    const int64_t nvec = (d + Tr::kVec - 1) / Tr::kVec;
    const int64_t full_end = d / Tr::kVec;  // vectors that lie wholly inside the row
    bool bad = false;
    auto count_key = [&](uint32_t bits) { atomicAdd(&sh_hist[Tr::key(bits) >> Tr::kShift1], 1u); };  // Inf / NaN: see the maxima
    auto vector_max = [&](const uint4& q) -> uint32_t {  // largest key of one vector
        return max(max(q.x & 0x7FFFFFFFu, q.y & 0x7FFFFFFFu), max(q.z & 0x7FFFFFFFu, q.w & 0x7FFFFFFFu));
    };
    constexpr int kBatch = kEmitGroupVecs / 32;
    static_assert(kBatch == 4, "a warp takes a batch in one trip of four vectors per lane");
    // Groups of 32 batches are dealt round-robin to the blocks of a worker (how fast a batch is counted depends on how
    // its keys collide in the shared-memory histogram, which differs from layer to layer).
    const int nbatch = tiles_per_worker * kEmitGroups;
    const int step = gridDim.x * (kHistThreads / 32);
    for (int b = blockIdx.x * (kHistThreads / 32) + warp; b < nbatch; b += step) {
        const int64_t v = (int64_t)b * kEmitGroupVecs + lane;
        uint32_t wm;
        if ((int64_t)(b + 1) * kEmitGroupVecs <= full_end) {  // warp-uniform
            uint4 q[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + v + j * 32);
            // the next batch as far as L2 (16 x 11.7M keys, with brackets: 145 us without, now 133; the batch after it 138)
            if (lane < 16 && (int64_t)(b + step + 1) * kEmitGroupVecs <= full_end)
                prefetch_line(reinterpret_cast<const uint4*>(row) + v + (int64_t)step * kEmitGroupVecs + lane * 7);
            uint32_t vm = 0;
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                count_key(q[j].x); count_key(q[j].y); count_key(q[j].z); count_key(q[j].w);
                vm = max(vm, vector_max(q[j]));
            }
            wm = __reduce_max_sync(0xFFFFFFFFu, vm);
            if constexpr (BR) {
                if (wm >= lo_min) {  // warp-uniform
#pragma unroll
                    for (int h = 0; h < kBatch; h += 2) {
                        uint32_t cm = 0;  // bit 4 j + e: element e of vector h + j lies in a bracket
#pragma unroll
                        for (int j = 0; j < 2; ++j) {
                            cm |= in_bracket(q[h + j].x) ? (1u << (4 * j)) : 0u;
                            cm |= in_bracket(q[h + j].y) ? (2u << (4 * j)) : 0u;
                            cm |= in_bracket(q[h + j].z) ? (4u << (4 * j)) : 0u;
                            cm |= in_bracket(q[h + j].w) ? (8u << (4 * j)) : 0u;
                        }
                        if (!__any_sync(0xFFFFFFFFu, cm != 0u)) continue;
                        if (cm) {  // this lane's keys go to the warp's stage at a position taken from the warp's counter
                            uint32_t pos = atomicAdd(wcount, (uint32_t)__popc(cm));
                            for (; cm; cm &= cm - 1u) wstage[pos++] = nth_key(q[h], q[h + 1], __ffs(cm) - 1);
                        }
                        __syncwarp();
                        if (*wcount > (uint32_t)(kWarpStage - 256)) flush_stage();  // room for another half
                        __syncwarp();
                    }
                }
            }
        } else {  // the row's end, vector by vector; batches past it have the largest key 0
            uint32_t vm = 0;
            for (int64_t u = v; u < min(nvec, (int64_t)(b + 1) * kEmitGroupVecs); u += 32) {
                for_each_in_vector<float>(row, u, d, [&](int64_t, uint32_t bits) {
                    count_key(bits);
                    vm = max(vm, Tr::key(bits));
                    if (BR && in_bracket(bits)) {
                        const uint32_t at = atomicAdd(&cand_count[m], 1u);
                        if ((int64_t)at < cand_cap) cand_keys[(int64_t)m * cand_cap + at] = bits & 0x7FFFFFFFu;
                        else cand_overflow[m] = 1;
                    }
                });
            }
            wm = __reduce_max_sync(0xFFFFFFFFu, vm);
        }
        bad |= wm >= Tr::kInfKey;  // a non-finite entry shows in the largest key of its batch
        if (lane == 0) tmax[b] = wm;
    }
    if (BR) {
        __syncwarp();
        flush_stage();
    }
    if (bad && lane == 0) {
        worker_err[m] = MLMC_ERR_NONFINITE;
        set_status(status, MLMC_ERR_NONFINITE);
    }
    __syncthreads();
    uint32_t* out = hist1 + (int64_t)m * kBins1;
    for (int b = threadIdx.x; b < kBins1; b += blockDim.x) {
        const uint32_t c = sh_hist[b];
        if (c) atomicAdd(&out[b], c);
    }
}

// The same sweep for bf16 rows.  With one count per bin 32 keys meet 3.5 deep in a bank (deeper in a layer whose keys share few bins), and
// the shared-memory atomics bound the sweep (bf16: 92 % of the L1 wavefronts).  Here a bin has 16 counts, one for every second lane, so
// that at most two lanes of a warp meet in a bank.  They have room for kWindow bins, from below the octave of the largest key that a
// sample of the row holds (magnitudes with a tail have few keys there), or from that octave on where more than one sampled key of
// kColumnMisses lies in it (32 x 25.6M keys +-1: 252 us with one count per bin, 333 beside the window, now 269; clipped at one standard
// deviation 355, 347, 334).  Beside the window, down to 12 octaves below it, a bin has one count; what lies outside of that is counted
// in memory, key by key, and the lowest bin (zeros) in a register.  A block whose sample lies below the window by more than one key
// of kColumnMisses keeps one count per bin for all, and so do short rows, where the sample takes longer than it saves
// (us per step without / with columns: 8 x 1M keys 60.9 / 62.7, 32 x 1.2M 113 / 118, 8 x 2M 75.7 / 74.9, 8 x 3M 95.5 / 93.4, from 8 x 4M on with).
// 32 x 25.6M keys in layers: 401 us with one count per bin, now 311 (floor 250); 8 x 40M 164, 129; 8 x 12M 59, 53.  On the way to it, where it
// took 337: all 32 keys of a warp by the general way whenever one lies outside the window (each lane its own way 355 us); every key by the
// general way 386; windows of 22 and 24 octaves leave too little L1 for the loads in flight (362 us, and 334 without the bins beside).
// fp32 rows, with half as many atomics per byte, gain nothing (16 x 11.7M 135.4 us, 135.9 so; with the stages of the brackets beside 139 and
// 159).
constexpr int kColumns = 16;
constexpr int kFarBelow = 12 * 128, kFarAbove = 8 * 128;
constexpr uint32_t kColumnMisses = 64;
constexpr int64_t kColumnBatches = 8;  // per warp, from which on a row is long enough

struct BinCounts {
    static constexpr int kWindow = 20 * 128;  // 20 octaves: 180 KB
    static constexpr int kFarBins = kFarBelow + kWindow + kFarAbove;  // numbered through the window
    static constexpr int kWords = kWindow * kColumns + kFarBins;
    static_assert(kWords >= kBins1 && kWords % 4 == 0 && kBins1 % 4 == 0, "either kind of counts");
    // Shared memory of rows that are sampled or not.  Short rows take no more than their counts, and have a kernel without the look at
    // `columns` (8 x 3M keys, layers: 22.1 us with the columns' memory and the look, 21.2 so; 8 x 4M 24.7 and 23.4).
    __host__ __device__ static constexpr int words(bool sample) { return sample ? kWords : kBins1; }
    uint32_t* counts;
    uint32_t* out;                       // [kBins1]
    uint32_t lowest = 0, zeros = 0;      // first bin of the window; keys of bin 0
    uint32_t column0 = 0, far0 = 0;      // shared-memory addresses of bin 0 (of this lane's column, and beside the window)
    bool columns = false;                // block-uniform

    __device__ __forceinline__ BinCounts(uint32_t* shared, uint32_t* memory) : counts(shared), out(memory) {}
    // By all threads: the window, from some bins of every thread.
    template <int N>
    __device__ __forceinline__ void place(const uint32_t (&bin)[N], uint32_t* sh_warp) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        uint32_t top = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) top = max(top, bin[i]);
        top = __reduce_max_sync(0xFFFFFFFFu, top);
        if (lane == 0) sh_warp[warp] = top;
        __syncthreads();
        const uint32_t octave = __reduce_max_sync(0xFFFFFFFFu, sh_warp[lane]) & ~127u;  // of the largest key
        lowest = octave > (uint32_t)kWindow ? octave - kWindow : 0u;
        uint32_t found = 0;  // of the sample: keys of that octave, and keys below the window
#pragma unroll
        for (int i = 0; i < N; ++i) found += (bin[i] >= octave ? 1u : 0u) + (bin[i] < lowest ? 1u << 16 : 0u);
        static_assert(N * kHistThreads < 1 << 16, "16 bits each");
        found = __reduce_add_sync(0xFFFFFFFFu, found);
        __syncthreads();
        if (lane == 0) sh_warp[warp] = found;
        __syncthreads();
        found = __reduce_add_sync(0xFFFFFFFFu, sh_warp[lane]);
        columns = (found >> 16) * kColumnMisses <= (uint32_t)(N * kHistThreads);
        // (an octave less below, then: its keys are counted beside the window)
        if ((found & 0xFFFFu) * kColumnMisses > (uint32_t)(N * kHistThreads))
            lowest = octave + 128u > (uint32_t)kWindow ? octave + 128u - kWindow : 0u;
        const uint32_t base = (uint32_t)__cvta_generic_to_shared(counts);
        column0 = base + (lane & (kColumns - 1)) * 4u - lowest * (kColumns * 4u);
        far0 = base + (kWindow * kColumns + kFarBelow - (int)lowest) * 4;
    }
    __device__ __forceinline__ static void bump(uint32_t address) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(address) : "memory"); }
    __device__ __forceinline__ bool in_window(uint32_t bin) const { return bin - lowest < (uint32_t)kWindow; }
    __device__ __forceinline__ bool near(uint32_t bin) const { return bin - lowest + (uint32_t)kFarBelow < (uint32_t)kFarBins; }
    __device__ __forceinline__ void add_column(uint32_t bin) { bump(column0 + bin * (kColumns * 4u)); }
    __device__ __forceinline__ void add_near(uint32_t bin) { bump(in_window(bin) ? column0 + bin * (kColumns * 4u) : far0 + bin * 4u); }
    __device__ __forceinline__ void add(uint32_t bin) {
        if (!columns) atomicAdd(&counts[bin], 1u);
        else if (near(bin)) add_near(bin);
        else if (bin == 0u) ++zeros;
        else atomicAdd(&out[bin], 1u);
    }
    // N bins of every lane of a warp, the least and the largest known; columns only.
    template <int N>
    __device__ __forceinline__ void add_all(const uint32_t (&bin)[N], uint32_t least, uint32_t most) {
        if (__all_sync(0xFFFFFFFFu, in_window(least) && in_window(most))) {
#pragma unroll
            for (int i = 0; i < N; ++i) add_column(bin[i]);
        } else if (near(least) && near(most)) {
#pragma unroll
            for (int i = 0; i < N; ++i) add_near(bin[i]);
        } else {
#pragma unroll 1
            for (int i = 0; i < N; ++i) {
                uint32_t x = 0;
#pragma unroll
                for (int j = 0; j < N; ++j) x = i == j ? bin[j] : x;
                add(x);
            }
        }
    }
    __device__ __forceinline__ void flush() {  // by all threads, after a barrier
        if (!columns) {
            for (int b = threadIdx.x; b < kBins1; b += kHistThreads) {
                const uint32_t c = counts[b];
                if (c) atomicAdd(&out[b], c);
            }
            return;
        }
        const int lane = threadIdx.x & 31;
        zeros = __reduce_add_sync(0xFFFFFFFFu, zeros);
        if (lane == 0 && zeros) atomicAdd(&out[0], zeros);
        for (int b = threadIdx.x; b < kWindow; b += kHistThreads) {
            uint32_t c = 0;
#pragma unroll
            for (int i = 0; i < kColumns; ++i) c += counts[b * kColumns + ((i + lane) & (kColumns - 1))];
            if (c) atomicAdd(&out[lowest + b], c);
        }
        for (int b = threadIdx.x; b < kFarBins; b += kHistThreads) {
            const uint32_t c = counts[kWindow * kColumns + b];
            if (c) atomicAdd(&out[(int)lowest - kFarBelow + b], c);
        }
    }
};

template <bool SAMPLE>
__global__ void __launch_bounds__(kHistThreads, 1)
hist1_bf16_kernel(const bf16_t* __restrict__ g, int64_t d, int64_t ld, uint32_t* __restrict__ hist1, uint32_t* __restrict__ tile_max,
                  int tiles_per_worker, int* status, int* worker_err) {
    extern __shared__ __align__(16) uint32_t sh_hist[];
    __shared__ uint32_t sh_warp[kHistThreads / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < BinCounts::words(SAMPLE) / 4; i += kHistThreads) reinterpret_cast<uint4*>(sh_hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    pdl_enter();
    const int m = blockIdx.y;
    const bf16_t* row = g + (int64_t)m * ld;
    const int64_t nvec = (d + 7) / 8, full_end = d / 8;  // vectors of the row, and those wholly inside it
    BinCounts counts(sh_hist, hist1 + (int64_t)m * kBins1);
    auto keys_of = [](const uint4& q, uint32_t (&key)[8], uint32_t& least, uint32_t& most) {  // Inf / NaN: see the maxima
        const uint32_t w[4] = {q.x & 0x7FFF7FFFu, q.y & 0x7FFF7FFFu, q.z & 0x7FFF7FFFu, q.w & 0x7FFF7FFFu};
        const uint32_t hi = __vmaxu2(__vmaxu2(w[0], w[1]), __vmaxu2(w[2], w[3])), lo = __vminu2(__vminu2(w[0], w[1]), __vminu2(w[2], w[3]));
        most = max(hi & 0xFFFFu, hi >> 16);
        least = min(lo & 0xFFFFu, lo >> 16);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            key[2 * i] = w[i] & 0xFFFFu;
            key[2 * i + 1] = w[i] >> 16;
        }
    };
    if constexpr (SAMPLE) {
        uint32_t key[8], least, most;
        const int64_t share = full_end / kHistThreads;  // a vector of every thread's share of the row
        keys_of(__ldg(reinterpret_cast<const uint4*>(row) + threadIdx.x * share + (blockIdx.x * 37 + threadIdx.x * 11) % share), key, least, most);
        counts.place(key, sh_warp);
    } else {
        __syncthreads();
    }
    uint32_t* tmax = tile_max + (int64_t)m * tiles_per_worker * kEmitGroups;
    constexpr int kBatch = kEmitGroupVecs / 32;
    const int nbatch = tiles_per_worker * kEmitGroups;
    bool bad = false;
    const int step = gridDim.x * (kHistThreads / 32);
    for (int b = blockIdx.x * (kHistThreads / 32) + warp; b < nbatch; b += step) {
        const int64_t v = (int64_t)b * kEmitGroupVecs + lane;
        uint32_t vm = 0;
        if ((int64_t)(b + 1) * kEmitGroupVecs <= full_end) {  // warp-uniform
            uint4 q[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + v + j * 32);
            // the next batch as far as L2 (32 x 25.6M keys: 5 % of the kernel)
            if (lane < 16 && (int64_t)(b + step + 1) * kEmitGroupVecs <= full_end)
                prefetch_line(reinterpret_cast<const uint4*>(row) + v + (int64_t)step * kEmitGroupVecs + lane * 7);
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                uint32_t key[8], least, most;
                keys_of(q[j], key, least, most);
                if (SAMPLE && counts.columns) {
                    counts.add_all(key, least, most);
                } else {
#pragma unroll
                    for (int i = 0; i < 8; ++i) atomicAdd(&sh_hist[key[i]], 1u);
                }
                vm = max(vm, most);
            }
        } else {  // the row's end, vector by vector; batches past it have the largest key 0
            for (int64_t u = v; u < min(nvec, (int64_t)(b + 1) * kEmitGroupVecs); u += 32)
                for_each_in_vector<bf16_t>(row, u, d, [&](int64_t, uint32_t bits) {
                    counts.add(bits & 0x7FFFu);
                    vm = max(vm, bits & 0x7FFFu);
                });
        }
        vm = __reduce_max_sync(0xFFFFFFFFu, vm);
        bad |= vm >= ElemTraits<bf16_t>::kInfKey;  // a non-finite entry shows in the largest key of its batch
        if (lane == 0) tmax[b] = vm;
    }
    if (bad && lane == 0) {
        worker_err[m] = MLMC_ERR_NONFINITE;
        set_status(status, MLMC_ERR_NONFINITE);
    }
    __syncthreads();
    counts.flush();
}

// Slots of queries that share what they look for, by a warp, a query per lane.  The live queries are contiguous and equal values are
// neighbours: the slots ascend from 0, and first[slot] is the first query of each.
__device__ __forceinline__ uint32_t shared_slot(bool live, uint32_t value, uint32_t* first) {
    const int lane = threadIdx.x & 31;
    const uint32_t before = __shfl_up_sync(0xFFFFFFFFu, value, 1), lives = __ballot_sync(0xFFFFFFFFu, live);
    const bool is_first = live && (lane == 0 || !((lives >> (lane - 1)) & 1u) || before != value);
    const uint32_t slot = (uint32_t)__popc(__ballot_sync(0xFFFFFFFFu, is_first) & ((2u << lane) - 1u)) - 1u;
    if (first && is_first) first[slot] = (uint32_t)lane;
    return slot;
}

// -------------------------------------------------------------------------------------------
// after sweep 1: every live query descends into its bin
// -------------------------------------------------------------------------------------------
// One block per worker; thread t owns the 32 bins from 32 t.  One scan over the 1024 sums, then a warp per query goes through the bins of
// the thread that holds its rank.  bf16: the digit is the whole key, so the query is resolved, and the energies of the
// intervals follow from the counts.  fp32: the kernel writes the bin table of the second sweep: a bin that holds no
// threshold maps to its open interval  #{ j : bin_j > b }  (code < 64); a bin that holds one maps to 64 + its slot.
__global__ void __launch_bounds__(kResolveThreads, 1)
resolve1_kernel(const uint32_t* hist1, Query* queries, uint8_t* table1, uint32_t* cand_floor, FinishPlan pl, int is_bf16,
                int* status, int* worker_err, EmitParams* emit, const uint4* bracket, int* bracket_hit, uint32_t* prev_bin,
                unsigned long long* bracket_stats, uint32_t* cand_count, int* cand_overflow, double* p_all,
                double* delta_all, int sampled, int* miss) {
    __shared__ uint32_t sh_warp[32];
    __shared__ Query sh_q[kMaxQueries];
    __shared__ int sh_bin[kMaxQueries];
    __shared__ uint32_t sh_slot[kMaxQueries];
    __shared__ uint2 sh_owner[kMaxQueries];      // thread whose bins hold the rank, keys above those
    __shared__ double sh_E[kMaxLevels];
    __shared__ double sh_part[kMaxLevels][kResolveThreads / 32];  // bf16, adaptive
    pdl_enter();
    const int m = blockIdx.x, nq = pl.nq;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // What is needed from memory is asked for at a time: the kernel is a chain of latencies.
    constexpr int per = kBins1 / kResolveThreads;
    static_assert(per == 32 && kResolveThreads == 1024, "32 bins per thread, 32 warps");
    uint4 vectors[per / 4];
    load_bins(hist1 + (int64_t)m * kBins1 + warp * 1024, vectors);
    uint4 br = make_uint4(0u, 0u, 0u, 0u);
    int drawn_level = 0, full = 0;
    if (threadIdx.x == 32 && bracket) {
        br = bracket[m];
        drawn_level = emit[m].level;
        full = cand_overflow[m];
    }
    Query query = {};
    if (threadIdx.x < nq) query = queries[m * kMaxQueries + threadIdx.x];
    const int missed_before = miss ? miss[m] : 0;
    if (worker_err[m]) {
        if (is_bf16 && threadIdx.x == 0) fail_worker(pl, m, &emit[m]);
        return;
    }
    if (miss && !sampled && !missed_before) return;  // resolved from the sampled brackets
    uint32_t cnt[per];
    {
        extern __shared__ __align__(16) uint4 sh_vectors[];  // [32 warps][256]
        hand_over_bins(vectors, sh_vectors + warp * 256, lane, cnt);
    }
    if (threadIdx.x < nq) {
        sh_q[threadIdx.x] = query;
        sh_bin[threadIdx.x] = -1;
        sh_owner[threadIdx.x] = make_uint2(0xFFFFFFFFu, 0u);
    }
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < per; ++i) sum += cnt[i];
    uint32_t suffix = sum;  // inclusive suffix sum within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_down_sync(0xFFFFFFFFu, suffix, o);
        if (lane + o < 32) suffix += y;
    }
    if (lane == 0) sh_warp[warp] = suffix;
    __syncthreads();
    uint32_t above = suffix - sum;  // keys in the bins above this thread's
    {
        const uint32_t w = sh_warp[lane];
        above += __reduce_add_sync(0xFFFFFFFFu, lane > warp ? w : 0u);
    }
    const int b0 = threadIdx.x * per;
    for (int j = 0; j < nq; ++j) {
        const uint32_t k = sh_q[j].k;
        if (sh_q[j].trivial == 0u && above < k && k <= above + sum) sh_owner[j] = make_uint2(threadIdx.x, above);  // whose bins hold rank k
    }
    __syncthreads();
    // A warp per query goes through the owner's 32 bins, which are still in shared memory.  (The owner alone, one query after the other where
    // a thread or a warp has several: 3 us more with 14 queries.)
    if (warp < nq && sh_q[warp].trivial == 0u && sh_owner[warp].x < (uint32_t)kResolveThreads) {
        extern __shared__ __align__(16) uint4 sh_vectors[];
        const uint32_t k = sh_q[warp].k, owner = sh_owner[warp].x, group = owner & 31u, i = 31u - lane;  // lane 0: the largest bin
        const uint32_t c = reinterpret_cast<const uint32_t*>(sh_vectors + (owner & ~31u) * 8u + group * 8u + (((i >> 2) ^ group) & 7u))[i & 3u];
        uint32_t upto = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if (lane >= o) upto += y;
        }
        const uint32_t ab = sh_owner[warp].y + upto - c;
        if (ab < k && k <= ab + c) {  // the largest bin b with #{digit >= b} >= k
            sh_bin[warp] = (int)(owner * per + i);
            sh_q[warp].c = ab;
            sh_q[warp].n = c;
            sh_q[warp].r = k - ab;
            if (is_bf16) sh_q[warp].T = owner * per + i;
        }
    }
    if (threadIdx.x < nq && sh_q[threadIdx.x].trivial)  // "nothing inside" sits above every bin, "everything inside" below
        sh_bin[threadIdx.x] = (sh_q[threadIdx.x].trivial == 2u) ? -1 : kBins1;
    __syncthreads();
    if (sampled) {
        // The histogram holds the keys of the sampled brackets only, and between them the number of keys there: a threshold
        // that does not lie in a bracket, or a full candidate list, sends the worker through the sweeps of the whole row.
        bool out = missed_before != 0;
        if (threadIdx.x < nq && sh_q[threadIdx.x].trivial == 0u) {
            const int bin = sh_bin[threadIdx.x];
            out |= bin < 0 || table1[(int64_t)m * kBins1 + bin] != nq + 1;  // so marked by the sample
        }
        const bool left_out = missed_before == kLeftOut;
        const bool missed = __syncthreads_or(out);
        if (threadIdx.x == 0) atomicAdd(&bracket_stats[4 + (!missed ? 0 : left_out ? 2 : 1)], 1ull);
        if (missed) {
            if (threadIdx.x == 0 && !left_out) miss[m] = 1;
            uint4* h = reinterpret_cast<uint4*>(const_cast<uint32_t*>(hist1) + (int64_t)m * kBins1);
            for (int i = threadIdx.x; i < kBins1 / 4; i += kResolveThreads) h[i] = make_uint4(0u, 0u, 0u, 0u);
            return;
        }
    }
    if (is_bf16) {
        if (pl.adaptive) {
            // open-interval energies: a bin lies in interval #{ j : bin_j > b } unless it is a threshold.  A thread's
            // bins meet few intervals; per interval a warp adds its lanes' shares, then the warp sums in warp order.
            for (int l = 0; l < pl.L; ++l) {
                double e = 0.0;
                const int hi = l ? sh_bin[l - 1] : kBins1, lo = (l < nq) ? sh_bin[l] : -1;  // bins strictly between
                if (sum != 0u && lo < b0 + per - 1 && hi > b0) {
#pragma unroll
                    for (int i = 0; i < per; ++i)
                        if (cnt[i] != 0u && b0 + i > lo && b0 + i < hi) {  // an empty bin may encode Inf / NaN
                            const double x = (double)__uint_as_float((uint32_t)(b0 + i) << 16);
                            e = fma((double)cnt[i], x * x, e);
                        }
                }
                if (__any_sync(0xFFFFFFFFu, e != 0.0)) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
                }
                if (lane == 0) sh_part[l][warp] = e;
            }
            __syncthreads();
            for (int l = warp; l < pl.L; l += kResolveThreads / 32) {
                double e = sh_part[l][lane];
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
                if (lane == 0) sh_E[l] = e;
            }
            __syncthreads();
        }
        finish_selection(pl, m, 1, sh_q, sh_E, p_all, delta_all, emit[m].level, p_all[m * kMaxLevels], &emit[m], status, worker_err);
        return;
    }
    // slots of the second digit pass: live queries in the same bin share one (bins descend with j)
    if (warp == 0) {
        const int j = lane;
        const bool live = j < nq && sh_q[j].trivial == 0u;
        const uint32_t slot = shared_slot(live, live ? (uint32_t)sh_bin[j] : 0u, nullptr);
        if (j < nq) {
            sh_slot[j] = live ? slot : kNoSlot;
            Query q = sh_q[j];
            if (live) {
                q.prefix = (uint32_t)sh_bin[j] << 16;
                q.rem = q.r;
                q.slot = q.slot2 = slot;
            }
            queries[m * kMaxQueries + j] = q;
        }
    }
    if (threadIdx.x == 32) {
        // the smallest key that can be a candidate: the lower edge of the lowest boundary bin (no live query: none)
        int lowest = kBins1;
        bool hit = true, had = false;
        for (int j = 0; j < nq; ++j) {
            const int bin = sh_bin[j];
            if (bin >= 0 && bin < lowest) lowest = bin;
        }
        cand_floor[m] = (lowest < kBins1) ? ((uint32_t)lowest << 16) : 0xFFFFFFFFu;
        if (bracket) {
            // Did the first sweep already collect the keys of both boundary bins of the drawn band?  If not, its
            // candidates are dropped and the candidate sweep runs.  Either way the bins are remembered.
            const int lv = drawn_level;
            hit = full == 0;
            for (int j = 0; j < nq; ++j) {
                if (sh_q[j].trivial) continue;
                const uint32_t bin = (uint32_t)sh_bin[j];
                had |= (j ? br.z : br.x) != 0xFFFFFFFFu;
                hit &= j ? (bin - br.z) <= br.w : (bin - br.x) <= br.y;
                prev_bin[m * kMaxLevels + lv - 1 + j] = bin;
            }
            bracket_hit[m] = hit ? 1 : 0;
            if (!hit) {
                cand_count[m] = 0u;
                cand_overflow[m] = 0;
            }
            atomicAdd(&bracket_stats[hit ? 0 : (had ? 1 : 2)], 1ull);
        }
    }
    __syncthreads();
    {
        // code of bin b: the number of leading queries whose bin lies above b, or 64 + slot if the first one that does
        // not lies in b itself.  Nearly every thread's 32 bins have one code.
        int j = 0;
        while (j < nq && sh_bin[j] > b0 + per - 1) ++j;
        uint4* tab = reinterpret_cast<uint4*>(table1 + (int64_t)m * kBins1 + b0);
        if (j == nq || sh_bin[j] < b0) {
            const uint32_t v = (uint32_t)j * 0x01010101u;
            tab[0] = tab[1] = make_uint4(v, v, v, v);
        } else {
            uint32_t w[8];
#pragma unroll
            for (int i = per - 1; i >= 0; --i) {
                const int b = b0 + i;
                while (j < nq && sh_bin[j] > b) ++j;
                const uint32_t code = (j < nq && sh_bin[j] == b) ? 64u + sh_slot[j] : (uint32_t)j;
                w[i / 4] = ((i & 3) == 3) ? (code << 24) : (w[i / 4] | (code << (8 * (i & 3))));
            }
            tab[0] = make_uint4(w[0], w[1], w[2], w[3]);
            tab[1] = make_uint4(w[4], w[5], w[6], w[7]);
        }
    }
}

// -------------------------------------------------------------------------------------------
// sweep 2 (fp32): per-interval energy of the bins that hold no threshold, and compaction of the keys
// of the bins that do ("candidates": a few percent of the data) for the remaining digit passes
// -------------------------------------------------------------------------------------------
// A warp takes one batch of the emit tiles at a time (four 16-byte vectors per lane, the next batch's vectors in flight) and
// nothing is exchanged between warps before the end: the energies are added up per thread (fp64, a column of shared memory per
// interval and thread), the candidates wait in slots of the thread's own, and a warp moves them on when a lane's fill up.
//   groups: 16 consecutive bins share a word {which of them hold a threshold (high half), boundary bins above the 16 (low
//   half)}: the interval of a key is the latter plus the bits at or above its bin.  The gradient's magnitudes in a warp fall
//   into a few dozen of the 2048 words, most of them in different banks; looked up bin by bin the banks collide three times.
//   A candidate's energy goes to a column that nobody reads, so that an entry costs no branch.
//   Below the lowest boundary bin there is one interval and no candidate: a batch whose largest key (recorded by the first
//   sweep) lies below is added to a register without a look-up.  In a gradient with per-layer scales those are whole layers.
// Without energies (given p) only the batches that reach the lowest boundary bin are read at all.
// The columns bound the kernel (load and store, two shared-memory wavefronts each, of about 6 per warp and entry), with the
// arithmetic pipe close behind; where no batch is looked up, DRAM does.
constexpr int kS2Threads = 1024;      // 512 where the columns of 1024 threads do not fit (many levels)
constexpr int kS2Slots = 8;           // candidates per thread; a vector adds at most 4
constexpr int kS2Groups = kBins1 / 16;
constexpr int kS2SmemMost = 226 * 1024;  // beside the static arrays

template <bool SUMS>
__global__ void __launch_bounds__(kS2Threads, 1)
sums_candidates_kernel(const float* __restrict__ g, int64_t d, int64_t ld, const uint8_t* table, const Query* queries, int nq, int L,
                       double* __restrict__ sum_partial, int sum_ctas,
                       uint32_t* __restrict__ cand_keys, int64_t cand_cap, uint32_t* cand_count, int* cand_overflow,
                       const int* worker_err, const uint32_t* tile_max,
                       int tiles_per_worker, const uint32_t* cand_floor, const int* bracket_hit, const int* only) {
    extern __shared__ __align__(16) uint8_t sh_raw[];
    __shared__ uint8_t sh_above[kMaxLevels + 1];   // boundary bins above a bin of code j
    __shared__ uint8_t sh_code[kMaxLevels + 1];    // interval (number of thresholds above) with so many boundary bins above it
    const int threads = blockDim.x, warps = threads / 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* sh_group = reinterpret_cast<uint32_t*>(sh_raw);                                        // [kS2Groups]
    uint32_t* slots = sh_group + kS2Groups + threadIdx.x;                                            // [kS2Slots][threads]
    double* column = reinterpret_cast<double*>(sh_group + kS2Groups + kS2Slots * threads);           // [L + 1][threads]  (SUMS)
    double* mine = column + threadIdx.x;
    pdl_enter();
    const int m = blockIdx.y;
    if (worker_err[m] || (only && !only[m])) return;
    if (!SUMS && bracket_hit && bracket_hit[m]) return;  // the first sweep collected every boundary-bin key already
    const uint32_t floor_key = cand_floor[m];
    if (warp == 0) {  // queries share boundary bins: the live ones are contiguous, their slots ascend
        const Query q = queries[m * kMaxQueries + min(lane, nq > 0 ? nq - 1 : 0)];
        const bool live = lane < nq && q.trivial == 0u;
        const uint32_t slot = live ? q.slot : kNoSlot, next = __shfl_down_sync(0xFFFFFFFFu, slot, 1);
        const uint32_t none = __ballot_sync(0xFFFFFFFFu, lane < nq && q.trivial == 1u);  // k = 0: thresholds above every bin
        if (lane == 0) {
            sh_above[0] = 0;
            sh_code[0] = (uint8_t)__popc(none);
        }
        if (live) {
            sh_above[lane + 1] = (uint8_t)(slot + 1u);
            if (lane == 31 || next != slot) sh_code[slot + 1u] = (uint8_t)(lane + 1);
        } else if (lane < nq) {
            sh_above[lane + 1] = 0;
        }
    }
    if (SUMS)
        for (int l = 0; l <= L; ++l) mine[l * threads] = 0.0;
    __syncthreads();
    for (int i = threadIdx.x; i < kS2Groups; i += threads) {
        const uint4 x = reinterpret_cast<const uint4*>(table + (int64_t)m * kBins1)[i];
        auto boundary = [](uint32_t w) {  // bit i: code i of the four is 64 or more
            const uint32_t c = __vcmpgeu4(w, 0x40404040u);
            return (c & 1u) | ((c >> 7) & 2u) | ((c >> 14) & 4u) | ((c >> 21) & 8u);
        };
        const uint32_t mask = boundary(x.x) | boundary(x.y) << 4 | boundary(x.z) << 8 | boundary(x.w) << 12, top = x.w >> 24;
        sh_group[i] = mask << 16 | (top >= 64u ? top - 64u : sh_above[top]);
    }
    __syncthreads();
    const float* row = g + (int64_t)m * ld;
    uint32_t* cand = cand_keys + (int64_t)m * cand_cap;
    const uint32_t* tmax = tile_max + (int64_t)m * tiles_per_worker * kEmitGroups;

    const uint32_t slots0 = (uint32_t)__cvta_generic_to_shared(slots), step = (uint32_t)threads * 4u;
    uint32_t at = slots0;
    bool over = false;  // without energies: the list is full (warp-uniform)
    auto flush = [&]() {  // called by the whole warp
        const uint32_t n = (at - slots0) / step;
        uint32_t upto = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if (lane >= o) upto += y;
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, upto, 31);
        if (total == 0u) return;
        uint32_t base = 0;
        if (lane == 0) base = atomicAdd(&cand_count[m], total);
        base = __shfl_sync(0xFFFFFFFFu, base, 0);
        if ((int64_t)base + total <= cand_cap) {
            uint32_t* to = cand + base + (upto - n);
            for (uint32_t i = 0; i < n; ++i) to[i] = slots[i * threads] & 0x7FFFFFFFu;
        } else {
            if (!SUMS) over = true;
            if (lane == 0) cand_overflow[m] = 1;  // too many keys share the boundary bins: the full-sweep passes take over
        }
        at = slots0;
    };
    double low[2] = {0.0, 0.0};  // energy of the batches below the floor
    auto add_low = [&](const uint4& q) {
        const double x0 = (double)__uint_as_float(q.x), x1 = (double)__uint_as_float(q.y), x2 = (double)__uint_as_float(q.z),
                     x3 = (double)__uint_as_float(q.w);
        low[0] = fma(x0, x0, low[0]);
        low[1] = fma(x1, x1, low[1]);
        low[0] = fma(x2, x2, low[0]);
        low[1] = fma(x3, x3, low[1]);
    };
    auto look_up = [&](uint32_t bits) -> uint32_t {  // byte offset of the group's word: four times key bits 30..20
        return *reinterpret_cast<const uint32_t*>(sh_raw + ((bits >> 18) & 0x1FFCu));
    };
    auto take = [&](uint32_t bits, uint32_t group) -> uint32_t {  // bit 0: a candidate
        const uint32_t u = __funnelshift_r(group, 0u, (bits >> 16) | 16u);  // the boundary bins from the key's own upwards
        if (SUMS) {
            const uint32_t n = (u & 1u) ? (uint32_t)L : (group & 0xFFFFu) + (uint32_t)__popc(u);
            double* a = mine + n * (uint32_t)threads;
            const double x = (double)__uint_as_float(bits);
            *a = fma(x, x, *a);
        }
        return u;
    };
    auto set_aside = [&](uint32_t u, uint32_t bits) { shared_push_if_negative((int)(u << 31), at, bits, step); };
    auto full = [&]() -> bool { return __any_sync(0xFFFFFFFFu, at > slots0 + (kS2Slots - 4) * step); };

    // Batches are dealt round-robin to the warps of all blocks of the worker: which batches are costly differs from layer to
    // layer.  A lane looks at the largest key of one of the warp's next 32 batches.
    const int nbatch = (int)((d + kBatchKeys - 1) / kBatchKeys), stride = gridDim.x * warps;
    auto load = [&](int b, uint4 (&q)[4]) {
        if ((int64_t)(b + 1) * kBatchKeys > d) return;  // the row's ragged end
#pragma unroll
        for (int j = 0; j < 4; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + (int64_t)b * kEmitGroupVecs + j * 32 + lane);
    };
    for (int64_t base = blockIdx.x * warps + warp; base < nbatch; base += (int64_t)32 * stride) {
        const int64_t own = base + (int64_t)lane * stride;
        const uint32_t high = __ballot_sync(0xFFFFFFFFu, own < nbatch && tmax[min(own, (int64_t)nbatch - 1)] >= floor_key);
        uint32_t todo = SUMS ? __ballot_sync(0xFFFFFFFFu, own < nbatch) : high;
        if (!todo) continue;
        uint4 cur[4], nxt[4];
        load((int)base + (__ffs(todo) - 1) * stride, nxt);
        while (todo) {
            const int i = __ffs(todo) - 1, b = (int)base + i * stride;
            todo &= todo - 1u;
#pragma unroll
            for (int j = 0; j < 4; ++j) cur[j] = nxt[j];
            if (todo) load((int)base + (__ffs(todo) - 1) * stride, nxt);
            if ((int64_t)(b + 1) * kBatchKeys > d) {
                for (int64_t e = (int64_t)b * kBatchKeys + lane; e - lane < d; e += 32) {
                    if (e < d) {
                        const uint32_t bits = reinterpret_cast<const uint32_t*>(row)[e];
                        set_aside(take(bits, look_up(bits)), bits);
                    }
                    __syncwarp();
                    if (full()) flush();
                }
            } else if (SUMS && !((high >> i) & 1u)) {
#pragma unroll
                for (int j = 0; j < 4; ++j) add_low(cur[j]);
            } else {
                if (!SUMS && over) return;  // nothing is left to do (a warp's own barriers only from here on)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint32_t g0 = look_up(cur[j].x), g1 = look_up(cur[j].y), g2 = look_up(cur[j].z), g3 = look_up(cur[j].w);
                    const uint32_t u0 = take(cur[j].x, g0), u1 = take(cur[j].y, g1), u2 = take(cur[j].z, g2), u3 = take(cur[j].w, g3);
                    if (__any_sync(0xFFFFFFFFu, ((u0 | u1 | u2 | u3) & 1u) != 0u)) {  // a store takes its turn even if no lane has one
                        set_aside(u0, cur[j].x);
                        set_aside(u1, cur[j].y);
                        set_aside(u2, cur[j].z);
                        set_aside(u3, cur[j].w);
                        if (full()) flush();
                    }
                }
            }
        }
    }
    __syncwarp();
    flush();
    if (SUMS) {
        const uint32_t lowest = sh_group[0], last = (lowest & 0xFFFFu) + (uint32_t)__popc(lowest >> 16);  // the interval below all
        mine[last * threads] += low[0] + low[1];
        if (threadIdx.x < L) sum_partial[((int64_t)m * sum_ctas + blockIdx.x) * kMaxLevels + threadIdx.x] = 0.0;
        __syncthreads();
        for (uint32_t c = warp; c <= last; c += warps) {  // in a fixed order
            double e = 0.0;
            for (int i = lane; i < threads; i += 32) e += column[c * threads + i];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
            if (lane == 0) sum_partial[((int64_t)m * sum_ctas + blockIdx.x) * kMaxLevels + sh_code[c]] = e;
        }
    }
}

// -------------------------------------------------------------------------------------------
// the two remaining digits (fp32), the energies of the boundary bins, and the end of the selection
// -------------------------------------------------------------------------------------------
// Both passes run over the compacted candidate keys, or over the whole row for a worker whose candidate buffer
// overflowed (many equal magnitudes).  The block of a worker that finishes last descends the queries.
// Pass 2 counts the second digit per boundary bin.  Its result splits every boundary bin into sub-bins: one that holds
// a threshold is counted by pass 3 digit by digit (its keys are then known exactly), any other lies wholly inside one
// interval, and pass 3 adds up its energy (adaptive p).  All keys of a boundary bin share their exponent, so
// g^2 = mant^2 2^(2 (max(e,1) - 150)) with a 48-bit integer mant^2, and the sums are taken in integers, where the
// (changing) order of the candidates does not matter.  An energy cell is a (boundary bin, interval) pair, numbered
// slot + interval (a threshold adds one to the interval, a boundary bin one to the slot: the sum is unique).
// The cells are kept as three 16-bit limbs in u32 words, one copy per lane: a warp's additions never meet in a bank,
// and a word takes 2^16 additions before it can overflow (kLimbTrips trips of at most 4 keys per lane and 16 warps).
constexpr int kCellWords = kEnergyCells * 3 * 32;
constexpr int kLimbTrips = 65536 / (4 * (kDigitThreads / 32));

// The candidates of a worker whose brackets held (topk_bracket.cu): `n` parts of `cap` keys each.
struct CandParts {
    const int* miss;         // null: no brackets
    uint32_t* count;         // [M][n]; pass 2 leaves the number of the keys that pass 3 needs
    int n;
    uint32_t cap;
    int n_sum;               // energy sums per interval that the sweep left
};

// The grid has kDigitBlocks blocks per SM, and the compiler may use the registers of as many: left to itself it takes 32 for the third
// digit with energies and spills (16 x 11.7M fp32 keys, 31 levels: 56 us, 46 with 40 registers, 42 so; the step 923, now 884).
constexpr int kDigitBlocks = 2;

template <int PASS, bool SUMS>
__global__ void __launch_bounds__(kDigitThreads, kDigitBlocks)
digit_pass_kernel(const float* __restrict__ g, int64_t d, int64_t ld, uint32_t* cand_keys, int64_t cand_cap,
                  const uint32_t* cand_count, const int* cand_overflow, const uint8_t* table1, uint8_t* map2,
                  uint32_t* hist_out, uint32_t* done, Query* queries, FinishPlan pl, unsigned long long* cand_S,
                  double* sum_partial, int sum_ctas, int n_sum, int* status, int* worker_err, EmitParams* emit,
                  double* p_all, double* delta_all, CandParts parts) {
    extern __shared__ __align__(16) uint32_t sh_digit[];  // [nq][256] counts, then (PASS 3, SUMS) the cells or (PASS 2, parts) the columns
    __shared__ Query sh_q[kMaxQueries];
    __shared__ double sh_E[kMaxLevels];
    pdl_enter();
    const int m = blockIdx.y, nq = pl.nq;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // asked for at a time, and the queries before the last block needs them
    const uint32_t listed = cand_count[m];
    const int full = cand_overflow[m], missed = SUMS && parts.miss ? parts.miss[m] : 1, bad = worker_err[m];
    if (threadIdx.x < nq) sh_q[threadIdx.x] = queries[m * kMaxQueries + threadIdx.x];
    if (bad) {
        if (PASS == 3 && blockIdx.x == 0 && threadIdx.x == 0) fail_worker(pl, m, &emit[m]);
        return;
    }
    uint32_t* sh_hist = sh_digit;
    uint32_t* sh_cell = sh_digit + nq * kBins23;
    const bool in_parts = SUMS && !missed;
    const bool over = !in_parts && full != 0;
    const uint32_t n = over || in_parts ? 0u : listed;
    uint32_t* out = hist_out + (int64_t)m * kMaxQueries * kBins23;
    // pass 2, parts: energy of the keys of a run's bins without a threshold, a column per interval and thread; the order of
    // the keys in the parts is fixed, so the sums are too
    constexpr bool COLUMNS = PASS == 2 && SUMS;
    double* column = reinterpret_cast<double*>(sh_digit + nq * kBins23) + threadIdx.x;
    if (over || (in_parts ? (uint64_t)blockIdx.x * (kDigitThreads / 32) < (uint64_t)parts.n : (uint64_t)blockIdx.x * kDigitThreads < n)) {
        constexpr bool CELLS = PASS == 3 && SUMS;
        if (COLUMNS && in_parts)
            for (int l = 0; l < pl.L; ++l) column[l * kDigitThreads] = 0.0;
        for (int i = threadIdx.x; i < nq * kBins23 + (CELLS ? kCellWords : 0); i += kDigitThreads) sh_digit[i] = 0u;
        __syncthreads();
        const uint8_t* tab = table1 + (int64_t)m * kBins1;
        const uint8_t* mp = map2 + (int64_t)m * kMaxQueries * kBins23;
        auto take = [&](uint32_t key, uint32_t code) {  // code: of the key's leading digit
            if (code < 64u) return;  // a bracket bin that holds no threshold after all
            const uint32_t s2 = code - 64u;
            if (PASS == 2) {
                atomicAdd(&sh_hist[s2 * kBins23 + ((key >> 8) & 0xFFu)], 1u);
            } else {
                const uint32_t c = mp[s2 * kBins23 + ((key >> 8) & 0xFFu)];
                if (c < 64u) {
                    atomicAdd(&sh_hist[c * kBins23 + (key & 0xFFu)], 1u);
                } else if (SUMS) {
                    const uint32_t mant = (key & 0x7FFFFFu) | ((key >> 23) ? 0x800000u : 0u);
                    const uint64_t m2 = (uint64_t)mant * mant;
                    uint32_t* a = sh_cell + (c - 64u) * 96u + lane;
                    atomicAdd(a, (uint32_t)m2 & 0xFFFFu);
                    atomicAdd(a + 32, (uint32_t)(m2 >> 16) & 0xFFFFu);
                    atomicAdd(a + 64, (uint32_t)(m2 >> 32));
                }
            }
        };
        auto flush_cells = [&]() {  // called by all threads
            __syncthreads();
            unsigned long long* S = cand_S + (int64_t)m * kEnergyCells * 2;
            for (int c = warp; c < kEnergyCells; c += kDigitThreads / 32) {
                const uint32_t l0 = sh_cell[c * 96 + lane], l1 = sh_cell[c * 96 + 32 + lane], l2 = sh_cell[c * 96 + 64 + lane];
                sh_cell[c * 96 + lane] = sh_cell[c * 96 + 32 + lane] = sh_cell[c * 96 + 64 + lane] = 0u;
                if (!__any_sync(0xFFFFFFFFu, (l0 | l1 | l2) != 0u)) continue;
                unsigned long long lo = (unsigned long long)l0 + ((unsigned long long)l1 << 16), hi = l2;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    lo += __shfl_xor_sync(0xFFFFFFFFu, lo, o);
                    hi += __shfl_xor_sync(0xFFFFFFFFu, hi, o);
                }
                // sum = hi 2^32 + lo, carried separately: 2^32 keys (the longest row) fit each half
                if (lane == 0) {
                    atomicAdd(&S[c * 2], lo);
                    atomicAdd(&S[c * 2 + 1], hi);
                }
            }
            __syncthreads();
        };
        int trips = 0;
        const uint32_t stride = gridDim.x * kDigitThreads;
        if (in_parts && PASS == 2) {
            // First the energies of the keys whose bin holds no threshold, four vectors in flight per lane (the others go to a
            // column that nobody reads, and to the front of the part); then the digits of those.  (Digits and energies in one
            // loop, both ways of every key: 105 us for 25M keys, now 87.)
            uint8_t* code_of = reinterpret_cast<uint8_t*>(column - threadIdx.x + (pl.L + 1) * kDigitThreads);
            for (int i = threadIdx.x; i < kBins1 / 16; i += kDigitThreads)
                reinterpret_cast<uint4*>(code_of)[i] = reinterpret_cast<const uint4*>(tab)[i];
            __syncthreads();
            for (int p = blockIdx.x * (kDigitThreads / 32) + warp; p < parts.n; p += gridDim.x * (kDigitThreads / 32)) {
                const uint32_t np = parts.count[(int64_t)m * parts.n + p];
                uint32_t* cand = cand_keys + (int64_t)m * cand_cap + (int64_t)p * parts.cap;
                uint32_t kept = 0;
                auto one = [&](uint32_t key, bool there) {
                    const uint32_t code = there ? code_of[key >> 16] : 0u;
                    const bool keep = code >= 64u;
                    if (there) {
                        double* a = column + (keep ? pl.L : (int)code) * kDigitThreads;
                        const double x = (double)__uint_as_float(key);
                        *a = fma(x, x, *a);
                    }
                    const uint32_t kept_mask = __ballot_sync(0xFFFFFFFFu, keep);
                    if (keep) cand[kept + __popc(kept_mask & ((1u << lane) - 1u))] = key;
                    kept += __popc(kept_mask);
                };
                uint32_t i = 0;
                // The keys are kept in place: kept <= i where a trip starts, but its writes reach up to its own last key.  Every lane
                // has its keys of a trip before the first write.
                for (; i + 512u <= np; i += 512u) {
                    uint4 q[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) q[j] = reinterpret_cast<const uint4*>(cand + i)[j * 32 + lane];
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        one(q[j].x, true);
                        one(q[j].y, true);
                        one(q[j].z, true);
                        one(q[j].w, true);
                    }
                }
                for (; i < np; i += 32u) {
                    const uint32_t key = i + lane < np ? cand[i + lane] : 0u;
                    __syncwarp();
                    one(key, i + lane < np);
                }
                __syncwarp();
                for (uint32_t k = lane; k < kept; k += 32u) take(cand[k], code_of[cand[k] >> 16]);
                if (lane == 0) parts.count[(int64_t)m * parts.n + p] = kept;
            }
        } else if (in_parts) {
            constexpr int kAhead = 8;  // keys in flight per lane
            constexpr uint32_t kTrip = 32 * kAhead;
            for (int p0 = blockIdx.x * (kDigitThreads / 32); p0 < parts.n; p0 += gridDim.x * (kDigitThreads / 32)) {  // block-uniform
                const int p = p0 + warp;
                const uint32_t np = p < parts.n ? parts.count[(int64_t)m * parts.n + p] : 0u;
                const uint32_t* cand = cand_keys + (int64_t)m * cand_cap + (int64_t)p * parts.cap;
                uint32_t i = 0;
                for (;;) {
                    const uint32_t stop = CELLS ? min(np, i + kTrip * (kLimbTrips * 4 / kAhead)) : np;
                    for (; i < stop; i += kTrip) {
                        uint32_t key[kAhead], code[kAhead];
#pragma unroll
                        for (int j = 0; j < kAhead; ++j) key[j] = i + j * 32 + lane < np ? cand[i + j * 32 + lane] : 0xFFFFFFFFu;
#pragma unroll
                        for (int j = 0; j < kAhead; ++j) code[j] = key[j] != 0xFFFFFFFFu ? tab[key[j] >> 16] : 0u;
#pragma unroll
                        for (int j = 0; j < kAhead; ++j)
                            if (key[j] != 0xFFFFFFFFu) take(key[j], code[j]);
                    }
                    if (!CELLS || !__syncthreads_or(i < np)) break;
                    flush_cells();
                }
                if (CELLS && p0 + (int)(gridDim.x * (kDigitThreads / 32)) < parts.n) flush_cells();
            }
        } else if (!over) {
            const uint32_t* cand = cand_keys + (int64_t)m * cand_cap;
            for (uint64_t base = blockIdx.x * kDigitThreads; base < n; base += 4ull * stride) {  // block-uniform
                uint32_t key[4], code[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint64_t i = base + threadIdx.x + (uint64_t)j * stride;
                    key[j] = (i < n) ? cand[i] : 0u;
                    code[j] = (i < n) ? 64u : 0u;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (code[j]) code[j] = tab[key[j] >> 16];
#pragma unroll
                for (int j = 0; j < 4; ++j) take(key[j], code[j]);
                if (CELLS && ++trips == kLimbTrips) {
                    trips = 0;
                    flush_cells();
                }
            }
        } else {
            const float* row = g + (int64_t)m * ld;
            const int64_t nvec = (d + 3) / 4;
            for (int64_t v0 = (int64_t)blockIdx.x * kDigitThreads; v0 < nvec; v0 += stride) {  // block-uniform
                if (v0 + threadIdx.x < nvec)
                    for_each_in_vector<float>(row, v0 + threadIdx.x, d, [&](int64_t, uint32_t bits) {
                        const uint32_t key = bits & 0x7FFFFFFFu;
                        take(key, tab[key >> 16]);
                    });
                if (CELLS && ++trips == kLimbTrips) {
                    trips = 0;
                    flush_cells();
                }
            }
        }
        if (CELLS) flush_cells();
        __syncthreads();
        for (int i = threadIdx.x; i < nq * kBins23; i += kDigitThreads) {
            const uint32_t c = sh_hist[i];
            if (c) atomicAdd(&out[i], c);
        }
    }
    if (COLUMNS && in_parts) {  // behind the sums of the sweep
        const bool used = blockIdx.x * (kDigitThreads / 32) < parts.n;
        for (int l = warp; l < pl.L; l += kDigitThreads / 32) {
            double e = 0.0;
            if (used)
                for (int i = lane; i < kDigitThreads; i += 32) e += column[l * kDigitThreads + i - (int)threadIdx.x];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
            if (lane == 0) sum_partial[((int64_t)m * sum_ctas + parts.n_sum + blockIdx.x) * kMaxLevels + l] = e;
        }
    }
    if (!last_block(&done[m], gridDim.x)) return;

    // one warp per query walks its 256-bin histogram from the top digit down
    __shared__ uint32_t sh_digit_of[kMaxQueries];
    for (int j = warp; j < nq; j += kDigitThreads / 32) {
        if (sh_q[j].trivial) continue;
        const uint32_t* h = out + sh_q[j].slot * kBins23;
        uint32_t cnt[8], local = 0;  // lane 0 owns the top 8 digits (255..248), lane 31 the bottom 8
#pragma unroll
        for (int i = 0; i < 8; ++i) cnt[i] = __ldcg(&h[255 - (lane * 8 + i)]);
#pragma unroll
        for (int i = 0; i < 8; ++i) local += cnt[i];
        uint32_t inc = local;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
            if (lane >= o) inc += y;
        }
        const uint32_t rem = sh_q[j].rem;
        __syncwarp();
        if (inc >= rem && inc - local < rem) {
            uint32_t above = inc - local;
            for (int i = 0; i < 8; ++i) {
                if (above + cnt[i] >= rem) {
                    const uint32_t digit = 255u - (uint32_t)(lane * 8 + i);
                    if (PASS == 2) {
                        sh_q[j].prefix |= digit << 8;
                        sh_q[j].rem = rem - above;
                        sh_digit_of[j] = digit;
                    } else {
                        sh_q[j].T = sh_q[j].prefix | digit;
                        sh_q[j].r = rem - above;
                        sh_q[j].n = cnt[i];
                        sh_q[j].c = sh_q[j].k - (rem - above);
                    }
                    break;
                }
                above += cnt[i];
            }
        }
    }
    __syncthreads();
    if (PASS == 2) {
        // slots of pass 3: live queries with the same prefix share one (prefixes descend with j)
        __shared__ uint32_t sh_first[kMaxQueries];  // first query of a boundary bin
        if (warp == 0) {
            const bool live = lane < nq && sh_q[lane].trivial == 0u;
            const uint32_t slot = shared_slot(live, live ? sh_q[lane].prefix : 0u, nullptr);
            if (live) sh_q[lane].slot = slot;
            shared_slot(live, live ? sh_q[lane].slot2 : 0u, sh_first);
        }
        __syncthreads();
        if (threadIdx.x < nq) queries[m * kMaxQueries + threadIdx.x] = sh_q[threadIdx.x];
        // code of every sub-bin: slot of pass 3 if a threshold lies in it, else 64 + energy cell
        int first = 0, last = nq;  // the live queries are contiguous: k == 0 come before them, k >= d after them
        while (first < nq && sh_q[first].trivial) ++first;
        while (last > first && sh_q[last - 1].trivial) --last;
        if (last > first) {
            const int nslot = (int)sh_q[last - 1].slot2 + 1;
            uint8_t* mp = map2 + (int64_t)m * kMaxQueries * kBins23;
            for (int i = threadIdx.x; i < nslot * kBins23; i += kDigitThreads) {
                const uint32_t s = (uint32_t)i / kBins23, x = (uint32_t)i % kBins23;
                int j = (int)sh_first[s];
                while (j < last && sh_q[j].slot2 == s && sh_digit_of[j] > x) ++j;
                const bool here = j < last && sh_q[j].slot2 == s && sh_digit_of[j] == x;
                mp[i] = here ? (uint8_t)sh_q[j].slot : (SUMS ? (uint8_t)(64u + (uint32_t)j + s) : (uint8_t)0xFFu);
            }
        }
        return;
    }
    if (SUMS) {
        // energy of every open interval (T_l, T_{l-1}), one warp each, in a fixed order: the threshold-free bins
        // (sweep 2), the keys next to a threshold that share its upper 23 bits (their counts), the cells
        for (int l = warp; l < pl.L; l += kDigitThreads / 32) {
            double e = 0.0;
            const int partials = in_parts ? parts.n_sum + (int)gridDim.x : n_sum;
            for (int c = lane; c < partials; c += 32) e += __ldcg(&sum_partial[((int64_t)m * sum_ctas + c) * kMaxLevels + l]);
            const Query* up = (l > 0 && !sh_q[l - 1].trivial) ? &sh_q[l - 1] : nullptr;
            const Query* dn = (l < nq && !sh_q[l].trivial) ? &sh_q[l] : nullptr;
            const uint32_t T_up = l > 0 ? sh_q[l - 1].T : kKeyNone, T_dn = l < nq ? sh_q[l].T : 0u;
            auto add_digits = [&](const Query* q) {
                const uint32_t* h = out + q->slot * kBins23;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t key = (q->T & ~0xFFu) | (uint32_t)(i * 32 + lane);
                    const uint32_t c = __ldcg(&h[i * 32 + lane]);
                    if (c && key < T_up && (key > T_dn || !dn)) {
                        const double x = (double)__uint_as_float(key);
                        e = fma((double)c, x * x, e);
                    }
                }
            };
            if (up) add_digits(up);
            if (dn && !(up && up->slot == dn->slot)) add_digits(dn);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
            if (lane == 0) {
                const unsigned long long* S = cand_S + (int64_t)m * kEnergyCells * 2;
                auto add_cell = [&](const Query* q) {
                    const int c = l + (int)q->slot2;
                    const unsigned __int128 tot = ((unsigned __int128)__ldcg(&S[c * 2 + 1]) << 32) + __ldcg(&S[c * 2]);
                    if (tot != 0) {
                        const double td = (double)(unsigned long long)(tot >> 64) * 0x1.0p64 + (double)(unsigned long long)tot;
                        const int ex = (int)(q->T >> 23);
                        e += ldexp(td, 2 * ((ex ? ex : 1) - 150));
                    }
                };
                if (up) add_cell(up);
                if (dn && !(up && up->slot2 == dn->slot2)) add_cell(dn);
                sh_E[l] = e;
            }
        }
        __syncthreads();
    }
    finish_selection(pl, m, 0, sh_q, sh_E, p_all, delta_all, emit[m].level, p_all[m * kMaxLevels], &emit[m], status, worker_err);
}

__global__ void copy_probs_kernel(const double* p_all, const double* delta_all, ProbList p_fixed, int fixed, int M, int L,
                                  double* p_out, double* delta_out, const int* worker_err) {
    pdl_enter();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M * L) return;
    const int m = i / L, l = i % L;
    const bool bad = worker_err[m] != 0;
    if (p_out) p_out[i] = fixed ? p_fixed.p[l] : (bad ? 0.0 : p_all[m * kMaxLevels + l]);
    if (delta_out) delta_out[i] = bad ? 0.0 : delta_all[m * kMaxLevels + l];
}

// Headers of the messages whose band and thresholds are already known (two queries per worker).
__global__ void band_header_kernel(FinishPlan pl, const Query* queries, const double* p_all, EmitParams* emit, int* status,
                                   int* worker_err, int M) {
    pdl_enter();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= M) return;
    if (worker_err[m]) {
        fail_worker(pl, m, &emit[m]);
        return;
    }
    const Query* q = queries + m * kMaxQueries;
    fill_emit(pl, m, emit[m].level, p_all[m * kMaxLevels], &q[0], &q[1], q[0].k, q[1].k, &emit[m], status, worker_err);
}

int blocks_per_worker(const Workspace& ws, int64_t d, int vec, int threads, int M, int waves) {
    const int64_t nvec = (d + vec - 1) / vec;
    const int64_t by_work = (nvec + (int64_t)threads * 4 - 1) / ((int64_t)threads * 4);
    int64_t by_sm = ((int64_t)ws.sm_count * waves) / M;  // rounded down: one block too many per worker costs a whole extra wave
    if (by_sm < 1) by_sm = 1;
    int64_t nb = by_work < by_sm ? by_work : by_sm;
    return (int)(nb < 1 ? 1 : nb);
}

size_t s2_smem(int L, bool sums, int threads) {
    return (size_t)(kS2Groups + kS2Slots * threads) * 4 + (sums ? (size_t)(L + 1) * threads * sizeof(double) : 0);
}

size_t digit_smem(int nq, bool cells) {
    return ((size_t)nq * kBins23 + (cells ? kCellWords : 0)) * sizeof(uint32_t);
}

}  // namespace

// Columns and table of pass 2 over the parts of a sampled selection.
size_t part_smem(int L) { return (size_t)(L + 1) * kDigitThreads * sizeof(double) + kBins1; }

// What a selection with nq queries per worker accumulates into.
ZeroList selection_state(Workspace& ws, int dtype, int64_t d, int M, int nq, bool sums) {
    ZeroList z = {};
    auto add = [&](void* p, size_t bytes) {
        z.ptr[z.n] = static_cast<uint32_t*>(p);
        z.words[z.n] = (uint32_t)(bytes / 4);
        ++z.n;  // at most ZeroList::kMost
    };
    add(ws.worker_err, sizeof(int) * M);
    add(ws.hist1, (size_t)M * kBins1 * sizeof(uint32_t));
    add(ws.level_desc, (size_t)M * emit_counts(emit_tiles_per_worker(d, dtype)).total() * sizeof(uint4));
    add(ws.list_n, sizeof(uint32_t));
    if (dtype == MLMC_F32) {
        add(ws.cand_count, sizeof(uint32_t) * M);
        add(ws.cand_overflow, sizeof(int) * M);
        ws.hist3 = ws.hist2 + (size_t)M * kMaxQueries * kBins23;  // right behind, so that one range is cleared
        if (nq > 0) {
            add(ws.hist2, (size_t)M * kMaxQueries * kBins23 * 2 * sizeof(uint32_t));
            if (sums) add(ws.cand_S, (size_t)M * kEnergyCells * 2 * sizeof(unsigned long long));
        }
    }
    return z;
}

// ---------------------------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------------------------
void launch_begin_adaptive(Workspace& ws, int dtype, int64_t d, int M, const int64_t* k, int L, cudaStream_t s) {
    RankList r = {};
    r.nq = L - 1;
    for (int j = 0; j < r.nq; ++j) r.k[j] = (uint32_t)k[j];
    launch_kernel(ws, K_BEGIN, begin_adaptive_kernel, dim3(ws.sm_count), 512, 0, s,
                  selection_state(ws, dtype, d, M, r.nq, true), r, ws.queries, d, M);
}

void launch_begin_drawn(Workspace& ws, int dtype, int64_t d, int M, const DrawnBand* bands, int L, bool brackets,
                        cudaStream_t s) {
    const ZeroList z = selection_state(ws, dtype, d, M, 2, false);
    uint4* br = brackets ? ws.bracket : nullptr;
    auto go = [&](auto list, auto kernel) {
        for (int m = 0; m < M; ++m) list.band[m] = bands[m];
        launch_kernel(ws, K_BEGIN, kernel, dim3(ws.sm_count), 512, 0, s, z, list, ws.queries, ws.emit, ws.p_all, d, M, L,
                      ws.prev_bin, br);
    };
    if (M <= 32) go(DrawnList<32>(), begin_drawn_kernel<32>);
    else go(DrawnList<kEmitMaxWorkers>(), begin_drawn_kernel<kEmitMaxWorkers>);
}

void launch_uniforms(Workspace& ws, int M, uint64_t seed, uint64_t step, cudaStream_t s) {
    launch_kernel(ws, K_UNIFORMS, uniforms_kernel, dim3((M + 127) / 128), 128, 0, s, ws.u_dev, M, seed, step);
}

void launch_hist1(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, bool brackets, const int* only, cudaStream_t s) {
    const int tpw = emit_tiles_per_worker(d, dtype);
    size_t smem = kBins1 * sizeof(uint32_t);
    // One wave of blocks (every block clears and flushes a whole histogram: two waves cost 2 % at 16 x 11.7M keys), unless
    // whole blocks per worker leave more than 5 % of the SMs idle (32 workers: 456 against 401 us for 26M bf16 keys each).
    const int waves = ws.sm_count / M * M * 20 < ws.sm_count * 19 ? 2 : 1;
    const int nb = blocks_per_worker(ws, d, dtype == MLMC_BF16 ? 8 : 4, kHistThreads, M, waves);
    auto go = [&](auto kernel) {
        const float* row = static_cast<const float*>(g);
        launch_kernel(ws, only ? K_MISSED_HIST : K_HIST1, kernel, dim3(nb, M), kHistThreads, smem, s, row, d, ld, ws.hist1, ws.tile_max, tpw,
                      ws.status, ws.worker_err, ws.bracket, ws.cand_keys, ws.cand_cap, ws.cand_count, ws.cand_overflow, only);
    };
    if (dtype == MLMC_BF16) {
        const int64_t batches = ((int64_t)tpw * kEmitGroups + nb * (kHistThreads / 32) - 1) / (nb * (kHistThreads / 32));  // per warp
        const bool sample = batches >= kColumnBatches;
        launch_kernel(ws, K_HIST1, sample ? hist1_bf16_kernel<true> : hist1_bf16_kernel<false>, dim3(nb, M), kHistThreads,
                      BinCounts::words(sample) * sizeof(uint32_t), s, static_cast<const bf16_t*>(g), d, ld, ws.hist1, ws.tile_max, tpw, ws.status,
                      ws.worker_err);
    } else if (brackets) {
        smem += (kHistThreads / 32) * (kWarpStage + 1) * sizeof(uint32_t);
        go(hist1_kernel<true>);
    } else {
        go(hist1_kernel<false>);
    }
}

void launch_resolve1(Workspace& ws, int dtype, int M, const FinishPlan& plan, bool brackets, bool sampled, int* miss, cudaStream_t s) {
    launch_kernel(ws, K_RESOLVE1, resolve1_kernel, dim3(M), kResolveThreads, kBinRowsSmem, s, ws.hist1, ws.queries, ws.table1,
                  ws.cand_floor, plan, dtype == MLMC_BF16 ? 1 : 0, ws.status, ws.worker_err, ws.emit,
                  brackets ? ws.bracket : nullptr, ws.bracket_hit, ws.prev_bin, ws.bracket_stats, ws.cand_count,
                  ws.cand_overflow, ws.p_all, ws.delta_all, sampled ? 1 : 0, miss);
}

// Sweep 2: energies of the threshold-free bins (adaptive only) and the candidate keys of the boundary bins.
void launch_sums_candidates(Workspace& ws, const void* g, int64_t d, int M, int64_t ld, const FinishPlan& plan, bool brackets,
                            const int* only, cudaStream_t s) {
    const bool sums = plan.adaptive != 0;
    const int threads = sums && s2_smem(plan.L, sums, kS2Threads) > (size_t)kS2SmemMost ? kS2Threads / 2 : kS2Threads;
    const int nb = std::min(blocks_per_worker(ws, d, 4, threads, M, 1), ws.sum_ctas);
    ws.cur_sum_ctas = nb;
    launch_kernel(ws, only ? K_MISSED_SUMS : K_SUMS_CAND, sums ? sums_candidates_kernel<true> : sums_candidates_kernel<false>, dim3(nb, M), threads,
                  s2_smem(plan.L, sums, threads), s, static_cast<const float*>(g), d, ld, ws.table1, ws.queries,
                  plan.nq, plan.L, ws.sum_partial, ws.sum_ctas, ws.cand_keys, ws.cand_cap, ws.cand_count, ws.cand_overflow, ws.worker_err, ws.tile_max,
                  emit_tiles_per_worker(d, MLMC_F32), ws.cand_floor, brackets ? ws.bracket_hit : nullptr, only);
}

// The second and third digit, and the end of the selection.
void launch_digit_passes(Workspace& ws, const void* g, int64_t d, int M, int64_t ld, const FinishPlan& plan, bool sampled, cudaStream_t s) {
    const bool sums = plan.adaptive != 0;
    const CandParts parts = {sampled ? ws.miss : nullptr, ws.part_n, ws.parts, ws.part_cap, ws.sweep_blocks};
    int nb = (ws.sm_count * kDigitBlocks) / M;
    const int64_t by_work = (d + kDigitThreads * 4 - 1) / (kDigitThreads * 4);
    if (nb > by_work) nb = (int)by_work;
    if (nb < 1) nb = 1;
    auto go = [&](int id, auto kernel, uint32_t* hist, bool cells) {
        launch_kernel(ws, id, kernel, dim3(nb, M), kDigitThreads,
                      digit_smem(plan.nq, cells) + (sampled && id == K_CAND2 ? part_smem(plan.L) : 0), s,
                      static_cast<const float*>(g), d,
                      ld, ws.cand_keys, ws.cand_cap, ws.cand_count, ws.cand_overflow, ws.table1, ws.map2, hist, ws.done,
                      ws.queries, plan, ws.cand_S, ws.sum_partial, ws.sum_ctas, ws.cur_sum_ctas, ws.status, ws.worker_err,
                      ws.emit, ws.p_all, ws.delta_all, parts);
    };
    if (plan.nq > 0 || sampled) {
        if (sums) go(K_CAND2, digit_pass_kernel<2, true>, ws.hist2, false);
        else go(K_CAND2, digit_pass_kernel<2, false>, ws.hist2, false);
    }
    if (sums) go(K_CAND3, digit_pass_kernel<3, true>, ws.hist3, true);
    else go(K_CAND3, digit_pass_kernel<3, false>, ws.hist3, false);
}

void launch_band_header(Workspace& ws, int M, const FinishPlan& plan, cudaStream_t s) {
    launch_kernel(ws, K_BAND_HEADER, band_header_kernel, dim3((M + 127) / 128), 128, 0, s, plan, ws.queries, ws.p_all, ws.emit,
                  ws.status, ws.worker_err, M);
}

void launch_copy_probs(Workspace& ws, int M, int L, const double* p_fixed, double* p_out, double* delta_out,
                       cudaStream_t s) {
    launch_kernel(ws, K_COPY_PROBS, copy_probs_kernel, dim3((M * L + 127) / 128), 128, 0, s, ws.p_all, ws.delta_all,
                  prob_list(p_fixed, L), p_fixed ? 1 : 0, M, L, p_out, delta_out, ws.worker_err);
}

int configure_select_kernels() {
    const int hist = (int)(kBins1 * sizeof(uint32_t));
    const int stage = (int)((kHistThreads / 32) * (kWarpStage + 1) * sizeof(uint32_t));
    const int digits = (int)digit_smem(kMaxQueries, true);
    const int columns = (int)(digit_smem(kMaxQueries, false) + part_smem(kMaxLevels));
    auto set = [](auto kernel, int bytes) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
    };
    const bool ok = set(resolve1_kernel, (int)kBinRowsSmem) && set(hist1_kernel<false>, hist) && set(hist1_kernel<true>, hist + stage) &&
                    set(hist1_bf16_kernel<true>, (int)(BinCounts::words(true) * sizeof(uint32_t))) &&
                    set(hist1_bf16_kernel<false>, (int)(BinCounts::words(false) * sizeof(uint32_t))) && set(sums_candidates_kernel<true>, kS2SmemMost) &&
                    set(sums_candidates_kernel<false>, (int)s2_smem(0, false, kS2Threads)) && set(digit_pass_kernel<2, true>, columns) &&
                    set(digit_pass_kernel<2, false>, digits) && set(digit_pass_kernel<3, true>, digits) &&
                    set(digit_pass_kernel<3, false>, digits);
    return ok ? MLMC_OK : MLMC_ERR_CUDA;
}

}  // namespace mlmc
