// The whole Top-k message of short rows in one launch: a thread-block cluster per worker holds the row in the shared
// memory of its blocks and does the selection, the probabilities, the draw and the ordered emission there, exchanging
// histograms and counts through distributed shared memory.
//
// On short rows the kernels of topk_select.cu and topk_emit.cu are chains of launches whose bodies are a few dependent
// memory round trips each (4 workers of 65,536 entries: 60 us for 10 launches); here the row is read from memory once and
// the steps are separated by cluster barriers (0.4 to 0.6 us each, with what was written before them).  Bound by the latency of
// the steps and, in rows of more than a few thousand keys per block, by the issue of the passes over the keys.  The cluster size is
// a constant of the kernel: loops over the blocks have all their reads in flight, and nothing is divided at run time (4 x 65,536
// entries, given p, on 4 blocks: 22.4 us per step with a run-time size, 20.0 so).  The steps:
//   1. the row is copied to shared memory (16-byte asynchronous copies); histogram of the leading 13 key bits, largest
//      key per batch, NaN / Inf check;
//   2. radix select of every query: 13 + 9 + 9 key bits (fp32) or 13 + 2 (bf16).  The blocks tell one another their counts of
//      128 ranges of bins; every block then finds the first digit of every query for itself, a warp per query that reads the
//      bins of one range.  Later digits are counted per boundary bin;
//   3. adaptive p: energy of the open intervals between the thresholds, mant^2 in 16-bit limbs per (interval, exponent)
//      cell: exact, whatever the order; then p and the draw, by every block for itself (same data, same result);
//   4. the band: counts per batch, exchanged between the blocks, then every batch is written at its final position.
#include <cooperative_groups.h>

#include <type_traits>

#include "topk_band.cuh"
#include "topk_finish.cuh"

namespace mlmc {

namespace {

namespace cg = cooperative_groups;

constexpr int kClThreads = 1024;
constexpr int kClMost = 16;                      // blocks per cluster (8 is the portable limit)
constexpr int kClDigit1 = 13;
constexpr int kClBins = 1 << kClDigit1;
constexpr int kClRange = 64;                     // bins that are first counted together
constexpr int kClRanges = kClBins / kClRange;
constexpr int kClHistWords = 8192;               // 16384 16-bit counts, or the energy cells
constexpr int kClBatches = 91;                   // batches per block at most: as much of the row (182 KB) as shared memory holds
constexpr int kClBatchesBf16 = 63;               // given p, bf16: a block's keys fit 16-bit counts
constexpr int kClSpread = 16;                    // batches per block from which on the cluster grows while all clusters run at a time,
constexpr int kClEasy = 32;                      // and where they do not
constexpr int kClFew = 64;                       // given p, fp32: from which on 16 blocks take the place of 8, if they run at a time
constexpr int kClTwoWaves = 56;                  // adaptive p, fp32: batches per block with which two waves of clusters are worth it
constexpr int kClCells = 32 + 256;               // interval + (largest exponent - exponent)
constexpr int kClCopiesLow = 8;                  // copies of a cell's limbs: 32 where the cells are few enough, else 8
static_assert(kClCells * 3 * kClCopiesLow <= kClHistWords, "the cells take the place of the histogram");
static_assert(kClBatches * kBatchWords < 65536 && kClBatchesBf16 * kBatchWords * 2 < 65536, "16-bit counts, and 16-bit limbs added at most 65535 times");

struct ClusterShared {
    Query q[kMaxQueries];
    uint32_t first[kMaxQueries], slots;          // first query of a boundary bin (slot), number of slots
    int bin[kMaxQueries];                        // leading-digit bin of a query; kClBins above, -1 below every bin
    uint32_t low_bin;                            // first bin of the row's lowest range with a key
    double E[kMaxLevels];
    EmitParams emit;
    uint32_t top[kClMost];                       // per block: its largest key
    __align__(16) uint16_t ranges[kClRanges];    // the block's keys in the ranges of leading-digit bins
    uint4 counts[kClMost];                       // per block: {C, A, B, batches}
    uint32_t warp[32];
    uint32_t batch_max[kClBatches];
    uint16_t batch_c[kClBatches], batch_a[kClBatches], batch_b[kClBatches];
};

constexpr size_t kClFixedSmem = kClHistWords * 4 + kClBins;  // histogram, bin codes; then the row
constexpr size_t kClSharedMost = 227 * 1024;
static_assert(kClFixedSmem + kClBatches * kBatchWords * 4 + sizeof(ClusterShared) + 64 <= kClSharedMost &&
              kClFixedSmem + (kClBatches + 1) * kBatchWords * 4 + sizeof(ClusterShared) > kClSharedMost, "the most that fits");

template <typename T, int CL, bool ADAPTIVE>  // CL: blocks per cluster
__global__ void __launch_bounds__(kClThreads, 1)
cluster_topk_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const __grid_constant__ FinishPlan pl,
                    const __grid_constant__ DrawnList<32> drawn, int batches, int per_block, double* p_all, double* delta_all,
                    uint32_t* __restrict__ idx_out, float* __restrict__ val_out, uint32_t* group_n, int* status,
                    int* worker_err) {
    using Tr = ElemTraits<T>;
    using EW = EmitWord<T>;
    constexpr int kKeyBits = Tr::kVec == 4 ? 31 : 15;
    constexpr int kShift1 = kKeyBits - kClDigit1;            // 18 / 2
    constexpr int kShift2 = Tr::kVec == 4 ? 9 : 0;           // of the second digit
    constexpr int kBits2 = kShift1 - kShift2;                // 9 / 2
    extern __shared__ __align__(16) uint8_t sh_raw[];
    uint32_t* sh_hist = reinterpret_cast<uint32_t*>(sh_raw);
    uint8_t* sh_tab = sh_raw + kClHistWords * 4;
    uint32_t* sh_row = reinterpret_cast<uint32_t*>(sh_raw + kClFixedSmem);
    __shared__ ClusterShared sh;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), m = blockIdx.x / CL;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nq = pl.nq;
    for (int i = t; i < kClHistWords; i += kClThreads) sh_hist[i] = 0u;
    if (t < nq) sh.q[t] = make_query(ADAPTIVE ? pl.k[t] : (t ? drawn.band[m].k_hi : drawn.band[m].k_lo), d);
    cluster.barrier_arrive();
    pdl_enter();

    // ---- 1. the block's batches (512 words each) into shared memory, chunks in the swizzled order of the emission; a warp
    // counts a batch as soon as its own copy of it has landed
    const int b0 = rank * per_block, nb = max(0, min(per_block, batches - b0));
    const T* row = g + (int64_t)m * ld;
    constexpr int kTrips = (kClBatches + 31) / 32;
#pragma unroll
    for (int i = 0; i < kTrips; ++i) {
        const int b = warp + i * 32;
        if (b < nb) copy_batch_async<T>(row, d, (b0 + b) / kEmitGroups, (b0 + b) % kEmitGroups, lane, sh_row + b * kBatchWords);
        cp_async_commit();
    }
    __syncthreads();  // the counts are zero
    uint32_t my_top = 0;
#pragma unroll
    for (int i = 0; i < kTrips; ++i) {
        const int b = warp + i * 32;
        if (i == 0) cp_async_wait<kTrips - 1>();
        else if (i + 1 < kTrips) cp_async_wait<1>();
        else cp_async_wait<0>();
        __syncwarp();
        if (b >= nb) continue;
        const uint32_t* w = sh_row + b * kBatchWords;
        const int64_t e0 = (int64_t)(b0 + b) * kBatchWords * EW::S;
        const bool whole = e0 + kBatchWords * EW::S <= d;  // warp-uniform
        uint32_t mx = 0;
#pragma unroll
        for (int c = 0; c < kBatchWords / 128; ++c) {
            const int chunk = c * 32 + lane;
            const uint4 q = *reinterpret_cast<const uint4*>(w + chunk * 4);
            const uint32_t x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
#pragma unroll
                for (int s = 0; s < EW::S; ++s) {
                    const uint32_t key = EW::key(x[k], s);
                    if (whole || e0 + (int64_t)(swz(chunk) * 4 + k) * EW::S + s < d) {  // the swizzle is its own inverse
                        const uint32_t bin = key >> kShift1;
                        atomicAdd(&sh_hist[bin >> 1], 1u << ((bin & 1u) * 16u));
                        mx = max(mx, key);
                    }
                }
            }
        }
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        if (lane == 0) sh.batch_max[b] = mx;
        my_top = max(my_top, mx);
    }
    static_assert(kTrips == 3, "the waits above");
    __syncwarp();
    if (lane == 0) sh.warp[warp] = my_top;
    __syncthreads();
    my_top = __reduce_max_sync(0xFFFFFFFFu, sh.warp[lane]);
    {  // the block's keys in every range of kClRange bins
        constexpr int kPer = kClRanges / 32;
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int range = warp * kPer + i;
            const uint32_t x = sh_hist[range * (kClRange / 2) + lane];
            const uint32_t n = __reduce_add_sync(0xFFFFFFFFu, (x & 0xFFFFu) + (x >> 16));
            if (lane == 0) sh.ranges[range] = (uint16_t)n;
        }
    }
    __syncthreads();
    cluster.barrier_wait();  // every block of the cluster runs: its shared memory can be written
    constexpr int kRangeVecs = kClRanges * 2 / 16;
    uint4* sh_part = reinterpret_cast<uint4*>(sh_hist + kClBins / 2);  // [block][kRangeVecs]: the half of the words that the counts do not use
    static_assert(kClHistWords - kClBins / 2 >= kClMost * kRangeVecs * 4, "the ranges of all blocks fit behind the counts");
    if (t < CL * kRangeVecs)
        cluster.map_shared_rank(sh_part, t / kRangeVecs)[rank * kRangeVecs + t % kRangeVecs] =
            reinterpret_cast<const uint4*>(sh.ranges)[t % kRangeVecs];
    if (t < CL) cluster.map_shared_rank(sh.top, t)[rank] = my_top;
    cluster.sync();
    uint32_t top = 0;
#pragma unroll
    for (int r = 0; r < CL; ++r) top = max(top, sh.top[r]);
    const bool bad = top >= Tr::kInfKey;
    if (rank == 0 && t == 0) {
        worker_err[m] = bad ? MLMC_ERR_NONFINITE : 0;
        if (bad) {
            set_status(status, MLMC_ERR_NONFINITE);
            fail_worker(pl, m, &sh.emit);
            group_n[m] = 0u;
        }
    }
    if (bad) return;  // the same in every block; nothing of another block's memory is touched after the barrier above

    if (ADAPTIVE && warp == kClThreads / 32 - 1) {  // without a query
        uint32_t low = kClRanges;
#pragma unroll
        for (int r = 0; r < CL; ++r) {
            const uint2 x = reinterpret_cast<const uint2*>(sh_part + r * kRangeVecs)[lane];
            if (x.x | x.y) low = min(low, 4u * lane + (x.x & 0xFFFFu ? 0u : x.x ? 1u : x.y & 0xFFFFu ? 2u : 3u));
        }
        low = __reduce_min_sync(0xFFFFFFFFu, low);
        if (lane == 0) sh.low_bin = low * kClRange;
    }
    static_assert(kMaxQueries <= kClThreads / 32 && kMaxLevels - 1 < kClThreads / 32, "a warp per query, and one more");
    // ---- 2. first digit: a warp per query, in every block alike.  The range that holds the rank, then its bins, of which the
    // counts come from all blocks at a time.  (With the bins divided among the blocks, a scan of them by all threads, and a
    // barrier for the answers, the step took 2.9 us in 4 blocks and 4.5 in 16, now 0.8 and 2.7.)
    if (warp < nq && sh.q[warp].trivial == 0u) {
        const uint32_t k = sh.q[warp].k;
        uint32_t c[4] = {};  // of ranges kClRanges - 1 - 4 lane, and down
#pragma unroll
        for (int r = 0; r < CL; ++r) {
            const uint2 x = reinterpret_cast<const uint2*>(sh_part + r * kRangeVecs)[31 - lane];
            c[0] += x.y >> 16; c[1] += x.y & 0xFFFFu; c[2] += x.x >> 16; c[3] += x.x & 0xFFFFu;
        }
        static_assert(kClRanges == 128 && kClRange == 64, "four ranges per lane, two bins per lane");
        uint32_t upto = c[0] + c[1] + c[2] + c[3], sum = upto;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if (lane >= o) upto += y;
        }
        int from = __ffs(__ballot_sync(0xFFFFFFFFu, upto >= k)) - 1;  // the first lane that reaches the rank
        uint32_t run = upto - sum, above = 0, range = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // the last range that is entered holds the rank
            if (run < k) {
                above = run;
                range = (uint32_t)(kClRanges - 1 - 4 * lane - i);
            }
            run += c[i];
        }
        above = __shfl_sync(0xFFFFFFFFu, above, from);
        range = __shfl_sync(0xFFFFFFFFu, range, from);
        const int word = (int)range * (kClRange / 2) + 31 - lane;
        uint32_t x[CL], hi = 0, lo = 0;
#pragma unroll
        for (int r = 0; r < CL; ++r) x[r] = cluster.map_shared_rank(sh_hist, r)[word];
#pragma unroll
        for (int r = 0; r < CL; ++r) {
            hi += x[r] >> 16;
            lo += x[r] & 0xFFFFu;
        }
        upto = sum = hi + lo;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if (lane >= o) upto += y;
        }
        upto += above;
        from = __ffs(__ballot_sync(0xFFFFFFFFu, upto >= k)) - 1;
        if (lane == from) {
            run = upto - sum;
            const bool second = run + hi < k;
            sh.q[warp].prefix = (uint32_t)(2 * word + (second ? 0 : 1)) << kShift1;
            sh.q[warp].rem = k - run - (second ? hi : 0u);
        }
    }
    __syncwarp();
    cluster.barrier_arrive();  // the block has read the others' counts; waited for before its own are cleared
    __syncthreads();
    // The live queries are contiguous (k = 0 before them, k >= d after them) and their prefixes descend: queries with the
    // same prefix share a histogram slot, numbered by the first of them.  By warp 0, a query per lane.
    auto number_slots = [&](bool first_digit) {
        const bool live = lane < nq && sh.q[lane].trivial == 0u;
        const uint32_t prefix = live ? sh.q[lane].prefix : kKeyNone, prev = __shfl_up_sync(0xFFFFFFFFu, prefix, 1);
        const bool is_first = live && (lane == 0 || prefix != prev);
        const uint32_t firsts = __ballot_sync(0xFFFFFFFFu, is_first);
        const uint32_t slot = (uint32_t)__popc(firsts & ((2u << lane) - 1u)) - 1u;
        if (live) sh.q[lane].slot = slot;
        if (first_digit) {
            if (live) sh.q[lane].slot2 = slot;
            if (is_first) sh.first[slot] = (uint32_t)lane;
            if (lane < nq) sh.bin[lane] = live ? (int)(prefix >> kShift1) : (sh.q[lane].trivial == 2u ? -1 : kClBins);
            if (lane == 0) sh.slots = (uint32_t)__popc(firsts);
        }
    };
    if (warp == 0) number_slots(true);
    __syncthreads();
    if constexpr (ADAPTIVE) {
        // codes of the bins: 64 + slot where a boundary lies in the bin, else the number of boundaries above it
        constexpr int per = kClBins / kClThreads;  // 8 consecutive bins per thread
        const int hi_bin = t * per + per - 1;
        int j = 0, n = nq;                         // the first query whose bin is not above the thread's
        while (n > 0) {
            const int half = n >> 1;
            if (sh.bin[j + half] > hi_bin) { j += half + 1; n -= half + 1; } else n = half;
        }
        uint32_t codes[2];
        if (j == nq || sh.bin[j] < t * per) {
            codes[0] = codes[1] = (uint32_t)j * 0x01010101u;
        } else {
            codes[0] = codes[1] = 0u;
#pragma unroll
            for (int i = per - 1; i >= 0; --i) {
                const int b = t * per + i;
                while (j < nq && sh.bin[j] > b) ++j;
                const uint32_t code = (j < nq && sh.bin[j] == b) ? 64u + sh.q[j].slot2 : (uint32_t)j;
                codes[i >> 2] |= code << (8 * (i & 3));
            }
        }
        reinterpret_cast<uint2*>(sh_tab)[t] = make_uint2(codes[0], codes[1]);
    }
    cluster.barrier_wait();
    // Two more digits (bf16: one) are counted per slot.  Few queries in small clusters: every block resolves all of them for
    // itself, and the third digit has counts of its own, so that nothing is exchanged but the counts.  Otherwise a block
    // resolves every CL-th query and tells the others, and the third digit takes the place of the second.
    const uint32_t hist_words = ((max(sh.slots << kBits2, (uint32_t)nq << kShift2) / 2 + 3u) & ~3u);
    const bool alike = nq * CL <= kClThreads / 32 && 4u * hist_words <= (uint32_t)kClHistWords;
    uint32_t* const sh_count2 = sh_hist;
    uint32_t* const sh_count3 = alike ? sh_hist + hist_words : sh_hist;
    const uint32_t list_from = alike ? 2u * hist_words : hist_words;
    for (uint32_t i = t; i < list_from; i += kClThreads) sh_hist[i] = 0u;
    __syncthreads();
    const int words4 = nb * kBatchWords / 4;
    // every key of the block's words (place: its element number in shared memory); the padding past the row's end has
    // keys above every finite one
    auto for_each_key = [&](auto&& f) {
        for (int i = t; i < words4; i += kClThreads) {
            const uint4 q = *reinterpret_cast<const uint4*>(sh_row + i * 4);
            const uint32_t x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int s = 0; s < EW::S; ++s) f(EW::key(x[c], s), (uint32_t)((i * 4 + c) * EW::S + s));
        }
    };
    // Slot of a boundary bin, 64 or more (64 less in `slot_of`) for the keys of other bins.  Given p: two bins.
    uint32_t bin_of[2], slot_of_bin[2];
    if constexpr (!ADAPTIVE)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const bool live = j < nq && sh.q[j].trivial == 0u;
            bin_of[j] = live ? sh.q[j].prefix >> kShift1 : 0xFFFFFFFFu;
            slot_of_bin[j] = live ? sh.q[j].slot2 : 0u;
        }
    auto slot_of = [&](uint32_t key, uint32_t& slot) -> bool {
        if constexpr (ADAPTIVE) {
            const uint32_t code = sh_tab[key >> kShift1];
            slot = code - 64u;
            return code >= 64u;
        } else {
            const uint32_t bin = key >> kShift1;
            slot = bin == bin_of[0] ? slot_of_bin[0] : slot_of_bin[1];
            return bin == bin_of[0] || bin == bin_of[1];
        }
    };
    // The places of the keys in boundary bins are listed by the first pass over them, behind the counts, every warp its own; a
    // warp whose list is too short looks at all its keys again.
    const uint32_t list_cap = 2u * (kClHistWords - list_from) / (kClThreads / 32);
    uint16_t* const list = reinterpret_cast<uint16_t*>(sh_hist + list_from) + warp * list_cap;
    uint32_t listed = 0;  // warp-uniform
    auto key_at = [&](uint32_t place) -> uint32_t { return EW::key(sh_row[place / EW::S], place % EW::S); };
    auto for_each_boundary_key = [&](auto&& f) {
        uint32_t slot;
        if (listed <= list_cap) {
            for (uint32_t i = lane; i < listed; i += 32) {
                const uint32_t key = key_at(list[i]);
                slot_of(key, slot);
                f(key, slot);
            }
        } else {
            for_each_key([&](uint32_t key, uint32_t) {
                if (slot_of(key, slot)) f(key, slot);
            });
        }
    };
    // One more digit of the queries, `bits` bits at `shift`.  2 CL warps take a query: a lane has eight of the 512 digits (a
    // 16-byte vector) in one block, the lanes of one vector add up over the blocks, and the warp whose digits hold the rank tells
    // this block or, where the blocks divide the queries, all of them.  (A warp per query that reads block after block: 6.7 and
    // 4.3 us for the two digits of 14 queries in 16 blocks.)  Digits of 2 bits: a warp per query, a block per lane.
    auto found = [&](int j, uint32_t prefix, uint32_t left, uint32_t n, bool last, bool tell_all) {  // by a whole warp
        const uint32_t k = sh.q[j].k;
        if (lane < (tell_all ? CL : 1)) {
            Query& q = tell_all ? cluster.map_shared_rank(sh.q, lane)[j] : sh.q[j];
            q.prefix = prefix;
            q.rem = left;
            if (last) {
                q.T = prefix;
                q.r = left;
                q.n = n;
                q.c = k - left;
            }
        }
    };
    auto descend = [&](auto bits_tag, int shift, bool last, uint32_t* counts) {
        constexpr int bits = decltype(bits_tag)::value;
        cluster.sync();  // every block's counts are complete
        if constexpr (bits == 2) {
            if (warp < nq && sh.q[warp].trivial == 0u) {
                uint2 x = make_uint2(0u, 0u);
                if (lane < CL) x = reinterpret_cast<const uint2*>(cluster.map_shared_rank(counts, lane))[sh.q[warp].slot];
                const uint32_t c[4] = {__reduce_add_sync(0xFFFFFFFFu, x.x & 0xFFFFu), __reduce_add_sync(0xFFFFFFFFu, x.x >> 16),
                                       __reduce_add_sync(0xFFFFFFFFu, x.y & 0xFFFFu), __reduce_add_sync(0xFFFFFFFFu, x.y >> 16)};
                uint32_t left = sh.q[warp].rem, digit = 3, n = c[3];
#pragma unroll
                for (int e = 3; e > 0; --e)
                    if (digit == (uint32_t)e && left > c[e]) {
                        left -= c[e];
                        n = c[e - 1];
                        digit = (uint32_t)e - 1u;
                    }
                __syncwarp();
                found(warp, sh.q[warp].prefix | (digit << shift), left, n, last, false);
            }
            __syncthreads();
        } else {
            static_assert(bits == 9, "64 vectors of eight counts");
            constexpr int warps_each = 2 * CL, at_a_time = (kClThreads / 32) / warps_each;
            const int part = warp % warps_each;
            constexpr int vecs = 32 / CL;  // per warp and block
            const int mine = alike ? nq : (nq - rank + CL - 1) / CL;
            for (int i0 = 0; i0 < mine; i0 += at_a_time) {
                const int i = i0 + warp / warps_each, j = alike ? i : rank + i * CL;
                const bool live = i < mine && sh.q[j].trivial == 0u;
                uint32_t c[8] = {}, rem = 0;  // digits 8 v + 7 .. 8 v
                const int v = 63 - (part * vecs + lane % vecs);
                if (live) {
                    const uint4 x = reinterpret_cast<const uint4*>(cluster.map_shared_rank(counts, lane / vecs))[sh.q[j].slot * 64u + v];
                    c[0] = x.w >> 16; c[1] = x.w & 0xFFFFu; c[2] = x.z >> 16; c[3] = x.z & 0xFFFFu;
                    c[4] = x.y >> 16; c[5] = x.y & 0xFFFFu; c[6] = x.x >> 16; c[7] = x.x & 0xFFFFu;
                    rem = sh.q[j].rem;
                }
#pragma unroll
                for (int o = vecs; o < 32; o <<= 1)
#pragma unroll
                    for (int e = 0; e < 8; ++e) c[e] += __shfl_xor_sync(0xFFFFFFFFu, c[e], o);
                uint32_t sum = 0;
#pragma unroll
                for (int e = 0; e < 8; ++e) sum += c[e];
                uint32_t upto = sum;  // over the vectors of the warp
#pragma unroll
                for (int o = 1; o < vecs; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o, vecs);
                    if (lane % vecs >= o) upto += y;
                }
                if (lane == vecs - 1) sh.warp[warp] = upto;
                __syncthreads();
                uint32_t run = upto - sum + __reduce_add_sync(0xFFFFFFFFu, lane < part ? sh.warp[warp - part + lane] : 0u);
                const bool here = live && run < rem && rem <= run + sum;
                const uint32_t from = __ballot_sync(0xFFFFFFFFu, here);  // a lane of every block, or none
                if (from) {
                    uint32_t digit = 0, left = 0, n = 0;
#pragma unroll
                    for (int e = 0; e < 8; ++e) {  // the last digit that is entered holds the rank
                        if (run < rem) {
                            digit = (uint32_t)(8 * v + 7 - e);
                            left = rem - run;
                            n = c[e];
                        }
                        run += c[e];
                    }
                    const int f = __ffs(from) - 1;
                    digit = __shfl_sync(0xFFFFFFFFu, digit, f);
                    left = __shfl_sync(0xFFFFFFFFu, left, f);
                    n = __shfl_sync(0xFFFFFFFFu, n, f);
                    const uint32_t prefix = sh.q[j].prefix | (digit << shift);
                    __syncwarp();
                    found(j, prefix, left, n, last, !alike);
                }
                __syncthreads();  // sh.warp has been read
            }
            if (!alike) cluster.sync();
        }
    };
    auto count = [&](uint32_t* counts, uint32_t i) { atomicAdd(&counts[i >> 1], 1u << ((i & 1u) * 16u)); };
    if (nq > 0) {
        for_each_key([&](uint32_t key, uint32_t place) {
            uint32_t slot;
            const bool hit = slot_of(key, slot);
            const uint32_t hits = __ballot_sync(0xFFFFFFFFu, hit);
            if (hits == 0u) return;
            if (hit) {
                count(sh_count2, (slot << kBits2) | ((key >> kShift2) & ((1u << kBits2) - 1u)));
                const uint32_t at = listed + (uint32_t)__popc(hits & ((1u << lane) - 1u));
                if (at < list_cap) list[at] = (uint16_t)place;
            }
            listed += (uint32_t)__popc(hits);
        });
        descend(std::integral_constant<int, kBits2>(), kShift2, kShift2 == 0, sh_count2);
        if constexpr (kShift2 > 0) {
            if (warp == 0) number_slots(false);
            if (!alike)
                for (uint32_t i = t; i < hist_words; i += kClThreads) sh_hist[i] = 0u;
            __syncthreads();
            for_each_boundary_key([&](uint32_t key, uint32_t s) {
                for (int j = (int)sh.first[s]; j < nq && sh.q[j].trivial == 0u && sh.q[j].slot2 == s; ++j) {
                    if ((sh.q[j].prefix >> kShift2) == (key >> kShift2)) {
                        count(sh_count3, (sh.q[j].slot << kShift2) | (key & ((1u << kShift2) - 1u)));
                        break;
                    }
                }
            });
            descend(std::integral_constant<int, (kShift2 > 0 ? kShift2 : 9)>(), 0, true, sh_count3);
        }
        cluster.barrier_arrive();  // the block has read the others' counts
    }

    // ---- 3. energies of the open intervals
    if constexpr (ADAPTIVE) {
        // A cell is (interval, exponent), numbered interval + (largest exponent - exponent): neither falls as the keys fall.
        auto exponent = [&](uint32_t key) -> int { return (int)((Tr::kVec == 4 ? key : key << 16) >> 23); };
        const int top_e = exponent(top);
        const int low_e = exponent(sh.low_bin << kShift1), span = nq + 1 + top_e - low_e;  // cells
        const bool many = span * 3 * 32 > kClHistWords;
        const int copies = many ? kClCopiesLow : 32, copy = lane & (copies - 1);
        // the keys of the boundary bins first, while their list is intact: their cells wait in a register each
        __syncthreads();
        const bool by_list = listed <= list_cap && listed <= 8u * 32u;  // warp by warp
        uint32_t held[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) held[i] = (by_list && (uint32_t)(lane + i * 32) < listed) ? list[lane + i * 32] : 0xFFFFFFFFu;
        __syncthreads();
        if (nq > 0) cluster.barrier_wait();
        for (int i = t; i < kClHistWords; i += kClThreads) sh_hist[i] = 0u;
        __syncthreads();
        auto add = [&](uint32_t interval, uint32_t key) {
            const uint32_t bits = Tr::kVec == 4 ? key : key << 16;
            const uint64_t m2 = mantissa_squared(bits);
            uint32_t* a = sh_hist + (interval + top_e - (bits >> 23)) * (3 * copies) + copy;
            atomicAdd(a, (uint32_t)m2 & 0xFFFFu);
            atomicAdd(a + copies, (uint32_t)(m2 >> 16) & 0xFFFFu);
            atomicAdd(a + 2 * copies, (uint32_t)(m2 >> 32));
        };
        auto add_boundary = [&](uint32_t key) {
            int j = (int)sh.first[sh_tab[key >> kShift1] - 64u];
            while (j < nq && sh.q[j].T > key) ++j;  // thresholds descend; a query with k >= d has T = 0
            if (j < nq && sh.q[j].T == key && sh.q[j].trivial == 0u) return;  // a threshold key: added from its count
            add((uint32_t)j, key);
        };
        for_each_key([&](uint32_t key, uint32_t) {
            const uint32_t code = sh_tab[key >> kShift1];
            if (key >= Tr::kInfKey || key == 0u) return;  // padding; zeros add nothing
            if (code < 64u) add(code, key);
            else if (!by_list) add_boundary(key);
        });
#pragma unroll
        for (int i = 0; i < 8; ++i)
            if (held[i] != 0xFFFFFFFFu) {
                const uint32_t key = key_at(held[i]);
                if (key != 0u) add_boundary(key);
            }
        __syncthreads();
        unsigned long long* sh_sum = reinterpret_cast<unsigned long long*>(sh_tab);  // [kClCells][2]: the codes are not needed any more
        static_assert(kClCells * 16 <= kClBins, "the sums take the place of the codes");
        if (t < kClCells) {
            unsigned long long lo = 0, hi = 0;
            if (many || t < span) {
                const uint32_t* a = sh_hist + t * (3 * copies);
                for (int r = 0; r < copies; ++r) {
                    const int c = (r + t) & (copies - 1);  // neighbours start in different banks
                    lo += (unsigned long long)a[c] + ((unsigned long long)a[copies + c] << 16);
                    hi += a[2 * copies + c];
                }
            }
            sh_sum[2 * t] = lo;
            sh_sum[2 * t + 1] = hi;
        }
        cluster.sync();
        double* sh_cell = reinterpret_cast<double*>(sh_hist);  // [kClCells]: sum of mant^2 over the row
        if (t < 2 * kClCells && (t & ~31) < 2 * span) {  // thread 2 c + h adds half h of cell c over the blocks
            unsigned long long x[CL], sum = 0;
#pragma unroll
            for (int r = 0; r < CL; ++r) x[r] = cluster.map_shared_rank(sh_sum, r)[t];
#pragma unroll
            for (int r = 0; r < CL; ++r) sum += x[r];
            const unsigned long long hi = __shfl_down_sync(0xFFFFFFFFu, sum, 1);
            const unsigned __int128 tot = ((unsigned __int128)hi << 32) + sum;
            if ((t & 1) == 0) sh_cell[t >> 1] = (double)(unsigned long long)(tot >> 64) * 0x1.0p64 + (double)(unsigned long long)tot;
        }
        static_assert(2 * kClCells % 32 == 0 && 2 * kClCells <= kClThreads, "whole warps");
        __syncthreads();
        // interval l, one warp each: the exponents between those of its two thresholds, in a fixed order
        for (int l = warp; l < pl.L; l += kClThreads / 32) {
            const uint32_t T_up = l ? sh.q[l - 1].T : kKeyNone, T_dn = l < nq ? sh.q[l].T : 0u;
            const int e_hi = T_up == kKeyNone ? top_e : exponent(T_up), e_lo = T_dn == kKeyNone ? 255 : exponent(T_dn);
            double e = 0.0;
            for (int x = e_hi - lane; x >= max(e_lo, low_e); x -= 32) {
                const double c = sh_cell[l + top_e - x];
                if (c != 0.0) e += ldexp(c, 2 * ((x ? x : 1) - 150));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
            if (lane == 0) sh.E[l] = e;
        }
        __syncthreads();
    }
    if (!ADAPTIVE && nq > 0) cluster.barrier_wait();
    {
        const int level = ADAPTIVE ? 0 : drawn.band[m].level;
        const double p_sel = ADAPTIVE ? 0.0 : drawn.band[m].p;
        finish_selection(pl, m, Tr::kVec == 8, sh.q, sh.E, p_all, delta_all, level, p_sel, &sh.emit, status, worker_err);
    }
    if (!pl.want_emit) {
        cluster.sync();  // no block leaves while another may still read its sums
        return;
    }
    __syncthreads();

    // ---- 4. the band
    const EmitParams ep = sh.emit;
    const bool on = ep.enabled && ep.expect > 0u;  // the same in every block
    const Band band = {min(ep.Tb, EW::kCap), min(ep.Ta, EW::kCap), ep.ra, ep.rb, (float)ep.inv_p};
    for (int b = warp; b < nb; b += 32) {
        uint32_t bC = 0, bA = 0, bB = 0;
        if (on && sh.batch_max[b] >= band.Tb) {
            uint32_t cur[kEmitRows];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const uint4 x = *reinterpret_cast<const uint4*>(sh_row + b * kBatchWords + (q * 32 + lane) * 4);
                cur[4 * q] = x.x; cur[4 * q + 1] = x.y; cur[4 * q + 2] = x.z; cur[4 * q + 3] = x.w;
            }
            uint32_t a1, b1;
            const uint32_t flags = batch_flags<T>(cur, band.Tb, band.Ta, &a1, &b1);
            const uint32_t ca = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)__popc(flags) | (a1 << 16));
            bB = __reduce_add_sync(0xFFFFFFFFu, b1);
            bC = ca & 0xFFFFu;
            bA = ca >> 16;
        }
        if (lane == 0) {
            sh.batch_c[b] = (uint16_t)bC;
            sh.batch_a[b] = (uint16_t)bA;
            sh.batch_b[b] = (uint16_t)bB;
        }
    }
    __syncthreads();
    if (warp == 0) {  // the block's totals, to every block
        uint32_t nC = 0, nA = 0, nB = 0, listed = 0;
        for (int b = lane; b < nb; b += 32) {
            nC += sh.batch_c[b];
            nA += sh.batch_a[b];
            nB += sh.batch_b[b];
            listed += (on && sh.batch_max[b] >= band.Tb) ? 1u : 0u;
        }
        nC = __reduce_add_sync(0xFFFFFFFFu, nC);
        nA = __reduce_add_sync(0xFFFFFFFFu, nA);
        nB = __reduce_add_sync(0xFFFFFFFFu, nB);
        listed = __reduce_add_sync(0xFFFFFFFFu, listed);
        if (lane < CL) cluster.map_shared_rank(sh.counts, lane)[rank] = make_uint4(nC, nA, nB, listed);
    }
    cluster.sync();  // also: nothing of another block's memory is read after this
    uint4 before = make_uint4(0u, 0u, 0u, 0u), all = before;
#pragma unroll
    for (int r = 0; r < CL; ++r) {
        const uint4 x = sh.counts[r];
        if (r < rank) { before.x += x.x; before.y += x.y; before.z += x.z; }
        all.x += x.x; all.y += x.y; all.z += x.z; all.w += x.w;
    }
    if (rank == 0 && t == 0) {
        group_n[m] = all.w;
        if (on && (all.w == 0u || band_prefix(all.x, all.y, all.z, ep.ra, ep.rb) != ep.expect)) set_status(status, MLMC_ERR_INTERNAL);
    }
    if (!on) return;
    uint32_t* idx_w = idx_out + (int64_t)m * pl.capacity;
    float* val_w = val_out + (int64_t)m * pl.capacity;
    // the offsets of a batch's entries take the place of the histogram (fp32: 1 KB per warp; those of bf16 do not fit)
    uint16_t* stage = EW::S == 1 ? reinterpret_cast<uint16_t*>(sh_hist + warp * (kClHistWords / 32)) : nullptr;
    static_assert(kBatchWords * 2 <= kClHistWords / 32 * 4, "a batch's offsets fit");
    for (int b = warp; b < nb; b += 32) {
        if (sh.batch_c[b] == 0) continue;
        uint32_t pc = 0, pa = 0, pb = 0;  // counts of the block's batches before this one
        for (int i = lane; i < b; i += 32) { pc += sh.batch_c[i]; pa += sh.batch_a[i]; pb += sh.batch_b[i]; }
        pc = __reduce_add_sync(0xFFFFFFFFu, pc);
        pa = __reduce_add_sync(0xFFFFFFFFu, pa);
        pb = __reduce_add_sync(0xFFFFFFFFu, pb);
        uint3 run = make_uint3(before.x + pc, before.y + pa, before.z + pb);
        __syncwarp();  // the stage has been read
        emit_batch<T>(sh_row + b * kBatchWords, stage, band, (sh.batch_a[b] | sh.batch_b[b]) != 0, (uint32_t)((b0 + b) * kBatchWords * EW::S), run,
                      idx_w, val_w, pl.capacity);
    }
}

size_t cluster_smem(int per_block) { return kClFixedSmem + (size_t)per_block * kBatchWords * 4; }

}  // namespace

// f(cluster size as a constant) for the size 2^i.
template <typename F>
static auto with_cluster(int i, F&& f) {
    switch (i) {
        case 0: return f(std::integral_constant<int, 1>());
        case 1: return f(std::integral_constant<int, 2>());
        case 2: return f(std::integral_constant<int, 4>());
        case 3: return f(std::integral_constant<int, 8>());
        default: return f(std::integral_constant<int, 16>());
    }
}

int configure_cluster_kernels() {
    auto set = [&](auto kernel) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cluster_smem(kClBatches)) != cudaSuccess) return false;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    };
    for (int i = 0; i < 5; ++i)
        if (!with_cluster(i, [&](auto cl) {
                return set(cluster_topk_kernel<float, cl(), true>) && set(cluster_topk_kernel<float, cl(), false>) &&
                       set(cluster_topk_kernel<bf16_t, cl(), true>) && set(cluster_topk_kernel<bf16_t, cl(), false>);
            }))
            return MLMC_ERR_CUDA;
    return MLMC_OK;
}

// Asked of one kernel for all: they have the same threads and shared memory, 64 registers at most (1024 threads take all of an SM's), and
// with the shared memory of the longest rows one block per SM.
void cluster_limits(KernelLimits* limits) {
    static_assert(kClThreads == 1024 && 2 * (kClFixedSmem + kClBatches * kBatchWords * 4) > kClSharedMost, "one block per SM");
    clusters_that_fit(cluster_topk_kernel<float, 16, true>, kClThreads, cluster_smem(kClBatches), limits->topk_fit);
}

// Blocks per cluster for this call, 0: the row is too long, or the workers are too many, for the cluster to be the faster way.
// kClSpread batches per block while the clusters of all workers run at a time, else kClEasy (4 x 65,536 entries: 18.9 us per step on 8
// blocks, 19.7 on 4, adaptive p 26.4 and 30.3; where M clusters of 16 would not fit, 131k x 8 adaptive takes 63 us on 16 and 36 on 8); longer
// rows are stretched over 16 blocks.  fp32 rows with given p have two digits of two queries to tell all of 16 blocks, which takes longer
// than it spares, and few clusters of 16 run at a time: 8 blocks up to kClFew batches in each, and as many as a block holds where the clusters of 16 would take turns
// (16 blocks / 8: 131k x 3 22.3 / 19.8, 262k x 3 24.4 / 22.8, 280k x 6 29.3 / 28.8, 310k x 2 26.2 / 26.7, 372k x 4 29.9 / 31.8; 131k x 8 40.7 / 22.7,
// 262k x 9 45 / 26.7, 372k x 12 57.9 / 37.7).  Clusters that do not fit the GPU at a time run one after the other, where the launch chain has
// the whole GPU: how far that pays depends on what the chain has to do.  us per step, cluster / chain, layered rows:
//   fp32, adaptive  700k x 3 53 / 76, 400k x 6 46 / 79; two waves 262k x 8 63 / 78, 400k x 12 82 / 90, 700k x 8 100 / 89; three
//                   262k x 16 95 / 90, 131k x 32 93 / 100
//   fp32, given p   700k x 3 34 / 56, 700k x 6 39 / 60; two waves 262k x 16 45 / 61, 262k x 28 54 / 78, 372k x 28 69 / 91, 500k x 8 52 / 60,
//                   700k x 12 67 / 69
//   bf16, adaptive  500k x 4 47 / 53, 700k x 4 61 / 55, 1M x 3 70 / 54; two waves 500k x 8 75 / 58
//   bf16, given p   500k x 4 23 / 33, 1M x 3 30 / 36; two waves 500k x 8 38 / 39, 1M x 8 53 / 45
int cluster_blocks(const Workspace& ws, int dtype, int64_t d, int M, bool given) {
    const int64_t batches = (int64_t)emit_tiles_per_worker(d, dtype) * kEmitGroups;
    if (M > 32) return 0;
    const int* fits = ws.limits.topk_fit;
    auto enough = [&](int i) {  // batches per block up to which 2^i blocks are not made 2^(i + 1)
        const bool at_a_time = M <= fits[i + 1];
        if (i == 3 && given && dtype == MLMC_F32) return at_a_time ? kClFew : kClBatches;
        return at_a_time ? kClSpread : kClEasy;
    };
    int i = 0;
    while (i < 4 && fits[i + 1] > 0 && batches > (int64_t)enough(i) << i) ++i;
    const int fit = fits[i];
    if (fit == 0) return 0;
    const int64_t per = (batches + (1 << i) - 1) >> i;
    const int waves = (M + fit - 1) / fit;
    int64_t most = 0;
    if (dtype == MLMC_BF16) {
        if (given) most = waves == 1 ? kClBatchesBf16 : waves == 2 ? kClEasy : 0;
        else most = waves == 1 ? kClEasy : 0;
    } else {
        if (given) most = waves <= 2 ? kClBatches : 0;
        else most = waves == 1 ? kClBatches : waves == 2 ? kClTwoWaves : 0;
    }
    return per <= most ? 1 << i : 0;
}

void launch_cluster_topk(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const FinishPlan& plan,
                         const DrawnBand* bands, const mlmc_topk_msgs* out, cudaStream_t s) {
    const int tiles = emit_tiles_per_worker(d, dtype);
    const int batches = tiles * kEmitGroups, cl = cluster_blocks(ws, dtype, d, M, bands != nullptr), per = (batches + cl - 1) / cl;
    if (out) ws.last_emit_tiles = tiles;
    DrawnList<32> drawn = {};
    if (bands)
        for (int m = 0; m < M; ++m) drawn.band[m] = bands[m];
    auto go = [&](auto kernel, auto* row) {
        launch_kernel_cluster(ws, K_CLUSTER_TOPK, cl, kernel, dim3(M * cl), kClThreads, cluster_smem(per), s, row, d, ld, plan, drawn,
                              batches, per, ws.p_all, ws.delta_all, out ? out->idx : nullptr, out ? out->val : nullptr, ws.group_n,
                              ws.status, ws.worker_err);
    };
    int log2 = 0;
    while (1 << log2 < cl) ++log2;
    with_cluster(log2, [&](auto size) {
        constexpr int CL = size();
        if (dtype == MLMC_BF16)
            go(bands ? cluster_topk_kernel<bf16_t, CL, false> : cluster_topk_kernel<bf16_t, CL, true>, static_cast<const bf16_t*>(g));
        else
            go(bands ? cluster_topk_kernel<float, CL, false> : cluster_topk_kernel<float, CL, true>, static_cast<const float*>(g));
    });
}

}  // namespace mlmc
