// The whole Top-k message of short rows in one launch: a thread-block cluster per worker holds the row in the shared
// memory of its blocks and does the selection, the probabilities, the draw and the ordered emission there, exchanging
// histograms and counts through distributed shared memory.
//
// On short rows the kernels of topk_select.cu and topk_emit.cu are chains of launches whose bodies are a few dependent
// memory round trips each (4 workers of 65,536 entries: 60 us for 10 launches); here the row is read from memory once and
// the steps are separated by cluster barriers (about a microsecond each).  The steps:
//   1. the row is copied to shared memory (16-byte asynchronous copies); histogram of the leading 13 key bits, largest
//      key per batch, NaN / Inf check;
//   2. radix select of every query: 13 + 9 + 9 key bits (fp32) or 13 + 2 (bf16).  The bins of the first digit are divided
//      among the blocks, later digits are counted per boundary bin and a block takes every CL-th query;
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
constexpr int kClHistWords = 8192;               // 16384 16-bit counts, or the energy cells
constexpr int kClBatches = 91;                   // batches per block at most: as much of the row (182 KB) as shared memory holds
constexpr int kClEasy = 32;                      // batches per block from which on the cluster grows (64 KB, 16 words per thread)
constexpr int kClCells = 32 + 256;               // interval + (largest exponent - exponent)
constexpr int kClCopiesLow = 8;                  // copies of a cell's limbs: 32 where the cells are few enough, else 8
static_assert(kClCells * 3 * kClCopiesLow <= kClHistWords, "the cells take the place of the histogram");
static_assert(kClBatches * kBatchWords < 65536 && kClEasy * kBatchWords * 2 < 65536, "16-bit counts, and 16-bit limbs added at most 65535 times");

struct ClusterShared {
    Query q[kMaxQueries];
    uint32_t first[kMaxQueries], slots;          // first query of a boundary bin (slot), number of slots
    int bin[kMaxQueries];                        // leading-digit bin of a query; kClBins above, -1 below every bin
    uint32_t listed, low_bin;                    // keys of the boundary bins; lowest bin with a key
    double E[kMaxLevels];
    EmitParams emit;
    uint32_t top[kClMost];                       // per block: its largest key
    uint16_t part[kClMost][kClMost];             // [block][range of bins]: the block's keys in the range
    uint4 counts[kClMost];                       // per block: {C, A, B, batches}
    uint32_t warp[32];
    uint32_t batch_max[kClBatches];
    uint16_t batch_c[kClBatches], batch_a[kClBatches], batch_b[kClBatches];
};

constexpr size_t kClFixedSmem = kClHistWords * 4 + kClBins;  // histogram, bin codes; then the row
constexpr size_t kClSharedMost = 227 * 1024;
static_assert(kClFixedSmem + kClBatches * kBatchWords * 4 + sizeof(ClusterShared) + 64 <= kClSharedMost &&
              kClFixedSmem + (kClBatches + 1) * kBatchWords * 4 + sizeof(ClusterShared) > kClSharedMost, "the most that fits");

template <typename T>
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
    const int rank = (int)cluster.block_rank(), CL = (int)cluster.num_blocks();
    const int m = blockIdx.x / CL;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nq = pl.nq;
    for (int i = t; i < kClHistWords; i += kClThreads) sh_hist[i] = 0u;
    if (t == 0) {
        sh.listed = 0u;
        sh.low_bin = kClBins;
    }
    if (t < nq) sh.q[t] = make_query(pl.adaptive ? pl.k[t] : (t ? drawn.band[m].k_hi : drawn.band[m].k_lo), d);
    cluster.barrier_arrive();
    pdl_enter();

    // ---- 1. the block's batches (512 words each) into shared memory, chunks in the swizzled order of the emission
    const int b0 = rank * per_block, nb = max(0, min(per_block, batches - b0));
    const T* row = g + (int64_t)m * ld;
    for (int b = warp; b < nb; b += 32)
        copy_batch_async<T>(row, d, (b0 + b) / kEmitGroups, (b0 + b) % kEmitGroups, lane, sh_row + b * kBatchWords);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    uint32_t my_top = 0;
    for (int b = warp; b < nb; b += 32) {
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
            for (int i = 0; i < 4; ++i) {
#pragma unroll
                for (int s = 0; s < EW::S; ++s) {
                    const uint32_t key = EW::key(x[i], s);
                    if (whole || e0 + (int64_t)(swz(chunk) * 4 + i) * EW::S + s < d) {  // the swizzle is its own inverse
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
    if (lane == 0) sh.warp[warp] = my_top;
    __syncthreads();
    my_top = __reduce_max_sync(0xFFFFFFFFu, sh.warp[lane]);
    cluster.barrier_wait();  // every block of the cluster runs: its shared memory can be written
    if (t < CL) cluster.map_shared_rank(sh.top, t)[rank] = my_top;
    const int own = kClBins / CL;  // bins of the first digit that a block resolves, two per word
    if (warp < CL) {  // warp r: how many of this block's keys lie in the range of block r
        uint32_t n = 0, low = kClBins;
        for (int i = lane; i < own / 2; i += 32) {
            const uint32_t x = sh_hist[warp * (own / 2) + i];
            n += (x & 0xFFFFu) + (x >> 16);
            if (x) low = min(low, (uint32_t)(warp * own + 2 * i));
        }
        n = __reduce_add_sync(0xFFFFFFFFu, n);
        low = __reduce_min_sync(0xFFFFFFFFu, low);
        if (lane < CL) cluster.map_shared_rank(&sh.part[0][0], lane)[rank * kClMost + warp] = (uint16_t)n;
        if (lane == 0 && low < kClBins) atomicMin(&sh.low_bin, low);
    }
    cluster.sync();
    uint32_t top = 0;
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
    if (bad) {  // the same in every block: no barrier is left waiting
        cluster.sync();
        return;
    }

    // ---- 2. first digit: this block takes the bins [rank, rank + 1) * own
    if (nq > 0) {
        // a thread owns `span` consecutive words of the block's range (more than one only in small clusters)
        constexpr int kMostWords = kClBins / 2 / kClThreads;
        const int span = max(1, own / 2 / kClThreads), word = (rank * own) / 2 + t * span;
        uint32_t c[2 * kMostWords] = {}, above = 0, sum = 0;
        if (t * span < own / 2) {
            if (span == 1) {
                uint32_t x[kClMost];
#pragma unroll
                for (int r = 0; r < kClMost; ++r) x[r] = (r < CL) ? cluster.map_shared_rank(sh_hist, r)[word] : 0u;
#pragma unroll
                for (int r = 0; r < kClMost; ++r) {
                    c[0] += x[r] & 0xFFFFu;
                    c[1] += x[r] >> 16;
                }
            } else {
                for (int r = 0; r < CL; ++r)
#pragma unroll
                    for (int i = 0; i < kMostWords; ++i) {
                        const uint32_t x = i < span ? cluster.map_shared_rank(sh_hist, r)[word + i] : 0u;
                        c[2 * i] += x & 0xFFFFu;
                        c[2 * i + 1] += x >> 16;
                    }
            }
        }
#pragma unroll
        for (int i = 0; i < 2 * kMostWords; ++i) sum += c[i];
        // keys in the ranges above this block's, then in the block's bins above this thread's
        for (int i = lane; i < CL * kClMost; i += 32) above += (i % kClMost > rank && i % kClMost < CL) ? sh.part[i / kClMost][i % kClMost] : 0u;
        above = __reduce_add_sync(0xFFFFFFFFu, above);
        uint32_t suffix = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(0xFFFFFFFFu, suffix, o);
            if (lane + o < 32) suffix += y;
        }
        __syncthreads();  // sh.warp has been read
        if (lane == 0) sh.warp[warp] = suffix;
        __syncthreads();
        above += suffix - sum + __reduce_add_sync(0xFFFFFFFFu, lane > warp ? sh.warp[lane] : 0u);
        if (sum) {
            for (int j = 0; j < nq; ++j) {
                const uint32_t k = sh.q[j].k;
                if (above < k && k <= above + sum && sh.q[j].trivial == 0u) {  // this thread's bins hold rank k
                    uint32_t bin = 0, ab = 0, run = above;
#pragma unroll
                    for (int i = 2 * kMostWords - 1; i >= 0; --i) {  // the last bin that is entered holds the rank
                        if (run < k) {
                            bin = (uint32_t)(2 * word + i);
                            ab = run;
                        }
                        run += c[i];
                    }
                    for (int r = 0; r < CL; ++r) {
                        Query& q = cluster.map_shared_rank(sh.q, r)[j];
                        q.prefix = bin << kShift1;
                        q.rem = k - ab;
                    }
                }
            }
        }
        cluster.sync();
    }
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
    for (int i = t; i < kClHistWords; i += kClThreads) sh_hist[i] = 0u;
    __syncthreads();
    {
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
    // The places of the keys in boundary bins are listed by the first pass over them, behind the counts (two digits of at
    // most `slots` slots), as far as they fit; otherwise the passes after it look at every key again.
    const uint32_t hist_words = (sh.slots << kBits2) / 2 > (uint32_t)(nq << kShift2) / 2 ? (sh.slots << kBits2) / 2 : (uint32_t)(nq << kShift2) / 2;
    uint16_t* sh_list = reinterpret_cast<uint16_t*>(sh_hist + ((hist_words + 3u) & ~3u));
    const uint32_t list_cap = 2u * (kClHistWords - ((hist_words + 3u) & ~3u));
    auto key_at = [&](uint32_t place) -> uint32_t { return EW::key(sh_row[place / EW::S], place % EW::S); };
    auto for_each_boundary_key = [&](auto&& f) {
        const uint32_t n = sh.listed;
        if (n <= list_cap) {
            for (uint32_t i = t; i < n; i += kClThreads) f(key_at(sh_list[i]));
        } else {
            for_each_key([&](uint32_t key, uint32_t) {
                if (sh_tab[key >> kShift1] >= 64u) f(key);
            });
        }
    };
    // One more digit of every query: `bits` bits at `shift`, counted per slot.  Warp w of block r takes query r + w CL: a
    // lane adds up its share of the slot's counts over the blocks, the warp finds the digit and tells every block.
    auto descend = [&](auto bits_tag, int shift, bool last) {
        constexpr int bits = decltype(bits_tag)::value;
        constexpr int words = (1 << bits) / 2 < 32 ? (1 << bits) / 2 : 32;  // lanes with counts
        constexpr int per = (1 << bits) / 2 / words;                       // words per lane: 8 (9 bits) or 1 (2 bits)
        cluster.sync();  // every block's counts are complete
        const int j = rank + warp * CL;
        if (j < nq && sh.q[j].trivial == 0u) {
            const int base = (int)(sh.q[j].slot << bits) / 2 + (words - 1 - lane) * per;  // lane 0 owns the largest digits
            uint32_t c[2 * per] = {}, sum = 0;
            if (lane < words) {
                for (int r = 0; r < CL; ++r) {
                    const uint32_t* src = cluster.map_shared_rank(sh_hist, r) + base;
                    if constexpr (per == 8) {
                        const uint4 a = reinterpret_cast<const uint4*>(src)[0], b = reinterpret_cast<const uint4*>(src)[1];
                        const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            c[2 * i] += x[i] & 0xFFFFu;
                            c[2 * i + 1] += x[i] >> 16;
                        }
                    } else {
                        c[0] += src[0] & 0xFFFFu;
                        c[1] += src[0] >> 16;
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 2 * per; ++i) sum += c[i];
            uint32_t upto = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
                if (lane >= o) upto += y;
            }
            const uint32_t rem = sh.q[j].rem;
            uint32_t run = upto - sum, digit = 0, left = 0, n = 0;
            const bool mine = run < rem && rem <= upto;
#pragma unroll
            for (int i = 2 * per - 1; i >= 0; --i) {
                if (run < rem) {  // the last digit that is entered holds the rank
                    digit = (uint32_t)((words - 1 - lane) * per * 2 + i);
                    left = rem - run;
                    n = c[i];
                }
                run += c[i];
            }
            const int from = __ffs(__ballot_sync(0xFFFFFFFFu, mine)) - 1;
            digit = __shfl_sync(0xFFFFFFFFu, digit, from);
            left = __shfl_sync(0xFFFFFFFFu, left, from);
            n = __shfl_sync(0xFFFFFFFFu, n, from);
            const uint32_t prefix = sh.q[j].prefix | (digit << shift), k = sh.q[j].k;
            __syncwarp();
            if (lane < CL) {
                Query& q = cluster.map_shared_rank(sh.q, lane)[j];
                q.prefix = prefix;
                q.rem = left;
                if (last) {
                    q.T = prefix;
                    q.r = left;
                    q.n = n;
                    q.c = k - left;
                }
            }
        }
        cluster.sync();
    };
    auto count = [&](uint32_t i) { atomicAdd(&sh_hist[i >> 1], 1u << ((i & 1u) * 16u)); };
    if (nq > 0) {
        for_each_key([&](uint32_t key, uint32_t place) {
            const uint32_t code = sh_tab[key >> kShift1];
            if (code >= 64u) {
                count(((code - 64u) << kBits2) | ((key >> kShift2) & ((1u << kBits2) - 1u)));
                const uint32_t at = atomicAdd(&sh.listed, 1u);
                if (at < list_cap) sh_list[at] = (uint16_t)place;
            }
        });
        descend(std::integral_constant<int, kBits2>(), kShift2, kShift2 == 0);
        if constexpr (kShift2 > 0) {
            if (warp == 0) number_slots(false);
            for (uint32_t i = t; i < hist_words; i += kClThreads) sh_hist[i] = 0u;
            __syncthreads();
            for_each_boundary_key([&](uint32_t key) {
                const uint32_t s = sh_tab[key >> kShift1] - 64u;
                for (int j = (int)sh.first[s]; j < nq && sh.q[j].trivial == 0u && sh.q[j].slot2 == s; ++j) {
                    if ((sh.q[j].prefix >> kShift2) == (key >> kShift2)) {
                        count((sh.q[j].slot << kShift2) | (key & ((1u << kShift2) - 1u)));
                        break;
                    }
                }
            });
            descend(std::integral_constant<int, (kShift2 > 0 ? kShift2 : 2)>(), 0, true);
        }
    }

    // ---- 3. energies of the open intervals
    if (pl.adaptive) {
        // A cell is (interval, exponent), numbered interval + (largest exponent - exponent): neither falls as the keys fall.
        auto exponent = [&](uint32_t key) -> int { return (int)((Tr::kVec == 4 ? key : key << 16) >> 23); };
        const int top_e = exponent(top);
        const int span = nq + 1 + top_e - exponent(min(sh.low_bin, (uint32_t)kClBins - 1u) << kShift1);  // cells of this block
        const bool many = span * 3 * 32 > kClHistWords;
        const int copies = many ? kClCopiesLow : 32, copy = lane & (copies - 1);
        // the keys of the boundary bins first, while their list is intact: their cells wait in a register each
        __syncthreads();
        const uint32_t nlist = sh.listed;
        const bool by_list = nq > 0 && nlist <= list_cap && nlist <= 8u * kClThreads;
        uint32_t held[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) held[i] = (by_list && (uint32_t)(t + i * kClThreads) < nlist) ? sh_list[t + i * kClThreads] : 0xFFFFFFFFu;
        __syncthreads();
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
        if (t < 2 * kClCells) {  // thread 2 c + h adds half h of cell c over the blocks
            unsigned long long x[kClMost], sum = 0;
#pragma unroll
            for (int r = 0; r < kClMost; ++r) x[r] = (r < CL) ? cluster.map_shared_rank(sh_sum, r)[t] : 0ull;
#pragma unroll
            for (int r = 0; r < kClMost; ++r) sum += x[r];
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
            for (int x = e_hi - lane; x >= e_lo; x -= 32) {
                const double c = sh_cell[l + top_e - x];
                if (c != 0.0) e += ldexp(c, 2 * ((x ? x : 1) - 150));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
            if (lane == 0) sh.E[l] = e;
        }
        __syncthreads();
    }
    {
        const int level = pl.adaptive ? 0 : drawn.band[m].level;
        const double p_sel = pl.adaptive ? 0.0 : drawn.band[m].p;
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
    uint32_t nC = 0, nA = 0, nB = 0, listed = 0;  // of this warp's batches
    for (int b = warp; b < nb; b += 32) {
        uint32_t bC = 0, bA = 0, bB = 0;
        if (on && sh.batch_max[b] >= band.Tb) {
            ++listed;
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
        nC += bC; nA += bA; nB += bB;
    }
    // the block's totals, by four warps' worth of shared words
    __shared__ uint32_t sh_tot[4];
    if (t < 4) sh_tot[t] = 0u;
    __syncthreads();
    if (lane == 0) {
        if (nC) atomicAdd(&sh_tot[0], nC);
        if (nA) atomicAdd(&sh_tot[1], nA);
        if (nB) atomicAdd(&sh_tot[2], nB);
        if (listed) atomicAdd(&sh_tot[3], listed);
    }
    __syncthreads();
    if (t < CL) cluster.map_shared_rank(sh.counts, t)[rank] = make_uint4(sh_tot[0], sh_tot[1], sh_tot[2], sh_tot[3]);
    cluster.sync();  // also: nothing of another block's memory is read after this
    uint4 before = make_uint4(0u, 0u, 0u, 0u), all = before;
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

int configure_cluster_kernels() {
    auto set = [&](auto kernel) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cluster_smem(kClBatches)) != cudaSuccess) return false;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    };
    return set(cluster_topk_kernel<float>) && set(cluster_topk_kernel<bf16_t>) ? MLMC_OK : MLMC_ERR_CUDA;
}

void cluster_limits(KernelLimits* limits) { clusters_that_fit(cluster_topk_kernel<float>, kClThreads, cluster_smem(kClBatches), limits->topk_fit); }

// Blocks per cluster for this call, 0: the row is too long, or the workers are too many, for the cluster to be the faster way.
// The smallest cluster whose blocks have at most kClEasy batches: a barrier and an exchange between more blocks take longer
// than the work that they share out.  Clusters that do not fit the GPU at a time run one after the other, where the launch
// chain has the whole GPU: two waves are worth it for fp32 rows whose blocks are not stretched beyond kClEasy batches, three never.
// bf16 rows (whose chain needs one sweep) only in one wave and not stretched.  us per call, cluster / chain, layered rows:
//   fp32, adaptive     131k x 12 33 / 77, x 16 (two waves) 61 / 77, x 32 (three) 93 / 90; 262k x 8 (two) 75 / 75, x 16 (three)
//                      112 / 83; 700k x 4 58 / 78, x 8 (two, stretched) 105 / 89, x 32 258 / 134
//   fp32, given p      262k x 4 24 / 54, x 8 (two) 46 / 55, x 16 (three) 68 / 60
//   bf16, adaptive     262k x 12 50 / 56, x 16 (two) 68 / 58; 500k x 4 46 / 51; 700k x 4 (stretched) 59 / 53, x 32 236 / 85
//   bf16, given p      500k x 4 22 / 36, x 8 (two) 40 / 36, x 32 99 / 55
int cluster_blocks(const Workspace& ws, int dtype, int64_t d, int M) {
    const int64_t batches = (int64_t)emit_tiles_per_worker(d, dtype) * kEmitGroups;
    if (M > 32) return 0;
    int i = 0;
    while (i < 4 && ws.limits.topk_fit[i + 1] > 0 && batches > (int64_t)kClEasy << i) ++i;
    const int fit = ws.limits.topk_fit[i];
    if (fit == 0) return 0;
    const int64_t per = (batches + (1 << i) - 1) >> i;
    const int waves = (M + fit - 1) / fit;
    const int64_t most = dtype == MLMC_BF16 ? (waves == 1 ? kClEasy : 0) : waves == 1 ? kClBatches : waves == 2 ? kClEasy : 0;
    return per <= most ? 1 << i : 0;
}

void launch_cluster_topk(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const FinishPlan& plan,
                         const DrawnBand* bands, const mlmc_topk_msgs* out, cudaStream_t s) {
    const int tiles = emit_tiles_per_worker(d, dtype);
    const int batches = tiles * kEmitGroups, cl = cluster_blocks(ws, dtype, d, M), per = (batches + cl - 1) / cl;
    if (out) ws.last_emit_tiles = tiles;
    DrawnList<32> drawn = {};
    if (bands)
        for (int m = 0; m < M; ++m) drawn.band[m] = bands[m];
    auto go = [&](auto kernel, auto* row) {
        launch_kernel_cluster(ws, K_CLUSTER_TOPK, cl, kernel, dim3(M * cl), kClThreads, cluster_smem(per), s, row, d, ld, plan, drawn,
                              batches, per, ws.p_all, ws.delta_all, out ? out->idx : nullptr, out ? out->val : nullptr, ws.group_n,
                              ws.status, ws.worker_err);
    };
    if (dtype == MLMC_BF16) go(cluster_topk_kernel<bf16_t>, static_cast<const bf16_t*>(g));
    else go(cluster_topk_kernel<float>, static_cast<const float*>(g));
}

}  // namespace mlmc
