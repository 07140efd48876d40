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
constexpr int kClBatches = 86;                   // batches per block at most: 172 KB of the row,
constexpr int kClBatchesBf16 = 63;               // for bf16 as many as a 16-bit count takes
constexpr int kClCells = 32 + 256;               // interval + (254 - exponent field)
constexpr int kClCopies = 8;                     // copies of a cell's limbs
static_assert(kClCells * 3 * kClCopies <= kClHistWords, "the cells take the place of the histogram");
static_assert(kClBatches * kBatchWords < 65536 && kClBatchesBf16 * kBatchWords * 2 < 65536, "16-bit counts, and 16-bit limbs added at most 65535 times");

struct ClusterShared {
    Query q[kMaxQueries];
    uint32_t first[kMaxQueries], slots;          // first query of a boundary bin (slot), number of slots
    double E[kMaxLevels];
    EmitParams emit;
    uint32_t total[kClMost], top[kClMost];       // per block: keys in its bins / its largest key
    uint4 counts[kClMost];                       // per block: {C, A, B, batches}
    uint32_t warp[32];
    uint32_t batch_max[kClBatches];
    uint16_t batch_c[kClBatches], batch_a[kClBatches], batch_b[kClBatches];
};

constexpr size_t kClFixedSmem = kClHistWords * 4 + kClBins;  // histogram, bin codes; then the row

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
    if (t < nq) sh.q[t] = make_query(pl.adaptive ? pl.k[t] : (t ? drawn.band[m].k_hi : drawn.band[m].k_lo), d);
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
    if (t < CL) cluster.map_shared_rank(sh.top, t)[rank] = my_top;
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

    // ---- 2. first digit: this block takes the bins [rank, rank + 1) * kClBins / CL
    if (nq > 0) {
        const int own = kClBins / CL;  // 512 or 1024 bins, two per word
        uint32_t c0 = 0, c1 = 0;
        const int word = (rank * own) / 2 + t;
        if (t < own / 2) {
#pragma unroll 8
            for (int r = 0; r < CL; ++r) {
                const uint32_t x = cluster.map_shared_rank(sh_hist, r)[word];
                c0 += x & 0xFFFFu;
                c1 += x >> 16;
            }
        }
        // keys of the block's bins above this thread's: suffix sums (threads past own / 2 hold none)
        const uint32_t sum = c0 + c1;
        uint32_t suffix = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_down_sync(0xFFFFFFFFu, suffix, o);
            if (lane + o < 32) suffix += y;
        }
        if (lane == 0) sh.warp[warp] = suffix;
        __syncthreads();
        const uint32_t w = sh.warp[lane];
        uint32_t above = suffix - sum + __reduce_add_sync(0xFFFFFFFFu, lane > warp ? w : 0u);
        const uint32_t mine = __reduce_add_sync(0xFFFFFFFFu, w);
        if (t < CL) cluster.map_shared_rank(sh.total, t)[rank] = mine;
        cluster.sync();
        for (int r = rank + 1; r < CL; ++r) above += sh.total[r];
        if (t < own / 2) {
            for (int j = 0; j < nq; ++j) {
                const uint32_t k = sh.q[j].k;
                if (sh.q[j].trivial == 0u && above < k && k <= above + sum) {  // this thread's bins hold rank k
                    const bool upper = k <= above + c1;
                    const uint32_t bin = (uint32_t)(2 * word + (upper ? 1 : 0)), ab = upper ? above : above + c1;
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
    // codes of the bins: 64 + slot where a boundary lies in the bin, else the number of boundaries above it
    if (t < kMaxQueries) {
        const int j = t;
        uint32_t slot = 0, prev = kKeyNone;
        bool is_first = false;
        if (j < nq) {
            for (int i = 0; i <= j; ++i) {
                if (sh.q[i].trivial) continue;
                const bool next = prev == kKeyNone || sh.q[i].prefix != prev;
                if (next && prev != kKeyNone) ++slot;
                if (i == j) is_first = next;
                prev = sh.q[i].prefix;
            }
            if (!sh.q[j].trivial) {
                sh.q[j].slot2 = slot;
                if (is_first) sh.first[slot] = (uint32_t)j;
            }
        }
        const uint32_t firsts = __ballot_sync(0xFFFFFFFFu, j < nq && is_first);
        if (j == 0) sh.slots = (uint32_t)__popc(firsts);
    }
    for (int i = t; i < kClHistWords; i += kClThreads) sh_hist[i] = 0u;
    __syncthreads();
    {
        constexpr int per = kClBins / kClThreads;  // 8 consecutive bins per thread
        int j = 0;
        auto bin_of = [&](int i) -> int {
            const Query& q = sh.q[i];
            return q.trivial == 0u ? (int)(q.prefix >> kShift1) : (q.trivial == 2u ? -1 : kClBins);
        };
        uint32_t codes[2] = {0u, 0u};
#pragma unroll
        for (int i = per - 1; i >= 0; --i) {
            const int b = t * per + i;
            while (j < nq && bin_of(j) > b) ++j;
            const uint32_t code = (j < nq && bin_of(j) == b) ? 64u + sh.q[j].slot2 : (uint32_t)j;
            codes[i >> 2] |= code << (8 * (i & 3));
        }
        reinterpret_cast<uint2*>(sh_tab)[t] = make_uint2(codes[0], codes[1]);
    }
    __syncthreads();
    const int words4 = nb * kBatchWords / 4;
    // every key of the block's words; the padding past the row's end has keys above every finite one
    auto for_each_key = [&](auto&& f) {
        for (int i = t; i < words4; i += kClThreads) {
            const uint4 q = *reinterpret_cast<const uint4*>(sh_row + i * 4);
            const uint32_t x[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int c = 0; c < 4; ++c)
#pragma unroll
                for (int s = 0; s < EW::S; ++s) f(EW::key(x[c], s));
        }
    };
    // one more digit of every query: count_bits bits at `shift`, counted per slot.  Every CL-th query is this block's.
    auto descend = [&](int shift, int bits, bool last) {
        cluster.sync();  // every block's counts are complete
        const int nwords = (1 << bits) / 2 > 0 ? (1 << bits) / 2 : 1;
        for (int j = rank; j < nq; j += CL) {
            if (sh.q[j].trivial) continue;  // block-uniform
            const uint32_t base = (sh.q[j].slot << bits) / 2;
            uint32_t c0 = 0, c1 = 0;
            if (t < nwords) {
#pragma unroll 8
                for (int r = 0; r < CL; ++r) {
                    const uint32_t x = cluster.map_shared_rank(sh_hist, r)[base + t];
                    c0 += x & 0xFFFFu;
                    c1 += x >> 16;
                }
            }
            const uint32_t sum = c0 + c1;
            uint32_t suffix = sum;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_down_sync(0xFFFFFFFFu, suffix, o);
                if (lane + o < 32) suffix += y;
            }
            __syncthreads();
            if (lane == 0) sh.warp[warp] = suffix;
            __syncthreads();
            const uint32_t w = sh.warp[lane];
            const uint32_t above = suffix - sum + __reduce_add_sync(0xFFFFFFFFu, lane > warp ? w : 0u);
            const uint32_t rem = sh.q[j].rem;
            __syncthreads();  // read by everyone before the owner rewrites it
            if (t < nwords && above < rem && rem <= above + sum) {
                const bool upper = rem <= above + c1;
                const uint32_t digit = (uint32_t)(2 * t + (upper ? 1 : 0)), left = rem - (upper ? above : above + c1);
                const uint32_t prefix = sh.q[j].prefix | (digit << shift), n = upper ? c1 : c0;
                for (int r = 0; r < CL; ++r) {
                    Query& q = cluster.map_shared_rank(sh.q, r)[j];
                    q.prefix = prefix;
                    q.rem = left;
                    if (last) {
                        q.T = prefix;
                        q.r = left;
                        q.n = n;
                        q.c = q.k - left;
                    }
                }
            }
        }
        cluster.sync();
    };
    if (nq > 0) {
        if (t < nq) sh.q[t].slot = sh.q[t].slot2;
        for_each_key([&](uint32_t key) {
            const uint32_t code = sh_tab[key >> kShift1];
            if (code >= 64u) {
                const uint32_t i = ((code - 64u) << kBits2) | ((key >> kShift2) & ((1u << kBits2) - 1u));
                atomicAdd(&sh_hist[i >> 1], 1u << ((i & 1u) * 16u));
            }
        });
        descend(kShift2, kBits2, kShift2 == 0);
        if constexpr (kShift2 > 0) {
            if (t < nq && !sh.q[t].trivial) {  // queries with the same prefix share a slot (prefixes descend)
                uint32_t slot = 0, prev = kKeyNone;
                for (int i = 0; i <= t; ++i) {
                    if (sh.q[i].trivial) continue;
                    if (prev != kKeyNone && sh.q[i].prefix != prev) ++slot;
                    prev = sh.q[i].prefix;
                }
                sh.q[t].slot = slot;
            }
            for (int i = t; i < kClHistWords; i += kClThreads) sh_hist[i] = 0u;
            __syncthreads();
            for_each_key([&](uint32_t key) {
                const uint32_t code = sh_tab[key >> kShift1];
                if (code >= 64u) {
                    const uint32_t s = code - 64u;
                    for (int j = (int)sh.first[s]; j < nq && !sh.q[j].trivial && sh.q[j].slot2 == s; ++j) {
                        if ((sh.q[j].prefix >> kShift2) == (key >> kShift2)) {
                            const uint32_t i = (sh.q[j].slot << kShift2) | (key & ((1u << kShift2) - 1u));
                            atomicAdd(&sh_hist[i >> 1], 1u << ((i & 1u) * 16u));
                            break;
                        }
                    }
                }
            });
            descend(0, kShift2, true);
        }
    }

    // ---- 3. energies of the open intervals
    if (pl.adaptive) {
        __syncthreads();
        for (int i = t; i < kClCells * 3 * kClCopies; i += kClThreads) sh_hist[i] = 0u;
        __syncthreads();
        const uint32_t copy = lane & (kClCopies - 1);
        const uint32_t top_e = 254u;
        for_each_key([&](uint32_t key) {
            uint32_t interval = sh_tab[key >> kShift1];
            if (interval >= 64u) {
                const uint32_t s = interval - 64u;
                int j = (int)sh.first[s];
                while (j < nq && sh.q[j].T > key) ++j;  // thresholds descend; a query with k = d has T = 0
                if (j < nq && sh.q[j].T == key && sh.q[j].trivial == 0u) return;  // a threshold key: added from its count
                interval = (uint32_t)j;
            }
            if (key >= Tr::kInfKey || key == 0u) return;  // padding; zeros add nothing
            const uint32_t bits = Tr::kVec == 4 ? key : key << 16;
            const uint64_t m2 = mantissa_squared(bits);
            uint32_t* a = sh_hist + (interval + top_e - (bits >> 23)) * (3 * kClCopies) + copy;
            atomicAdd(a, (uint32_t)m2 & 0xFFFFu);
            atomicAdd(a + kClCopies, (uint32_t)(m2 >> 16) & 0xFFFFu);
            atomicAdd(a + 2 * kClCopies, (uint32_t)(m2 >> 32));
        });
        __syncthreads();
        unsigned long long* sh_sum = reinterpret_cast<unsigned long long*>(sh_tab);  // [kClCells][2]: the codes are not needed any more
        static_assert(kClCells * 16 <= kClBins, "the sums take the place of the codes");
        if (t < kClCells) {
            unsigned long long lo = 0, hi = 0;
            const uint32_t* a = sh_hist + t * (3 * kClCopies);
#pragma unroll
            for (int r = 0; r < kClCopies; ++r) {
                lo += (unsigned long long)a[r] + ((unsigned long long)a[kClCopies + r] << 16);
                hi += a[2 * kClCopies + r];
            }
            sh_sum[2 * t] = lo;
            sh_sum[2 * t + 1] = hi;
        }
        cluster.sync();
        double* sh_cell = reinterpret_cast<double*>(sh_hist);  // [kClCells]: sum of mant^2 over the row
        if (t < kClCells) {
            unsigned long long lo = 0, hi = 0;
#pragma unroll 4
            for (int r = 0; r < CL; ++r) {
                const unsigned long long* o = cluster.map_shared_rank(sh_sum, r);
                lo += o[2 * t];
                hi += o[2 * t + 1];
            }
            const unsigned __int128 tot = ((unsigned __int128)hi << 32) + lo;
            sh_cell[t] = (double)(unsigned long long)(tot >> 64) * 0x1.0p64 + (double)(unsigned long long)tot;
        }
        __syncthreads();
        // interval l, one warp each: the exponents between those of its two thresholds, in a fixed order
        for (int l = warp; l < pl.L; l += kClThreads / 32) {
            const uint32_t T_up = l ? sh.q[l - 1].T : kKeyNone, T_dn = l < nq ? sh.q[l].T : 0u;
            auto exponent = [&](uint32_t key) -> int { return (int)((Tr::kVec == 4 ? key : key << 16) >> 23); };
            const int e_hi = T_up == kKeyNone ? 254 : exponent(T_up), e_lo = T_dn == kKeyNone ? 255 : exponent(T_dn);
            double e = 0.0;
            for (int x = e_hi - lane; x >= e_lo; x -= 32) e += ldexp(sh_cell[l + 254 - x], 2 * ((x ? x : 1) - 150));
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
    for (int b = warp; b < nb; b += 32) {
        if (sh.batch_c[b] == 0) continue;
        uint32_t pc = 0, pa = 0, pb = 0;  // counts of the block's batches before this one
        for (int i = lane; i < b; i += 32) { pc += sh.batch_c[i]; pa += sh.batch_a[i]; pb += sh.batch_b[i]; }
        pc = __reduce_add_sync(0xFFFFFFFFu, pc);
        pa = __reduce_add_sync(0xFFFFFFFFu, pa);
        pb = __reduce_add_sync(0xFFFFFFFFu, pb);
        uint3 run = make_uint3(before.x + pc, before.y + pa, before.z + pb);
        emit_batch<T>(sh_row + b * kBatchWords, band, (sh.batch_a[b] | sh.batch_b[b]) != 0, (uint32_t)((b0 + b) * kBatchWords * EW::S), run,
                      idx_w, val_w, pl.capacity);
    }
}

size_t cluster_smem(int per_block) { return kClFixedSmem + (size_t)per_block * kBatchWords * 4; }

}  // namespace

int configure_cluster_kernels(Workspace& ws) {
    ws.cluster_most = 0;
    auto set = [&](auto kernel) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cluster_smem(kClBatches)) != cudaSuccess) return false;
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    };
    if (!set(cluster_topk_kernel<float>) || !set(cluster_topk_kernel<bf16_t>)) return MLMC_ERR_CUDA;
    // the largest cluster that the device can place with the largest blocks
    for (int cl : {16, 8}) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(cl);
        cfg.blockDim = dim3(kClThreads);
        cfg.dynamicSmemBytes = cluster_smem(kClBatches);
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = cl;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int n = 0;
        if (cudaOccupancyMaxActiveClusters(&n, cluster_topk_kernel<float>, &cfg) == cudaSuccess && n >= 1) {
            ws.cluster_most = cl;
            break;
        }
        cudaGetLastError();
    }
    return MLMC_OK;
}

// Blocks per cluster for this call, 0: the row is too long (or the workers too many) for it.
int cluster_blocks(const Workspace& ws, int dtype, int64_t d, int M) {
    const int batches = emit_tiles_per_worker(d, dtype) * kEmitGroups;
    if (M > 32 || ws.cluster_most == 0) return 0;
    int cl = 8;
    if (batches > 8 * 32 && ws.cluster_most >= 16) cl = 16;  // more than 64 KB per block: twice the blocks
    return (batches + cl - 1) / cl <= (dtype == MLMC_BF16 ? kClBatchesBf16 : kClBatches) ? cl : 0;
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
