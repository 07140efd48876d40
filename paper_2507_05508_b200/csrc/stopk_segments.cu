// s-Top-k with adaptive probabilities and more segments than kMaxLevels (Sec. 2.2 "s-segmented Top-k", App. D,
// Lemma 3.4: p^l proportional to the norm of segment l of the sorted vector).
//
// The norms of all L segments are needed, but not the sorted vector: segment l is the ranks (s l, s (l + 1)], so it is
// known once the thresholds of the L - 1 segment boundaries and the energy between them are.  The leading-digit
// histogram (hist1) tells which of its 2^15 bins hold a boundary.
//   fp32: a sweep over the row adds up the energy of every other bin and moves the keys of the boundary bins ("buckets",
//   a few to all of the row's keys, depending on L) to one place per bucket; a block per bucket then finds the
//   boundaries in it by two 8-bit digits.  All keys of a bin share their exponent, so their energies are sums of the
//   48-bit integers mant^2: exact, whatever the order of the keys.
//   bf16: a bin is one key; the segment energies and the thresholds follow from the histogram alone.
// Then p, the draw and the two thresholds of the drawn segment; the band is emitted like every other Top-k message.
// Rows are taken together while their scratch memory fits in a fixed budget.
// A row whose buckets would hold most of its keys, or one of them a large share, is sorted instead (stopk_sort.cu): a bucket is
// the work of one block, and ties and zeros meet in one.
#include <algorithm>

#include "stopk_sort.cuh"

namespace mlmc {

namespace {

constexpr int kSegThreads = 1024;
constexpr int kBucketThreads = 256;
constexpr int kMaxCells = kBins1;                            // (segment, exponent) pairs of bins without a boundary
constexpr size_t kSegScratchBudget = size_t(1) << 30;

// A row is sorted (stopk_sort.cu) where too many of its keys lie in buckets, or more than 1/32 of them in one bucket; not where that
// is fewer than kFewKeys keys in all, or kFewEqual in one bucket: the passes of a sort take that long at least.
//   Moving a key to its bucket costs more the more blocks of a row meet at the buckets' counters: 45 us per 10^6 keys with 4 rows in
//   flight, 27 with 16, where a sort takes 25 per 10^6 keys of the row.  So the share from which on a row is sorted is 9/16 with
//   up to 8 rows and 13/16 with more.  Normal entries, 11.7M x 4, buckets against sort: share 0.53 1412 and 1410 us, 0.66 1732
//   and 1408; 11.7M x 16: 0.75 3364 and 5003, 0.89 4708 and 5001; 2M x 16: 0.75 1018 and 1091, 0.89 1163 and 1020.
//   A bucket is the work of one block: 10^6 keys of different values 0.2 ms, equal ones 1.9 ms.
constexpr uint32_t kFewKeys = 1u << 18, kFewEqual = 1u << 14;
uint32_t sort_from(uint32_t d, int rows) { return std::max(kFewKeys, d / 16 * (rows <= 8 ? 9 : 13)); }

// One boundary bin of a row.
struct Bucket {
    uint32_t bin, count;     // its keys
    uint32_t above;          // keys above it
    uint32_t offset;         // where its keys are collected
    uint32_t first, n;       // boundaries first .. first + n - 1 lie in it
    uint32_t pad[2];
};

struct Wide {  // a sum of mant^2 (below 2^80): hi 2^64 + lo
    unsigned long long lo, hi;
};
__device__ __forceinline__ Wide wide(unsigned __int128 x) { return {(unsigned long long)x, (unsigned long long)(x >> 64)}; }
__device__ __forceinline__ unsigned __int128 wide128(const Wide& w) { return ((unsigned __int128)w.hi << 64) | w.lo; }
__device__ __forceinline__ double wide_to_double(unsigned __int128 x) {
    return (double)(unsigned long long)(x >> 64) * 0x1.0p64 + (double)(unsigned long long)x;
}
// mant^2 units of a bin with biased exponent ex, as a power of two
__device__ __forceinline__ double energy_unit(double x, int ex) { return ldexp(x, 2 * ((ex ? ex : 1) - 150)); }

// Scratch memory of the rows that are taken together, by row strides.
struct SegScratch {
    uint32_t* keys;          // [rows][d]           keys of the buckets
    uint16_t* table;         // [rows][kBins1]      bin -> cell, or 0x8000 | bucket
    Bucket* bucket;          // [rows][kBins1]
    Wide* bucket_sum;        // [rows][kBins1]      energy of a bucket
    uint32_t* cursor;        // [rows][kBins1]      next free place of a bucket
    unsigned long long* cell; // [rows][kMaxCells][2] energy of a cell: sum = hi 2^32 + lo
    uint8_t* cell_exp;       // [rows][kMaxCells]
    uint2* seg_cells;        // [rows][seg_cap]     {first cell, one past the last cell} of a segment
    uint2* bound;            // [rows][seg_cap]     {T, r} of boundary j
    Wide* prefix;            // [rows][seg_cap]     energy of the keys of its bucket inside boundary j
    double* delta;           // [rows][seg_cap]     norm of segment l
    RowHead* head;           // [rows]
    SortBuffers sort;        // of the rows that are sorted; the first buffer is `keys`
    int64_t key_stride, seg_cap;
};

__device__ __forceinline__ uint32_t block_exclusive_sum(uint32_t x, uint32_t* sh_warp, uint32_t* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t inc = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    __syncthreads();
    if (lane == 31) sh_warp[warp] = inc;
    __syncthreads();
    const uint32_t w = sh_warp[lane];
    const uint32_t before = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u);
    *total = __reduce_add_sync(0xFFFFFFFFu, w);
    return before + inc - x;
}

// Walks the bins in falling order: `run` keys so far, `passed` boundaries (ranks s, 2 s, .., top s) at or above them.
struct Boundaries {
    uint32_t run, passed, s_len, top;
    uint64_t next;  // rank of the next boundary
    __device__ Boundaries(uint32_t above, uint32_t s, uint32_t most) : run(above), passed(min(above / s, most)), s_len(s), top(most) {
        next = (uint64_t)s * (passed + 1u);
    }
    __device__ __forceinline__ bool advance(uint32_t n) {  // true: the bin holds a boundary
        run += n;
        if ((uint64_t)run < next || passed == top) return false;
        passed = min(run / s_len, top);
        next = (uint64_t)s_len * (passed + 1u);
        return true;
    }
};

// Which bins hold a boundary.  One block per row; thread t owns the 32 bins from 32 (1023 - t), so that the order of
// the threads is the order of falling keys.  Boundary j is rank s (j + 1), j < L - 1.
// sort_all, sort_one: with more keys than that in buckets, or in one of them, the row is sorted.
// bf16: only the running counts are needed: hist[b] becomes #{key >= b}.
template <bool BF16>
__global__ void __launch_bounds__(kSegThreads, 1)
segment_resolve_kernel(uint32_t* hist1, int m0, uint32_t sort_all, uint32_t sort_one, uint32_t s_len, uint32_t L, SegScratch sc, const int* worker_err) {
    __shared__ uint32_t sh_warp[32], sh_most[32];
    pdl_enter();
    const int row = blockIdx.x, m = m0 + row;
    const int group = kSegThreads - 1 - (int)threadIdx.x, warp = threadIdx.x >> 5;
    uint4 vectors[8];
    load_bins(hist1 + (int64_t)m * kBins1 + (31 - warp) * 1024, vectors);
    if (worker_err[m]) {
        if (threadIdx.x == 0) sc.head[row].sorted = 0u;
        return;
    }
    uint4* src = reinterpret_cast<uint4*>(hist1 + (int64_t)m * kBins1 + group * 32);
    uint32_t cnt[32];
    {
        extern __shared__ __align__(16) uint4 sh_vectors[];  // [32 warps][256]
        hand_over_bins(vectors, sh_vectors + warp * 256, group & 31, cnt);
    }
    uint32_t sum = 0, total;
#pragma unroll
    for (int i = 0; i < 32; ++i) sum += cnt[i];
    const uint32_t above = block_exclusive_sum(sum, sh_warp, &total);
    if constexpr (BF16) {
        uint32_t run = above;
#pragma unroll
        for (int i = 31; i >= 0; --i) cnt[i] = run += cnt[i];
#pragma unroll
        for (int i = 0; i < 8; ++i) src[i] = make_uint4(cnt[4 * i], cnt[4 * i + 1], cnt[4 * i + 2], cnt[4 * i + 3]);
        return;
    }
    uint2* seg_cells = sc.seg_cells + (int64_t)row * sc.seg_cap;
    for (uint32_t l = threadIdx.x; l < L; l += kSegThreads) seg_cells[l] = make_uint2(0xFFFFFFFFu, 0u);
    // first pass over the bins: how many buckets, cells and collected keys this thread has.  A cell is the bins of one
    // segment without a boundary and of one exponent: the four threads of an exponent carry it on.
    const uint32_t top = L - 1;  // boundaries
    uint32_t nb = 0, nc = 0, nk = 0, most = 0, carry = 0xFFFFFFFFu;
    {
        uint32_t last = 0xFFFFFFFFu, first = 0xFFFFFFFFu;
        Boundaries at(above, s_len, top);
#pragma unroll
        for (int i = 31; i >= 0; --i) {
            if (cnt[i] == 0u) continue;
            const uint32_t lo = at.passed;
            if (at.advance(cnt[i])) {
                ++nb;
                nk += cnt[i];
                most = max(most, cnt[i]);
            } else if (lo != last) {
                ++nc;
                if (last == 0xFFFFFFFFu) first = lo;
                last = lo;
            }
        }
#pragma unroll
        for (int o = 3; o > 0; --o) {  // the last segment of the nearest thread before that has one
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, last, o);
            if ((threadIdx.x & 3) >= (unsigned)o && y != 0xFFFFFFFFu) carry = y;
        }
        if (carry != 0xFFFFFFFFu && carry == first) --nc;
    }
    most = __reduce_max_sync(0xFFFFFFFFu, most);
    if ((threadIdx.x & 31) == 0) sh_most[threadIdx.x >> 5] = most;  // read after the barriers of the scans
    uint32_t all_b, all_c, all_k;
    uint32_t b = block_exclusive_sum(nb, sh_warp, &all_b), c = block_exclusive_sum(nc, sh_warp, &all_c),
             k = block_exclusive_sum(nk, sh_warp, &all_k);
    most = __reduce_max_sync(0xFFFFFFFFu, sh_most[threadIdx.x & 31]);
    const bool sorted = all_k > sort_all || most > sort_one;
    if (threadIdx.x == 0) sc.head[row] = {all_b, all_c, sorted ? 1u : 0u, 0u};
    if (sorted) return;
    unsigned long long* cell = sc.cell + (int64_t)row * kMaxCells * 2;
    for (uint32_t i = threadIdx.x; i < all_c * 2; i += kSegThreads) cell[i] = 0ull;
    uint16_t* table = sc.table + (int64_t)row * kBins1 + group * 32;
    uint32_t last = carry;
    Boundaries at(above, s_len, top);
    uint32_t code[32];
#pragma unroll
    for (int i = 31; i >= 0; --i) {
        code[i] = 0u;
        if (cnt[i] == 0u) continue;
        const uint32_t lo = at.passed, run = at.run;
        if (at.advance(cnt[i])) {
            sc.bucket[(int64_t)row * kBins1 + b] = {(uint32_t)(group * 32 + i), cnt[i], run, k, lo, at.passed - lo, {0u, 0u}};
            sc.cursor[(int64_t)row * kBins1 + b] = k;
            code[i] = 0x8000u | b;
            ++b;
            k += cnt[i];
        } else {
            if (lo != last) {  // a new cell of segment lo
                last = lo;
                sc.cell_exp[(int64_t)row * kMaxCells + c] = (uint8_t)((group * 32 + i) >> 7);
                atomicMin(&seg_cells[lo].x, c);  // ordered after the clearing above by the barriers of the scans
                atomicMax(&seg_cells[lo].y, c + 1u);
                ++c;
            }
            code[i] = c - 1u;
        }
    }
    uint4* tab = reinterpret_cast<uint4*>(table);
#pragma unroll
    for (int i = 0; i < 4; ++i)
        tab[i] = make_uint4(code[8 * i] | (code[8 * i + 1] << 16), code[8 * i + 2] | (code[8 * i + 3] << 16),
                            code[8 * i + 4] | (code[8 * i + 5] << 16), code[8 * i + 6] | (code[8 * i + 7] << 16));
}

// Sweep of the row (fp32): the energies of the cells and the keys of the buckets.  One block of 1024 threads per SM; a trip is
// 8 keys per thread, the vectors of the next two trips in flight.
//   cells: three 16-bit limbs of mant^2 in u32 words, in up to 32 copies picked by the lane (as many as fit), so that a warp's
//   additions do not meet in a bank; a copy takes 2^16 additions before its words can overflow, then it is added up.
//   The table in shared memory holds the cell's first word, so an entry costs one look-up, one multiplication and three
//   additions at constant offsets, without a branch (the keys of the buckets are added to a cell that nobody reads).
//   buckets: every warp stages its keys in a buffer of its own (places from a warp scan).  Every few trips the
//   block asks whether one fills up, and if so counts all staged keys per bucket, reserves their places with one atomic per
//   bucket, and writes them (up to kSlotSmem buckets; with more, an atomic per key).  A warp whose buffer runs full between
//   two questions (more than a third of its keys lie in buckets) writes its keys alone, with an atomic per key.
//   16 x 11.7M keys, L = 100: 401 us with a barrier per trip to ask whether a buffer is full, now 338 (asking every 2 or 8 trips: 368, 386).
constexpr int kTripVecs = 2;                                  // 16-byte vectors per thread
constexpr int kTripKeys = kSegThreads * kTripVecs * 4;
constexpr int kWarpBuffer = 640;                              // staged keys per warp
constexpr int kSegStage = kWarpBuffer * (kSegThreads / 32);
constexpr int kAskTrips = 4;                                  // trips between two questions whether a buffer fills up,
constexpr int kAskFill = 288;                                 // that is, whether it holds more than so many keys
constexpr int kSlotSmem = 1024;
constexpr int kLimbWords = 6 * 1024;                          // words of one limb of all cells and copies, and of the unread cell
constexpr int kCellWords = kLimbWords - 32;
constexpr uint32_t kFarCell = 0x7FFFu;                       // table entry of a cell that does not fit: looked up in global memory
constexpr size_t kSegSweepSmem = kBins1 * 2 + (size_t)(kSegStage + kSlotSmem * 2 + kLimbWords * 3) * 4;

// FAR: there may be more cells than fit (L + 255 > kCellWords); their entries go to global memory one by one.
template <bool FAR>
__global__ void __launch_bounds__(kSegThreads, 1)
segment_sweep_kernel(const float* __restrict__ g, int64_t d, int64_t ld, int m0, SegScratch sc, const int* worker_err) {
    extern __shared__ __align__(16) uint8_t sh_seg[];
    uint16_t* sh_tab = reinterpret_cast<uint16_t*>(sh_seg);
    uint32_t* sh_stage = reinterpret_cast<uint32_t*>(sh_seg + kBins1 * 2);
    uint32_t* sh_count = sh_stage + kSegStage;   // [kSlotSmem]
    uint32_t* sh_base = sh_count + kSlotSmem;    // [kSlotSmem]
    uint32_t* sh_cell = sh_base + kSlotSmem;     // [3][cells][copies]
    pdl_enter();
    const int row = blockIdx.y, m = m0 + row;
    if (worker_err[m]) return;
    const RowHead head = sc.head[row];
    if (head.sorted) return;
    const int lane = threadIdx.x & 31;
    const uint32_t cells = head.cells;
    int copies_log = 5;
    while (copies_log > 0 && (cells << copies_log) > (uint32_t)kCellWords) --copies_log;
    const uint32_t copies = 1u << copies_log;
    const uint32_t cells_here = min(cells, (uint32_t)kCellWords >> copies_log);
    const int trips_per_flush = (int)(copies * 65536u / (uint32_t)kTripKeys);
    const uint16_t* table = sc.table + (int64_t)row * kBins1;
    {
        auto place = [&](uint32_t c) -> uint32_t { return (c & 0x8000u) ? c : (c < cells_here ? c << copies_log : kFarCell); };
        const uint4* src = reinterpret_cast<const uint4*>(table);
        for (int i = threadIdx.x; i < kBins1 / 8; i += kSegThreads) {
            uint4 x = src[i];
            uint32_t* w = &x.x;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = place(w[j] & 0xFFFFu) | (place(w[j] >> 16) << 16);
            reinterpret_cast<uint4*>(sh_tab)[i] = x;
        }
        for (int i = threadIdx.x; i < kSlotSmem; i += kSegThreads) sh_count[i] = 0u;
        for (int i = threadIdx.x; i < kLimbWords * 3; i += kSegThreads) sh_cell[i] = 0u;
    }
    const bool slots_here = head.buckets <= (uint32_t)kSlotSmem;
    unsigned long long* cell = sc.cell + (int64_t)row * kMaxCells * 2;
    uint32_t* cursor = sc.cursor + (int64_t)row * kBins1;
    uint32_t* keys = sc.keys + (int64_t)row * sc.key_stride;
    __syncthreads();

    auto flush_cells = [&]() {  // called by all threads, after a barrier
        for (uint32_t c = threadIdx.x; c < cells_here; c += kSegThreads) {
            unsigned long long lo = 0, hi = 0;
            for (uint32_t r = 0; r < copies; ++r) {
                uint32_t* a = sh_cell + c * copies + ((r + c) & (copies - 1u));  // neighbours start in different banks
                lo += (unsigned long long)a[0] + ((unsigned long long)a[kLimbWords] << 16);
                hi += a[2 * kLimbWords];
                a[0] = a[kLimbWords] = a[2 * kLimbWords] = 0u;
            }
            if (lo) atomicAdd(&cell[c * 2], lo);
            if (hi) atomicAdd(&cell[c * 2 + 1], hi);
        }
    };
    uint32_t* buffer = sh_stage + (threadIdx.x >> 5) * kWarpBuffer;
    const uint32_t buffer0 = (uint32_t)__cvta_generic_to_shared(buffer);
    uint32_t fill = 0;  // keys in the warp's buffer (the same in every lane)
    auto flush_alone = [&]() {  // called by a warp
        __syncwarp();
        for (uint32_t i = lane; i < fill; i += 32) {
            const uint32_t key = buffer[i] & 0x7FFFFFFFu;
            keys[atomicAdd(&cursor[sh_tab[key >> 16] & 0x7FFFu], 1u)] = key;
        }
        fill = 0;
        __syncwarp();
    };
    auto flush_stage = [&]() {  // called by all threads, after a barrier
        auto slot_of = [&](uint32_t key) -> uint32_t { return sh_tab[key >> 16] & 0x7FFFu; };
        if (slots_here) {
            for (uint32_t i = lane; i < fill; i += 32) atomicAdd(&sh_count[slot_of(buffer[i] & 0x7FFFFFFFu)], 1u);
            __syncthreads();
            for (uint32_t b = threadIdx.x; b < head.buckets; b += kSegThreads) {
                const uint32_t c = sh_count[b];
                if (c) {
                    sh_base[b] = atomicAdd(&cursor[b], c);
                    sh_count[b] = 0u;
                }
            }
            __syncthreads();
            for (uint32_t i = lane; i < fill; i += 32) {
                const uint32_t key = buffer[i] & 0x7FFFFFFFu;
                keys[atomicAdd(&sh_base[slot_of(key)], 1u)] = key;
            }
        } else {
            for (uint32_t i = lane; i < fill; i += 32) {
                const uint32_t key = buffer[i] & 0x7FFFFFFFu;
                keys[atomicAdd(&cursor[slot_of(key)], 1u)] = key;
            }
        }
        fill = 0;
        __syncwarp();
    };
    const uint32_t cell0 = (uint32_t)__cvta_generic_to_shared(sh_cell) + (lane & (copies - 1u)) * 4u;
    const uint32_t unread = (uint32_t)__cvta_generic_to_shared(sh_cell) + (kCellWords + lane) * 4u;
    // the entry of a bucket is negative
    auto look_up = [&](uint32_t bits) -> int {  // the table's byte offset is twice the bin
        return *reinterpret_cast<const int16_t*>(reinterpret_cast<const char*>(sh_tab) + ((bits >> 15) & 0xFFFEu));
    };
    auto take = [&](uint32_t bits, int code) {
        const uint64_t m2 = mantissa_squared(bits);
        if (FAR && code == (int)kFarCell) {
            const uint32_t c = table[(bits >> 16) & 0x7FFFu];
            atomicAdd(&cell[c * 2], (unsigned long long)(uint32_t)m2);
            atomicAdd(&cell[c * 2 + 1], (unsigned long long)(m2 >> 32));
            code = -1;
        }
        shared_add_limbs<kLimbWords * 4>(code < 0 ? unread : cell0 + (uint32_t)code * 4u, m2);
    };
    const float* src = g + (int64_t)m * ld;
    const int64_t trips_of_row = d / kTripKeys;  // whole trips, dealt round-robin; the rest of the row is the last block's
    uint4 ring[2][kTripVecs];
    int trips_left = trips_per_flush;
    auto load = [&](int64_t trip, uint4 (&q)[kTripVecs]) {
        if (trip >= trips_of_row) return;
#pragma unroll
        for (int j = 0; j < kTripVecs; ++j)
            q[j] = __ldg(reinterpret_cast<const uint4*>(src) + trip * (kTripKeys / 4) + j * kSegThreads + threadIdx.x);
    };
    auto process = [&](uint4 (&q)[kTripVecs], int64_t next) {  // one trip; its registers take the vectors of trip `next`
        uint32_t x[kTripVecs * 4], mine = 0;
        int code[kTripVecs * 4];
#pragma unroll
        for (int j = 0; j < kTripVecs; ++j) {
            x[4 * j] = q[j].x; x[4 * j + 1] = q[j].y; x[4 * j + 2] = q[j].z; x[4 * j + 3] = q[j].w;
        }
        load(next, q);
#pragma unroll
        for (int e = 0; e < kTripVecs * 4; ++e) code[e] = look_up(x[e]);
#pragma unroll
        for (int e = 0; e < kTripVecs * 4; ++e) mine += (uint32_t)code[e] >> 31;
        uint32_t upto = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if (lane >= o) upto += y;
        }
        uint32_t at = buffer0 + (fill + upto - mine) * 4u;
        fill += __shfl_sync(0xFFFFFFFFu, upto, 31);
#pragma unroll
        for (int e = 0; e < kTripVecs * 4; ++e) {
            take(x[e], code[e]);
            shared_push_if_negative(code[e], at, x[e], 4u);
        }
        if (fill > (uint32_t)(kWarpBuffer - 32 * kTripVecs * 4)) flush_alone();  // no room for another trip
        if ((--trips_left & (kAskTrips - 1)) == 0) {  // the same for every thread, and a multiple of kAskTrips to begin with
            const bool due = __syncthreads_or(fill > (uint32_t)kAskFill);
            if (trips_left == 0) {
                flush_cells();
                trips_left = trips_per_flush;
                __syncthreads();
            }
            if (due) {
                flush_stage();
                __syncthreads();  // settled before the next trip adds to them
            }
        }
    };
    load(blockIdx.x, ring[0]);
    load((int64_t)blockIdx.x + gridDim.x, ring[1]);
    for (int64_t trip = blockIdx.x; trip < trips_of_row; trip += 2 * (int64_t)gridDim.x) {
        process(ring[0], trip + 2 * (int64_t)gridDim.x);
        if (trip + gridDim.x < trips_of_row) process(ring[1], trip + 3 * (int64_t)gridDim.x);  // block-uniform
    }
    if (blockIdx.x == gridDim.x - 1) {  // fewer than kTripKeys entries, at most 8 per thread
        __syncthreads();
        flush_stage();  // room for them
        flush_cells();
        __syncthreads();
        for (int64_t i0 = trips_of_row * kTripKeys; i0 < d; i0 += kSegThreads) {
            const int64_t i = i0 + threadIdx.x;
            const uint32_t bits = i < d ? __ldg(reinterpret_cast<const uint32_t*>(src) + i) : 0u;
            const int code = i < d ? look_up(bits) : 0;
            const uint32_t flags = __ballot_sync(0xFFFFFFFFu, code < 0);
            if (i < d) take(bits, code);
            if (code < 0) buffer[fill + __popc(flags & ((1u << lane) - 1u))] = bits;
            fill += __popc(flags);
        }
    }
    __syncthreads();
    flush_cells();
    flush_stage();
}

// The boundaries of one bucket, one block per bucket at a time.  First pass over its keys: counts and sums of the low byte
// and of its square per second digit (the energy of a sub-bin of base mantissa B is n B^2 + 2 B sum y + sum y^2, exact).
// The sub-bins that hold a boundary are then counted by their low byte in a second pass, kSubBins of them at a time;
// a warp per boundary reads off its threshold and the energy of the bucket's keys inside it.
constexpr int kSubBins = 32;
constexpr int kBucketFlush = 65536;  // keys between two flushes of the 32-bit sums of squares

__global__ void __launch_bounds__(kBucketThreads)
bucket_kernel(int m0, uint32_t s_len, SegScratch sc, const int* worker_err) {
    __shared__ uint32_t sh_cnt[256], sh_y[256], sh_y2[256];
    __shared__ unsigned long long sh_sum_y[256], sh_sum_y2[256];
    __shared__ uint32_t sh_num[256];     // keys per second digit
    __shared__ uint32_t sh_above[256];   // keys of the bucket above the sub-bin
    __shared__ Wide sh_energy[256];      // their energy
    __shared__ uint32_t sh_flag[256];    // sub-bin holds a boundary; then its number among those (falling digits)
    __shared__ uint32_t sh_hist[kSubBins][256];
    __shared__ uint32_t sh_wsum[8];
    __shared__ Wide sh_wenergy[8];
    __shared__ uint32_t sh_marked;
    pdl_enter();
    const int row = blockIdx.y;
    if (worker_err[m0 + row] || sc.head[row].sorted) return;  // (so a bucket has at most 2^27 keys)
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const uint32_t buckets = sc.head[row].buckets;
    for (uint32_t bi = blockIdx.x; bi < buckets; bi += gridDim.x) {
        const Bucket bk = sc.bucket[(int64_t)row * kBins1 + bi];
        const uint32_t* keys = sc.keys + (int64_t)row * sc.key_stride + bk.offset;
        sh_cnt[t] = sh_y[t] = sh_y2[t] = sh_flag[t] = sh_num[t] = 0u;
        sh_sum_y[t] = sh_sum_y2[t] = 0ull;
        __syncthreads();
        for (uint32_t i0 = 0; i0 < bk.count;) {
            const uint32_t end = min(bk.count, i0 + (uint32_t)kBucketFlush);
            for (uint32_t i = i0 + t; i < end; i += 4 * kBucketThreads) {
                uint32_t key[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) key[j] = (i + j * kBucketThreads < end) ? keys[i + j * kBucketThreads] : 0u;
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if (i + j * kBucketThreads < end) {
                        const uint32_t x = (key[j] >> 8) & 0xFFu, y = key[j] & 0xFFu;
                        atomicAdd(&sh_cnt[x], 1u);
                        atomicAdd(&sh_y[x], y);
                        atomicAdd(&sh_y2[x], y * y);
                    }
                }
            }
            __syncthreads();
            sh_num[t] += sh_cnt[t];
            sh_sum_y[t] += sh_y[t];
            sh_sum_y2[t] += sh_y2[t];
            sh_cnt[t] = sh_y[t] = sh_y2[t] = 0u;
            __syncthreads();
            i0 = end;
        }
        // running totals over the sub-bins in falling order: thread t takes digit 255 - t
        const uint32_t ex = bk.bin >> 7;
        const uint32_t base = ((bk.bin & 0x7Fu) << 16) | (ex ? 0x800000u : 0u);  // mantissa of the bucket's smallest key
        const uint32_t x = 255u - (uint32_t)t;
        const uint32_t num = sh_num[x];
        {
            const unsigned long long B = base + (x << 8);
            const unsigned __int128 e = (unsigned __int128)num * (B * B) + (unsigned __int128)sh_sum_y[x] * (2ull * B) + sh_sum_y2[x];
            uint32_t inc = num;
            unsigned __int128 ie = e;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t yn = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                const Wide w = wide(ie);
                const Wide yw = {__shfl_up_sync(0xFFFFFFFFu, w.lo, o), __shfl_up_sync(0xFFFFFFFFu, w.hi, o)};
                if (lane >= o) {
                    inc += yn;
                    ie += wide128(yw);
                }
            }
            if (lane == 31) {
                sh_wsum[warp] = inc;
                sh_wenergy[warp] = wide(ie);
            }
            __syncthreads();
            uint32_t before = 0;
            unsigned __int128 ebefore = 0;
            for (int w = 0; w < warp; ++w) {
                before += sh_wsum[w];
                ebefore += wide128(sh_wenergy[w]);
            }
            sh_above[x] = before + inc - num;
            sh_energy[x] = wide(ebefore + ie - e);
            if (t == kBucketThreads - 1) sc.bucket_sum[(int64_t)row * kBins1 + bi] = wide(ebefore + ie);
        }
        __syncthreads();
        // the sub-bin of every boundary: the largest digit with #{keys of the bucket in it or above} >= its rank
        auto sub_bin = [&](uint32_t rank) -> uint32_t {  // 1 <= rank <= count
            uint32_t lo = 0, hi = 255;  // the answer is the largest x with above[x] + num[x] >= rank
            while (lo < hi) {
                const uint32_t mid = (lo + hi + 1) >> 1;
                if (sh_above[mid] + sh_num[mid] >= rank) lo = mid; else hi = mid - 1;
            }
            return lo;
        };
        auto local_rank = [&](uint32_t j) -> uint32_t { return s_len * (j + 1u) - bk.above; };  // s (j + 1) < d < 2^32
        for (uint32_t j = t; j < bk.n; j += kBucketThreads) sh_flag[sub_bin(local_rank(bk.first + j))] = 1u;
        __syncthreads();
        uint32_t marked;
        {  // number the marked sub-bins in falling order
            const uint32_t f = sh_flag[x];
            uint32_t inc = f;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                if (lane >= o) inc += y;
            }
            __syncthreads();
            if (lane == 31) sh_wsum[warp] = inc;
            __syncthreads();
            uint32_t before = 0;
            for (int w = 0; w < warp; ++w) before += sh_wsum[w];
            sh_flag[x] = f ? before + inc - 1u : 0xFFFFFFFFu;
            if (t == kBucketThreads - 1) sh_marked = before + inc;
            __syncthreads();
            marked = sh_marked;
        }
        for (uint32_t g0 = 0; g0 < marked; g0 += kSubBins) {
            const uint32_t here = min((uint32_t)kSubBins, marked - g0);
            for (uint32_t i = t; i < here * 256u; i += kBucketThreads) (&sh_hist[0][0])[i] = 0u;
            __syncthreads();
            for (uint32_t i = t; i < bk.count; i += 4 * kBucketThreads) {
                uint32_t key[4], f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    key[j] = (i + j * kBucketThreads < bk.count) ? keys[i + j * kBucketThreads] : 0u;
                    f[j] = (i + j * kBucketThreads < bk.count) ? sh_flag[(key[j] >> 8) & 0xFFu] - g0 : 0xFFFFFFFFu;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (f[j] < here) atomicAdd(&sh_hist[f[j]][key[j] & 0xFFu], 1u);
            }
            __syncthreads();
            for (uint32_t j = warp; j < bk.n; j += kBucketThreads / 32) {
                const uint32_t rank = local_rank(bk.first + j), xs = sub_bin(rank);
                const uint32_t f = sh_flag[xs] - g0;
                if (f >= here) continue;  // warp-uniform: another group's
                const uint32_t rem = rank - sh_above[xs];
                uint32_t c[8], local = 0;  // lane 0 owns the low bytes 255..248, lane 31 7..0
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    c[i] = sh_hist[f][255 - (lane * 8 + i)];
                    local += c[i];
                }
                uint32_t inc = local;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
                    if (lane >= o) inc += y;
                }
                const bool mine = inc >= rem && inc - local < rem;
                uint32_t y_T = 0, r = 0, run = inc - local;
                unsigned long long n_up = 0, sy = 0, sy2 = 0;  // keys above the threshold in this sub-bin
                bool found = false;
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const uint32_t y = 255u - (uint32_t)(lane * 8 + i);
                    if (mine && !found && run + c[i] >= rem) {
                        found = true;
                        y_T = y;
                        r = rem - run;
                    } else if (!found && run + c[i] < rem) {  // wholly above the boundary (lanes past it never qualify)
                        n_up += c[i];
                        sy += (unsigned long long)c[i] * y;
                        sy2 += (unsigned long long)c[i] * (y * y);
                    }
                    run += c[i];
                }
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    n_up += __shfl_xor_sync(0xFFFFFFFFu, n_up, o);
                    sy += __shfl_xor_sync(0xFFFFFFFFu, sy, o);
                    sy2 += __shfl_xor_sync(0xFFFFFFFFu, sy2, o);
                }
                if (mine) {
                    const unsigned long long B = base + (xs << 8), mt = B + y_T;
                    const unsigned __int128 e = wide128(sh_energy[xs]) + (unsigned __int128)n_up * (B * B) +
                                                (unsigned __int128)sy * (2ull * B) + sy2 + (unsigned __int128)r * (mt * mt);
                    const int64_t at = (int64_t)row * sc.seg_cap + bk.first + j;
                    sc.bound[at] = make_uint2((bk.bin << 16) | (xs << 8) | y_T, r);
                    sc.prefix[at] = wide(e);
                }
            }
            __syncthreads();
        }
        __syncthreads();
    }
}

// Norm of every segment, one warp each.  fp32: the rest of the bucket in which the segment begins, its cells, and the
// part of the bucket in which it ends (or the difference of two boundaries of one bucket).  bf16: the bins it meets.
template <bool BF16>
__global__ void __launch_bounds__(256)
segment_norm_kernel(const uint32_t* hist1 /* bf16: #{key >= b} */, int m0, uint32_t d, uint32_t s_len, uint32_t L, SegScratch sc,
                    const int* worker_err) {
    pdl_enter();
    const int row = blockIdx.y, m = m0 + row, lane = threadIdx.x & 31;
    const uint32_t l = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (l >= L || worker_err[m] || (!BF16 && sc.head[row].sorted)) return;
    double e = 0.0;
    if constexpr (BF16) {
        const uint32_t* S = hist1 + (int64_t)m * kBins1;
        const uint32_t k0 = s_len * l, k1 = (l == L - 1) ? d : s_len * (l + 1);  // ranks (k0, k1]
        auto bin_of = [&](uint32_t k) -> int {  // the largest bin b with #{key >= b} >= k
            int lo = 0, hi = kBins1 - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (S[mid] >= k) lo = mid; else hi = mid - 1;
            }
            return lo;
        };
        const int b0 = bin_of(k0 + 1), b1 = bin_of(k1);
        for (int b = b0 - lane; b >= b1; b -= 32) {
            const uint32_t above = b == kBins1 - 1 ? 0u : S[b + 1], upto = S[b];
            const uint32_t n = min(upto, k1) - max(min(above, k1), k0);
            if (upto > above && n) {
                const double x = (double)__uint_as_float((uint32_t)b << 16);
                e = fma((double)n, x * x, e);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
    } else {
        const uint2 cells = sc.seg_cells[(int64_t)row * sc.seg_cap + l];
        const unsigned long long* cell = sc.cell + (int64_t)row * kMaxCells * 2;
        if (cells.x != 0xFFFFFFFFu)
            for (uint32_t c = cells.x + lane; c < cells.y; c += 32) {
                const unsigned __int128 sum = ((unsigned __int128)cell[c * 2 + 1] << 32) + cell[c * 2];
                e += energy_unit(wide_to_double(sum), sc.cell_exp[(int64_t)row * kMaxCells + c]);
            }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
        if (lane == 0) {
            const int64_t at = (int64_t)row * sc.seg_cap + l;
            const uint16_t* table = sc.table + (int64_t)row * kBins1;
            const uint32_t T_lo = l ? sc.bound[at - 1].x : kKeyNone, T_hi = (l < L - 1) ? sc.bound[at].x : kKeyNone;
            if (T_lo != kKeyNone && T_hi != kKeyNone && (T_lo >> 16) == (T_hi >> 16)) {
                e += energy_unit(wide_to_double(wide128(sc.prefix[at]) - wide128(sc.prefix[at - 1])), (int)(T_hi >> 23));
            } else {
                if (T_lo != kKeyNone) {
                    const uint32_t b = table[T_lo >> 16] & 0x7FFFu;
                    e += energy_unit(wide_to_double(wide128(sc.bucket_sum[(int64_t)row * kBins1 + b]) - wide128(sc.prefix[at - 1])), (int)(T_lo >> 23));
                }
                if (T_hi != kKeyNone) e += energy_unit(wide_to_double(wide128(sc.prefix[at])), (int)(T_hi >> 23));
            }
        }
    }
    if (lane == 0) sc.delta[(int64_t)row * sc.seg_cap + l] = sqrt(e);
}

// p_l = Delta_l / sum Delta (Lemma 3.4), the level draw by the running sums, and the two thresholds of the drawn segment
// as the queries of the header kernel.  One block per row; every thread has a contiguous chunk of the segments.
template <bool BF16>
__global__ void __launch_bounds__(kSegThreads)
segment_draw_kernel(const uint32_t* hist1, int m0, uint32_t d, uint32_t s_len, uint32_t L, SegScratch sc, uint64_t seed,
                    uint64_t step, double* p_all, EmitParams* emit, Query* queries, const int* worker_err) {
    __shared__ double sh_warp[32];
    __shared__ double sh_upto[kSegThreads];
    __shared__ uint32_t sh_first[32], sh_last[32], sh_level;
    pdl_enter();
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int row = blockIdx.x, m = m0 + row;
    if (worker_err[m]) return;
    const double* delta = sc.delta + (int64_t)row * sc.seg_cap;
    const uint32_t per = (L + kSegThreads - 1) / kSegThreads;
    const uint32_t l0 = min((uint32_t)t * per, L), l1 = min(l0 + per, L);
    double part = 0.0;
    uint32_t last = 0;  // 1 + the last level of the chunk with a positive norm
    for (uint32_t l = l0; l < l1; ++l) {
        part += delta[l];
        if (delta[l] > 0.0) last = l + 1;
    }
    double inc = part;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
    }
    if (lane == 31) sh_warp[warp] = inc;
    const uint32_t wlast = __reduce_max_sync(0xFFFFFFFFu, last);
    if (lane == 0) sh_last[warp] = wlast;
    __syncthreads();
    double before_warp = 0.0, total = 0.0;
    for (int w = 0; w < 32; ++w) {
        if (w == warp) before_warp = total;
        total += sh_warp[w];
    }
    const double upto = before_warp + inc;
    sh_upto[t] = upto;
    const double u = counter_uniform(seed, step, (uint64_t)m);
    // l* = min{ l : u < cdf_l }, cdf_l = (Delta_0 + ... + Delta_l) / total: the first chunk whose running sum passes u
    const uint32_t chunk = (part > 0.0 && u < upto / total) ? (uint32_t)t : 0xFFFFFFFFu;
    const uint32_t wfirst = __reduce_min_sync(0xFFFFFFFFu, chunk);
    if (lane == 0) sh_first[warp] = wfirst;
    __syncthreads();
    uint32_t first = __reduce_min_sync(0xFFFFFFFFu, sh_first[lane]);
    const uint32_t last_all = __reduce_max_sync(0xFFFFFFFFu, sh_last[lane]);
    if (t == 0) sh_level = (total > 0.0 && last_all) ? last_all - 1u : 0u;  // if rounding hides the crossing
    __syncthreads();
    if ((uint32_t)t == first) {
        double c = t ? sh_upto[t - 1] : 0.0;
        uint32_t found = last - 1u;
        for (uint32_t l = l0; l < l1; ++l) {
            c += delta[l];
            if (delta[l] > 0.0 && u < c / total) {
                found = l;
                break;
            }
        }
        sh_level = found;
    }
    __syncthreads();
    const uint32_t level = sh_level;
    if (t == 0) {
        p_all[m * kMaxLevels] = (total > 0.0) ? delta[level] / total : 1.0;
        emit[m].level = (int32_t)level;
    }
    if (t < 2) {
        const uint32_t k = t ? ((level == L - 1) ? d : s_len * (level + 1)) : s_len * level;
        Query q = {};
        q.k = k;
        q.slot = kNoSlot;
        q.trivial = (k == 0u) ? 1u : (k >= d ? 2u : 0u);
        if (q.trivial == 1u) {
            q.T = kKeyNone;
        } else if (q.trivial == 2u) {
            q.T = 0u;
            q.r = 0xFFFFFFFFu;
        } else if constexpr (BF16) {
            const uint32_t* S = hist1 + (int64_t)m * kBins1;
            int lo = 0, hi = kBins1 - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (S[mid] >= k) lo = mid; else hi = mid - 1;
            }
            q.T = (uint32_t)lo;
            q.r = k - (lo == kBins1 - 1 ? 0u : S[lo + 1]);
        } else if (sc.head[row].sorted) {
            const uint32_t* keys = sc.sort.a + (int64_t)row * sc.sort.stride;
            const uint32_t at = keys[k - 1u];
            uint32_t lo = 0, hi = k - 1u;  // the first place of that key
            while (lo < hi) {
                const uint32_t mid = lo + (hi - lo) / 2;
                if (keys[mid] < at) lo = mid + 1; else hi = mid;
            }
            q.T = kSortFlip - at;
            q.r = k - lo;
        } else {
            const uint2 b = sc.bound[(int64_t)row * sc.seg_cap + k / s_len - 1u];
            q.T = b.x;
            q.r = b.y;
        }
        queries[m * kMaxQueries + t] = q;
    }
}

struct SegPlanner {
    char* base;
    size_t off = 0;
    template <typename T>
    T* take(size_t n) {
        off = (off + 255) & ~size_t(255);
        T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
        off += n * sizeof(T);
        return p;
    }
};

size_t plan_scratch(char* base, int rows, int64_t d, int64_t seg_cap, SegScratch* sc) {
    SegPlanner pl{base};
    const size_t r = (size_t)rows;
    sc->keys = pl.take<uint32_t>(r * d);
    sc->table = pl.take<uint16_t>(r * kBins1);
    sc->bucket = pl.take<Bucket>(r * kBins1);
    sc->bucket_sum = pl.take<Wide>(r * kBins1);
    sc->cursor = pl.take<uint32_t>(r * kBins1);
    sc->cell = pl.take<unsigned long long>(r * kMaxCells * 2);
    sc->cell_exp = pl.take<uint8_t>(r * kMaxCells);
    sc->seg_cells = pl.take<uint2>(r * seg_cap);
    sc->bound = pl.take<uint2>(r * seg_cap);
    sc->prefix = pl.take<Wide>(r * seg_cap);
    sc->delta = pl.take<double>(r * seg_cap);
    sc->head = pl.take<RowHead>(r);
    const size_t tiles = (size_t)sort_tiles(d), slots = (size_t)sort_slots(d, rows);
    sc->sort.a = sc->keys;
    sc->sort.b = pl.take<uint32_t>(slots * d);
    sc->sort.table = pl.take<uint32_t>(slots * 256 * tiles);
    sc->sort.totals = pl.take<uint32_t>(slots * 256);
    sc->sort.stride = d;
    sc->sort.slots = (int)slots;
    sc->key_stride = d;
    sc->seg_cap = seg_cap;
    return pl.off + 256;
}

// Rows whose scratch memory fits in so many bytes, at least one.
int rows_within(size_t bytes, int most, int64_t d, int64_t L) {
    SegScratch sc;
    int lo = 1, hi = most;
    while (lo < hi) {
        const int mid = lo + (hi - lo + 1) / 2;
        if (plan_scratch(nullptr, mid, d, L, &sc) <= bytes) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

}  // namespace

int configure_segment_kernels() {
    const bool ok =
        cudaFuncSetAttribute(segment_sweep_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSegSweepSmem) == cudaSuccess &&
        cudaFuncSetAttribute(segment_sweep_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSegSweepSmem) == cudaSuccess &&
        cudaFuncSetAttribute(segment_resolve_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBinRowsSmem) == cudaSuccess &&
        cudaFuncSetAttribute(segment_resolve_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBinRowsSmem) == cudaSuccess;
    return ok ? MLMC_OK : MLMC_ERR_CUDA;
}

// Scratch memory, taken at the first call and kept as it is until the context is destroyed: room for as many rows of d_max
// keys and 4096 segments as fit in the budget (at most M_max), and in any case for one row with the most segments.  How many
// rows a call takes together follows from its own d and L.  (It never moves, so that a captured graph keeps valid addresses and
// no later call has to allocate.)
int reserve_segments(Workspace& ws) {
    if (ws.seg_scratch) return MLMC_OK;
    SegScratch sc;
    const int64_t few = std::min(ws.big_cap, (int64_t)4096);
    ws.seg_bytes = std::max(plan_scratch(nullptr, rows_within(kSegScratchBudget, ws.M_max, ws.d_max, few), ws.d_max, few, &sc),
                            plan_scratch(nullptr, 1, ws.d_max, ws.big_cap, &sc));
    if (cudaMalloc(&ws.seg_scratch, ws.seg_bytes) != cudaSuccess) {
        cudaGetLastError();
        ws.seg_scratch = nullptr;
        return MLMC_ERR_NOMEM;
    }
    return MLMC_OK;
}

// Segment norms, the draw and the two queries of every row (hist1 has run).
void launch_segments(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, int64_t s_len, int64_t L,
                     uint64_t seed, uint64_t step, cudaStream_t s) {
    SegScratch sc;
    const int together = rows_within(ws.seg_bytes, M, d, L);
    plan_scratch(static_cast<char*>(ws.seg_scratch), together, d, L, &sc);
    const uint32_t sl = (uint32_t)s_len, nl = (uint32_t)L, du = (uint32_t)d;
    for (int m0 = 0; m0 < M; m0 += together) {
        const int rows = std::min(together, M - m0);
        auto resolve = [&](auto kernel) {
            launch_kernel(ws, K_SEG_RESOLVE, kernel, dim3(rows), kSegThreads, kBinRowsSmem, s, ws.hist1, m0, sort_from(du, rows),
                          std::max(kFewEqual, du / 32), sl, nl, sc, ws.worker_err);
        };
        auto norms = [&](auto norm, auto draw) {
            launch_kernel(ws, K_SEG_NORMS, norm, dim3((nl + 7) / 8, rows), 256, 0, s, ws.hist1, m0, du, sl, nl, sc, ws.worker_err);
            launch_kernel(ws, K_SEG_DRAW, draw, dim3(rows), kSegThreads, 0, s, ws.hist1, m0, du, sl, nl, sc, seed, step, ws.p_all,
                          ws.emit, ws.queries, ws.worker_err);
        };
        if (dtype == MLMC_BF16) {
            resolve(segment_resolve_kernel<true>);
            norms(segment_norm_kernel<true>, segment_draw_kernel<true>);
            continue;
        }
        resolve(segment_resolve_kernel<false>);
        const int64_t by_work = (d + kTripKeys - 1) / kTripKeys;
        const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(by_work, ws.sm_count / rows));
        launch_kernel(ws, K_SEG_SWEEP, L + 255 > kCellWords ? segment_sweep_kernel<true> : segment_sweep_kernel<false>, dim3(nb, rows), kSegThreads, kSegSweepSmem, s,
                      static_cast<const float*>(g), d, ld, m0, sc, ws.worker_err);
        if (d > kFewEqual)  // shorter rows are never sorted
            launch_sorted_rows(ws, static_cast<const float*>(g) + (int64_t)m0 * ld, d, rows, ld, sc.head, sc.sort, sl, nl, sc.delta, sc.seg_cap, s);
        // a block per bucket while there are few; at most as many buckets as boundaries
        const int most = (int)std::min<int64_t>(L - 1, kBins1);
        const int blocks = std::max(1, std::min(most, ws.sm_count * 16 / rows));
        launch_kernel(ws, K_SEG_BUCKETS, bucket_kernel, dim3(blocks, rows), kBucketThreads, 0, s, m0, sl, sc, ws.worker_err);
        norms(segment_norm_kernel<false>, segment_draw_kernel<false>);
    }
}

}  // namespace mlmc
