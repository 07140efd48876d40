// Band emission (ordered stream compaction) and the server-side average for MLMC-Top-k.
//
// emit: writes the band of the drawn level of every worker,
//   { i : k_{l-1} < rank(i) <= k_l },  as (i, g_i / p_l) in ascending i  (Eq. 5 with g^0 = 0; Alg. 2 "Send").
// Membership is decided from the two thresholds (Ta, ra), (Tb, rb) of the band; equal-key elements
// are admitted by their index-ordered rank, so the position of an entry follows from the running counts
//   C = #{ Tb <= key <= Ta },  A = #{ key == Ta },  B = #{ key == Tb }
// over the elements before it.  The row is cut into tiles of kEmitTile 32-bit words, each of kEmitGroups batches;
// only the batches whose largest key (recorded by the first selection sweep) reaches Tb can hold band entries,
// the others are never read.  Three kernels, no waiting between thread blocks:
//   tile_list   one thread per tile: appends the tiles that hold such a batch, with the mask of those batches, to one list
//               of all workers' tiles (its order does not matter);
//   band_count  the warps stride over the list, count C, A, B of every tile and add them to the totals of the item,
//               super-item and hyper-item the tile lies in;
//   band_write  the warps stride over the list again: a tile's position is the sum of the counts before it (hyper-items,
//               super-items, items, tiles: one load per lane each); its entries are written there.
// How much there is to read differs from worker to worker (their levels differ) and from layer to layer; striding over
// the list gives every warp the same share.
//
// aggregate: the dense mean (1/M) sum_m g~_m (Alg. 2 "Server aggregates") tiled over the index
// space; because every message is index-sorted, a tile's entries are one contiguous range per
// worker; they are added into a shared-memory tile in worker order and the tile is written once.
#include <algorithm>
#include <atomic>

#include "topk_band.cuh"

namespace mlmc {

namespace {

constexpr int kBandThreads = 256;               // 8 warps per block, one tile per warp at a time
// Shared-memory batches per warp of the write pass, and blocks per SM.  fp32, three and three / two and four: 16 x 11.7M in layers, level
// 0, 10, 50 and 99 of 100 (a few batches listed to all) 42.5 / 40.7, 56 / 53, 120 / 106, 147 / 132 us; 8 x 124M, 20 levels, level 0, 10,
// 19: 309 / 281, 789 / 737, 843 / 791; 8 x 3M the same (17 to 28).  bf16 has as many entries in half of the batches: 32 x 25.6M 176 / 179,
// 442 / 444, 457 / 457, 8 x 40M 90 / 90, 187 / 186, 199 / 198, and the steps of 8 x 3M become 5 to 8 % longer (75 / 81).
template <typename T>
constexpr int kWriteSlots = EmitWord<T>::S == 1 ? 2 : 3;
template <typename T>
constexpr int kWriteBlocks = EmitWord<T>::S == 1 ? 4 : 3;
// words of shared memory per warp of the write pass: the batches and the offsets of one batch's entries
template <typename T>
constexpr int kWriteWords = kWriteSlots<T> * kEmitRows * 32 + kEmitRows * 32 * EmitWord<T>::S / 2;

// Where a tile's counts are added up: {C, A, B, batches} per item, super-item and hyper-item of every worker.
struct CountLevels {
    uint4 *items, *supers, *hypers;
    int n_items, n_supers, n_hypers;  // per worker
};

// A batch whose largest key is below the lower threshold Tb of the drawn band holds no band entry and no tie of Tb either;
// it is not read.  List entry: {worker << kTileBits | tile, mask of the batches to read}.
__global__ void __launch_bounds__(kBandThreads)
tile_list_kernel(const uint32_t* tile_max, int tiles_per_worker, const EmitParams* emit, uint32_t key_cap, uint4* tiles,
                 uint2* list, uint32_t* list_n) {
    pdl_enter();
    const int m = blockIdx.y, t = blockIdx.x * kBandThreads + threadIdx.x, lane = threadIdx.x & 31;
    uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
    const bool inside = t < tiles_per_worker;
    if (inside) {  // the batch maxima of a tile are two 16-byte vectors
        const uint4* mx = reinterpret_cast<const uint4*>(tile_max) + ((int64_t)m * tiles_per_worker + t) * 2;
        a = mx[0];
        b = mx[1];
    }
    const EmitParams e = emit[m];
    const uint32_t Tb = min(e.Tb, key_cap);
    uint32_t mask = 0;
    if (inside && e.enabled && e.level >= 0 && e.expect > 0u)
        mask = (a.x >= Tb ? 1u : 0u) | (a.y >= Tb ? 2u : 0u) | (a.z >= Tb ? 4u : 0u) | (a.w >= Tb ? 8u : 0u) |
               (b.x >= Tb ? 16u : 0u) | (b.y >= Tb ? 32u : 0u) | (b.z >= Tb ? 64u : 0u) | (b.w >= Tb ? 128u : 0u);
    const uint32_t listed = __ballot_sync(0xFFFFFFFFu, mask != 0u);
    uint32_t base = 0;
    if (lane == 0 && listed) base = atomicAdd(list_n, (uint32_t)__popc(listed));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (mask) list[base + __popc(listed & ((1u << lane) - 1u))] = make_uint2(((uint32_t)m << kTileBits) | (uint32_t)t, mask);
    else if (inside) tiles[(int64_t)m * tiles_per_worker + t] = make_uint4(0u, 0u, 0u, 0u);
}

// Pass 1: tiles[m][t] = {C, A, B, tie flag} of every tile (the tie flag: the tile holds a key equal to a threshold).
// A warp walks the batches of its tiles as one sequence, the next batch in flight while the current one is counted.
template <typename T>
__global__ void __launch_bounds__(kBandThreads)
band_count_kernel(const T* __restrict__ g, int64_t d, int64_t ld, int tiles_per_worker, int M, const EmitParams* emit,
                  uint4* tiles, CountLevels lv, const uint2* list, const uint32_t* list_n) {
    using EW = EmitWord<T>;
    extern __shared__ uint2 sh_thr[];  // [M] {Tb, Ta}
    pdl_enter();
    for (int m = threadIdx.x; m < M; m += kBandThreads) sh_thr[m] = make_uint2(min(emit[m].Tb, EW::kCap), min(emit[m].Ta, EW::kCap));
    const uint32_t total = *list_n;
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t warps = gridDim.x * (kBandThreads / 32);
    uint32_t f = blockIdx.x * (kBandThreads / 32) + (threadIdx.x >> 5);
    if (f >= total) return;
    uint2 here = list[f], next = make_uint2(0u, 0u);
    if (f + warps < total) next = list[f + warps];
    uint32_t todo = here.y, cC = 0, cA = 0, cB = 0, batches = 0;
    uint32_t cur[kEmitRows], nxt[kEmitRows];
    auto load = [&](const uint2& e, uint32_t& left, uint32_t (&w)[kEmitRows]) {
        load_batch<T>(g + (int64_t)(e.x >> kTileBits) * ld, d, e.x & ((1u << kTileBits) - 1u), __ffs(left) - 1, lane, w);
        left &= left - 1u;
    };
    load(here, todo, cur);
#pragma unroll 1
    for (;;) {
        const bool last = todo == 0u, more = f + warps < total;  // last batch of the tile; another tile follows
        uint32_t todo_next = next.y;
        if (!last) load(here, todo, nxt);
        else if (more) load(next, todo_next, nxt);
        const int m = (int)(here.x >> kTileBits);
        const uint2 thr = sh_thr[m];
        uint32_t a1, b1;
        const uint32_t flags = batch_flags<T>(cur, thr.x, thr.y, &a1, &b1);
        cC += __popc(flags);
        cA += a1;
        cB += b1;
        ++batches;
        if (last) {
            const uint32_t totCA = __reduce_add_sync(0xFFFFFFFFu, cC | (cA << 16));  // at most 8192 elements per tile
            const uint32_t tB = __reduce_add_sync(0xFFFFFFFFu, cB);
            const uint32_t tC = totCA & 0xFFFFu, tA = totCA >> 16;
            const int tile = (int)(here.x & ((1u << kTileBits) - 1u));
            if (lane == 31) tiles[(int64_t)m * tiles_per_worker + tile] = make_uint4(tC, tA, tB, (tA | tB) ? 1u : 0u);
            if (lane < 12) {  // three levels of four components
                const int item = tile / kItemTiles, sup = item / kSuperItems, c = lane & 3;
                uint4* rec = lane < 4 ? lv.items + (int64_t)m * lv.n_items + item
                           : lane < 8 ? lv.supers + (int64_t)m * lv.n_supers + sup
                                      : lv.hypers + (int64_t)m * lv.n_hypers + sup / kSuperItems;
                const uint32_t x = c == 0 ? tC : c == 1 ? tA : c == 2 ? tB : batches;
                if (x) atomicAdd(reinterpret_cast<uint32_t*>(rec) + c, x);
            }
            if (!more) return;
            cC = cA = cB = batches = 0u;
            here = next;
            todo = todo_next;
            f += warps;
            if (f + warps < total) next = list[f + warps];
        }
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i) cur[i] = nxt[i];
    }
}

// Pass 2: every listed tile is read again and its band entries are written at their final positions.
template <typename T>
__global__ void __launch_bounds__(kBandThreads, kWriteBlocks<T>)
band_write_kernel(const T* __restrict__ g, int64_t d, int64_t ld, int tiles_per_worker, int M, const EmitParams* emit,
                  const uint4* tiles, CountLevels lv, const uint2* list, const uint32_t* list_n,
                  uint32_t* __restrict__ idx_out, float* __restrict__ val_out, int64_t capacity, uint32_t* group_n,
                  int* status) {
    using EW = EmitWord<T>;
    constexpr int S = EW::S;
    // every warp stages its batches in a ring of shared-memory slots: the next copies are in flight while a batch is ranked, and the
    // words of a batch can be addressed by a run-time index
    extern __shared__ __align__(16) uint32_t sh_dyn[];  // [warps][kWriteWords]
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int warps = gridDim.x * (kBandThreads / 32), gw = blockIdx.x * (kBandThreads / 32) + (threadIdx.x >> 5);
    // the band of every worker has exactly k_l - k_{l-1} entries, and they lie in some batch
    for (int m = gw; m < M; m += warps) {
        uint4 x = make_uint4(0u, 0u, 0u, 0u);
        for (int i = lane; i < lv.n_hypers; i += 32) {
            const uint4 y = lv.hypers[(int64_t)m * lv.n_hypers + i];
            x.x += y.x; x.y += y.y; x.z += y.z; x.w += y.w;
        }
        x.x = __reduce_add_sync(0xFFFFFFFFu, x.x);
        x.y = __reduce_add_sync(0xFFFFFFFFu, x.y);
        x.z = __reduce_add_sync(0xFFFFFFFFu, x.z);
        x.w = __reduce_add_sync(0xFFFFFFFFu, x.w);
        if (lane == 0) {
            const EmitParams e = emit[m];
            group_n[m] = x.w;
            if (e.enabled && e.level >= 0 && e.expect > 0u && (x.w == 0u || band_prefix(x.x, x.y, x.z, e.ra, e.rb) != e.expect))
                set_status(status, MLMC_ERR_INTERNAL);
        }
    }
    const uint32_t total = *list_n;
    uint32_t* ring = sh_dyn + (threadIdx.x >> 5) * kWriteWords<T>;
    uint16_t* stage = reinterpret_cast<uint16_t*>(ring + kWriteSlots<T> * kBatchWords);
    uint2 next = gw < (int)total ? list[gw] : make_uint2(0u, 0u);
    for (uint32_t f = gw; f < total; f += warps) {
        const uint2 entry = next;
        if (f + warps < total) next = list[f + warps];
        const int m = (int)(entry.x >> kTileBits);
        const int64_t tile = entry.x & ((1u << kTileBits) - 1u);
        const EmitParams ep = emit[m];
        const uint32_t flags = tiles[(int64_t)m * tiles_per_worker + tile].w;
        uint4 before = make_uint4(0u, 0u, 0u, 0u);  // counts before this tile
        {
            const int item = (int)tile / kItemTiles, sup = item / kSuperItems, hyp = sup / kSuperItems;
            auto add = [&](const uint4& x) { before.x += x.x; before.y += x.y; before.z += x.z; };
            if (lane < (int)tile % kItemTiles) add(tiles[(int64_t)m * tiles_per_worker + item * kItemTiles + lane]);
            if (lane < item % kSuperItems) add(lv.items[(int64_t)m * lv.n_items + sup * kSuperItems + lane]);
            if (lane < sup % kSuperItems) add(lv.supers[(int64_t)m * lv.n_supers + hyp * kSuperItems + lane]);
            for (int i = lane; i < hyp; i += 32) add(lv.hypers[(int64_t)m * lv.n_hypers + i]);
            before.x = __reduce_add_sync(0xFFFFFFFFu, before.x);
            before.y = __reduce_add_sync(0xFFFFFFFFu, before.y);
            before.z = __reduce_add_sync(0xFFFFFFFFu, before.z);
        }
        const Band band = {min(ep.Tb, EW::kCap), min(ep.Ta, EW::kCap), ep.ra, ep.rb, (float)ep.inv_p};
        const T* row = g + (int64_t)m * ld;
        uint32_t* idx_w = idx_out + (int64_t)m * capacity;
        float* val_w = val_out + (int64_t)m * capacity;
        uint3 run = make_uint3(before.x, before.y, before.z);  // running totals before the current batch
        const bool tile_ties = flags != 0u;           // found by the count pass
        // Only the batches of the tile that can hold band entries are read (mask from the listing): `todo` walks them
        // for processing, `ahead` two batches further for the copies.
        uint32_t todo = entry.y, ahead = todo;
        __syncwarp();  // the previous tile's last batches have been read by every lane
        copy_batch_async<T>(row, d, tile, __ffs(ahead) - 1, lane, ring);
        ahead &= ahead - 1u;
        cp_async_commit();
        if (ahead) {
            copy_batch_async<T>(row, d, tile, __ffs(ahead) - 1, lane, ring + kBatchWords);
            ahead &= ahead - 1u;
        }
        cp_async_commit();
#pragma unroll 1
        for (int it = 0; todo; ++it) {
            const int b = __ffs(todo) - 1;
            todo &= todo - 1u;
            auto copy_two_ahead = [&]() {  // into a slot whose batch has been read by every lane
                __syncwarp();
                if (ahead) {
                    copy_batch_async<T>(row, d, tile, __ffs(ahead) - 1, lane, ring + ((it + 2) % kWriteSlots<T>) * kBatchWords);
                    ahead &= ahead - 1u;
                }
                cp_async_commit();  // one group per step, empty at the end of the tile
            };
            if (kWriteSlots<T> == 3) copy_two_ahead();
            cp_async_wait<kWriteSlots<T> == 3 ? 2 : 1>();  // this batch has landed
            __syncwarp();
            const uint32_t e0 = (uint32_t)((tile * kEmitTile + (int64_t)b * kBatchWords) * S);
            emit_batch<T>(ring + (it % kWriteSlots<T>) * kBatchWords, stage, band, tile_ties, e0, run, idx_w, val_w, capacity);
            if (kWriteSlots<T> == 2) copy_two_ahead();
        }
    }
    cp_async_wait<0>();
}

// Entries of worker m's message; a voided one, or a count below 0, has none.
__device__ __forceinline__ uint32_t message_entries(const int64_t* count, const int32_t* level, int m) {
    return level[m] < 0 ? 0u : (uint32_t)max(count[m], (int64_t)0);
}

// First of the n entries of an index-sorted list that is not below `target`, by 2^lanes_log2 neighbouring lanes (of a warp that is here
// with all its lanes): of the entries that are left, every lane looks at the first of its share.  One lane: halves.
__device__ __forceinline__ uint32_t first_not_below(const uint32_t* __restrict__ a, uint32_t n, uint64_t target, int lanes_log2) {
    const int lane = threadIdx.x & 31, part = lane & ((1 << lanes_log2) - 1);
    uint32_t lo = 0, hi = n;
    if (lanes_log2 == 0) {
        while (lo < hi) {
            const uint32_t mid = lo + ((hi - lo) >> 1);
            if ((uint64_t)__ldg(&a[mid]) < target) lo = mid + 1u; else hi = mid;
        }
        return lo;
    }
    while (__any_sync(0xFFFFFFFFu, lo < hi)) {
        const uint32_t left = hi - lo;  // wraps where the search has ended: that lane looks at nothing
        auto place = [&](uint32_t l) { return lo + (uint32_t)(((uint64_t)left * l) >> lanes_log2); };
        const bool below = lo < hi && (uint64_t)__ldg(&a[place((uint32_t)part)]) < target;
        const uint32_t votes = __ballot_sync(0xFFFFFFFFu, below) >> (lane - part);
        const uint32_t c = (uint32_t)__popc(lanes_log2 == 5 ? votes : votes & ((1u << (1 << lanes_log2)) - 1u));
        if (lo < hi) {
            const uint32_t from = c ? place(c - 1u) + 1u : lo, to = c == 0u ? lo : c >> lanes_log2 ? hi : place(c);
            lo = from;
            hi = to;
        }
    }
    return lo;
}

// offsets[m][t] = first message entry of worker m whose index is >= t * kAggTile  (t = 0..ntiles), by 2^lanes_log2 lanes each: four
// take half as many loads one after the other (8 x 3M 12.6 us, now 10.5), one where so many searches are bound by their loads
// (8 x 124M 18 us, with two lanes 26).
constexpr int64_t kFewOffsets = 1 << 17;
inline int offset_lanes(int64_t n_off) { return n_off <= kFewOffsets ? 2 : 0; }
__global__ void __launch_bounds__(256)
agg_offsets_kernel(const uint32_t* idx, const int64_t* count, const int32_t* level, int64_t capacity, int M, int ntiles, int lanes_log2,
                   uint32_t* offsets) {
    pdl_enter();
    const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> lanes_log2;
    const bool there = i < (int64_t)M * (ntiles + 1);
    const int m = there ? (int)(i / (ntiles + 1)) : 0, t = there ? (int)(i % (ntiles + 1)) : 0;
    const uint32_t n = there ? message_entries(count, level, m) : 0u;
    const uint32_t at = first_not_below(idx + (int64_t)m * capacity, n, (uint64_t)t * kAggTile, lanes_log2);
    if (there && (threadIdx.x & ((1 << lanes_log2) - 1)) == 0) offsets[i] = at;
}
inline unsigned offset_blocks(int64_t n_off) { return (unsigned)(((n_off << offset_lanes(n_off)) + 255) / 256); }

// M is at most kEmitMaxWorkers: the offsets of all workers for one tile are fetched together.
__global__ void __launch_bounds__(256)
aggregate_topk_kernel(const uint32_t* __restrict__ idx, const float* __restrict__ val, int64_t capacity, int M,
                      int64_t d, int ntiles, const uint32_t* offsets, float* __restrict__ out) {
    pdl_enter();
    __shared__ __align__(16) float acc[kAggTile];
    extern __shared__ uint32_t sh_off[];  // [2 M]: first and one-past-last message entry of every worker in this tile
    const float inv_M = 1.0f / (float)M;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t base = (int64_t)t * kAggTile;
        for (int i = threadIdx.x; i < 2 * M; i += blockDim.x)
            sh_off[i] = offsets[(int64_t)(i >> 1) * (ntiles + 1) + t + (i & 1)];
        for (int i = threadIdx.x; i < kAggTile / 4; i += blockDim.x)
            reinterpret_cast<float4*>(acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncthreads();
        for (int m = 0; m < M; ++m) {  // fixed worker order: reproducible fp32 sums
            const uint32_t o0 = sh_off[2 * m], o1 = sh_off[2 * m + 1];
            if (o1 > o0) {  // block-uniform
                const uint32_t* a = idx + (int64_t)m * capacity;
                const float* v = val + (int64_t)m * capacity;
                for (uint32_t j = o0 + threadIdx.x; j < o1; j += blockDim.x) {
                    const uint32_t off = a[j] - (uint32_t)base;  // indices are unique within a worker
                    if (off < (uint32_t)kAggTile) acc[off] += v[j];  // a message that is not index-sorted cannot reach outside the tile
                }
                __syncthreads();
            }
        }
        if (base + kAggTile <= d && reinterpret_cast<uintptr_t>(out) % 16 == 0) {
            for (int i = threadIdx.x; i < kAggTile / 4; i += blockDim.x) {
                float4 x = reinterpret_cast<const float4*>(acc)[i];
                x.x *= inv_M; x.y *= inv_M; x.z *= inv_M; x.w *= inv_M;
                reinterpret_cast<float4*>(out + base)[i] = x;
            }
        } else {
            for (int i = threadIdx.x; i < kAggTile; i += blockDim.x)
                if (base + i < d) out[base + i] = acc[i] * inv_M;
        }
        __syncthreads();
    }
}


// The same average without a block barrier per worker: every warp owns kAggSub consecutive coordinates of the
// tile and adds the workers' entries that fall into them in worker order 0..M-1 (the order of the fp32 additions per
// coordinate is the same as in the kernel above, so the two give identical results).  Lane l finds, for worker
// m0 + l, where the warp's coordinates begin and end inside that worker's slice of the tile (two binary searches in
// an index-sorted slice); the warp then walks the workers one after the other.
// Bound by the latency of the entries while a worker's were added before the next one's were asked for (205 us for 32 x
// 25.6M coordinates, 84 us for 3 x 22.6M dense ones); with the next chunk in flight 143 and 45 us.  Chunks of 64 entries:
// 128 cost registers and blocks per SM (137 -> 151 us on the sparse messages of 8 x 124M coordinates, with 64: 127).
constexpr int kAggSub = 512;
constexpr int kAggWarps = kAggTile / kAggSub;
constexpr int kChunk = 2;

__global__ void __launch_bounds__(kAggWarps * 32)
aggregate_topk_warps_kernel(const uint32_t* __restrict__ idx, const float* __restrict__ val, int64_t capacity, int M,
                            int64_t d, int ntiles, const uint32_t* offsets, float* __restrict__ out) {
    pdl_enter();
    __shared__ __align__(16) float acc_all[kAggTile];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    float* acc = acc_all + warp * kAggSub;
    const float inv_M = 1.0f / (float)M;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t base = (int64_t)t * kAggTile + (int64_t)warp * kAggSub;  // first coordinate of this warp
#pragma unroll
        for (int i = 0; i < kAggSub / 128; ++i)
            reinterpret_cast<float4*>(acc)[i * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
        __syncwarp();
        if (base < d) {
            for (int m0 = 0; m0 < M; m0 += 32) {
                const int m = m0 + lane;
                uint32_t s0 = 0, s1 = 0;
                if (m < M) {
                    const uint32_t o0 = offsets[(int64_t)m * (ntiles + 1) + t], o1 = offsets[(int64_t)m * (ntiles + 1) + t + 1];
                    const uint32_t* a = idx + (int64_t)m * capacity;
                    auto first_at_least = [&](uint64_t target) -> uint32_t {
                        uint32_t lo = o0, hi = o1;
                        while (lo < hi) {
                            const uint32_t mid = lo + ((hi - lo) >> 1);
                            if ((uint64_t)__ldg(&a[mid]) < target) lo = mid + 1; else hi = mid;
                        }
                        return lo;
                    };
                    s0 = (warp == 0) ? o0 : first_at_least((uint64_t)base);
                    s1 = (warp == kAggWarps - 1) ? o1 : first_at_least((uint64_t)base + kAggSub);
                }
                // The entries in chunks of 32 kChunk, worker by worker (fixed order: reproducible fp32 sums); the next chunk is
                // in flight while one is added.  A chunk's missing entries lie outside the warp's coordinates.
                uint32_t live = __ballot_sync(0xFFFFFFFFu, s1 > s0);
                uint32_t at = 0, end = 0, off[kChunk];
                float v[kChunk];
                const uint32_t* a = idx;
                const float* x = val;
                auto fetch = [&](uint32_t (&o)[kChunk], float (&y)[kChunk]) -> bool {  // the next chunk, if there is one
                    if (at >= end) {
                        if (!live) return false;
                        const int mm = __ffs(live) - 1;
                        live &= live - 1u;
                        at = __shfl_sync(0xFFFFFFFFu, s0, mm);
                        end = __shfl_sync(0xFFFFFFFFu, s1, mm);
                        a = idx + (int64_t)(m0 + mm) * capacity;
                        x = val + (int64_t)(m0 + mm) * capacity;
                    }
#pragma unroll
                    for (int k = 0; k < kChunk; ++k) {
                        const uint32_t j = k * 32 + lane;
                        o[k] = j < end - at ? __ldg(&a[at + j]) : (uint32_t)base - 1u;
                        y[k] = j < end - at ? __ldg(&x[at + j]) : 0.0f;
                    }
                    at += min((uint32_t)kChunk * 32u, end - at);
                    return true;
                };
                bool more = fetch(off, v);
                while (more) {
                    uint32_t off_n[kChunk];
                    float v_n[kChunk];
                    more = fetch(off_n, v_n);
#pragma unroll
                    for (int k = 0; k < kChunk; ++k) {
                        const uint32_t o = off[k] - (uint32_t)base;      // indices are unique within a worker
                        if (o < (uint32_t)kAggSub) acc[o] += v[k];       // an unsorted message cannot reach outside
                        off[k] = off_n[k];
                        v[k] = v_n[k];
                    }
                    __syncwarp();
                }
            }
        }
        if (base + kAggSub <= d && reinterpret_cast<uintptr_t>(out) % 16 == 0) {
#pragma unroll
            for (int i = 0; i < kAggSub / 128; ++i) {
                float4 x = reinterpret_cast<const float4*>(acc)[i * 32 + lane];
                x.x *= inv_M; x.y *= inv_M; x.z *= inv_M; x.w *= inv_M;
                reinterpret_cast<float4*>(out + base)[i * 32 + lane] = x;
            }
        } else {
            for (int i = lane; i < kAggSub; i += 32)
                if (base + i < d) out[base + i] = acc[i] * inv_M;
        }
        __syncwarp();
    }
}

// The same average in one launch for short vectors: a block finds its TILE coordinates in every message by itself, some lanes
// per edge, and adds the entries worker after worker with all threads, the next worker's on their way meanwhile.  Bound by
// latency: the searches are 3 to 8 loads one after the other (a thread per edge: up to 15), and tiles of 1024 spread short vectors over
// more SMs.  us per step of 8 x 1M fp32 entries (ten kernels before it) 69.3, now 64.7, 4 x 262,145 54.9, now 51.5.
constexpr int kDirectThreads = 256;
constexpr int kDirectMost = 32;    // workers
constexpr int kDirectEntries = 2;  // per thread and trip

template <int TILE>
__global__ void __launch_bounds__(kDirectThreads)
aggregate_topk_direct_kernel(const uint32_t* __restrict__ idx, const float* __restrict__ val, const int64_t* count,
                             const int32_t* level, int64_t capacity, int M, int lanes_log2, int64_t d, float* __restrict__ out) {
    __shared__ __align__(16) float acc[TILE];
    __shared__ uint32_t sh_edge[2 * kDirectMost];  // first entry of a worker in the tile, and one past its last
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const int64_t base = (int64_t)blockIdx.x * TILE;
    {   // an edge is the first entry that is not below its coordinate
        const int edge = threadIdx.x >> lanes_log2, m = edge >> 1, part = threadIdx.x & ((1 << lanes_log2) - 1);
        const uint64_t target = (uint64_t)base + (edge & 1 ? TILE : 0);
        const uint32_t n = m < M ? message_entries(count, level, m) : 0u;
        const uint32_t at = first_not_below(idx + (int64_t)(m < M ? m : 0) * capacity, n, target, lanes_log2);
        if (part == 0 && m < M) sh_edge[edge] = at;
    }
    for (int i = threadIdx.x; i < TILE / 4; i += kDirectThreads) reinterpret_cast<float4*>(acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    uint32_t off[kDirectEntries];
    float v[kDirectEntries];
    int m = -1;
    uint32_t at = 0, end = 0;
    auto fetch = [&]() -> bool {  // the next entries, worker after worker; all of one worker's lie at different coordinates
        while (at >= end) {
            if (++m >= M) return false;
            at = sh_edge[2 * m];
            end = sh_edge[2 * m + 1];
        }
        const int64_t row = (int64_t)m * capacity;
#pragma unroll
        for (int i = 0; i < kDirectEntries; ++i) {
            const uint32_t j = threadIdx.x + i * kDirectThreads;
            const bool there = j < end - at;
            off[i] = there ? __ldg(&idx[row + at + j]) - (uint32_t)base : 0xFFFFFFFFu;
            v[i] = there ? __ldg(&val[row + at + j]) : 0.0f;
        }
        at += min((uint32_t)(kDirectEntries * kDirectThreads), end - at);
        return true;
    };
    const float inv_M = 1.0f / (float)M;
    bool more = fetch();
    int of = m;
    while (more) {  // block-uniform; fixed worker order: reproducible fp32 sums
        uint32_t o[kDirectEntries];
        float x[kDirectEntries];
#pragma unroll
        for (int i = 0; i < kDirectEntries; ++i) {
            o[i] = off[i];
            x[i] = v[i];
        }
        more = fetch();
#pragma unroll
        for (int i = 0; i < kDirectEntries; ++i)
            if (o[i] < (uint32_t)TILE) acc[o[i]] += x[i];  // an unsorted message cannot reach outside
        if (m != of) __syncthreads();
        of = m;
    }
    __syncthreads();
    if (base + TILE <= d && reinterpret_cast<uintptr_t>(out) % 16 == 0) {
        for (int i = threadIdx.x; i < TILE / 4; i += kDirectThreads) {
            float4 x = reinterpret_cast<const float4*>(acc)[i];
            x.x *= inv_M; x.y *= inv_M; x.z *= inv_M; x.w *= inv_M;
            reinterpret_cast<float4*>(out + base)[i] = x;
        }
    } else {
        for (int i = threadIdx.x; i < TILE; i += kDirectThreads)
            if (base + i < d) out[base + i] = acc[i] * inv_M;
    }
}

}  // namespace

int configure_emit_kernels() {
    auto set = [](auto kernel, int words) {
        return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (kBandThreads / 32) * words * (int)sizeof(uint32_t)) == cudaSuccess;
    };
    return set(band_write_kernel<float>, kWriteWords<float>) && set(band_write_kernel<bf16_t>, kWriteWords<bf16_t>) ? MLMC_OK
                                                                                                                   : MLMC_ERR_CUDA;
}

void emit_limits(KernelLimits* limits) {
    limits->band_count[0] = resident_blocks(band_count_kernel<float>, kBandThreads, 256);
    limits->band_count[1] = resident_blocks(band_count_kernel<bf16_t>, kBandThreads, 256);
    limits->aggregate_topk = resident_blocks(aggregate_topk_warps_kernel, kAggWarps * 32, 0);
}

namespace {

template <typename T>
void launch_emit_t(Workspace& ws, const T* g, int dtype, int64_t d, int M, int64_t ld, const mlmc_topk_msgs& out,
                   cudaStream_t s) {
    const int tpw = emit_tiles_per_worker(d, dtype);
    const EmitCounts n = emit_counts(tpw);
    const CountLevels lv = {ws.level_desc, ws.level_desc + (int64_t)M * n.items, ws.level_desc + (int64_t)M * (n.items + n.supers),
                            n.items, n.supers, n.hypers};
    const int wpb = kBandThreads / 32;
    const size_t smem_w = (size_t)wpb * kWriteWords<T> * sizeof(uint32_t);
    ws.last_emit_tiles = tpw;
    launch_kernel(ws, K_TILE_LIST, tile_list_kernel, dim3((tpw + kBandThreads - 1) / kBandThreads, M), kBandThreads, 0, s,
                  ws.tile_max, tpw, ws.emit, EmitWord<T>::kCap, ws.tile_desc, ws.tile_list, ws.list_n);
    // two whole waves: the warps stride over the list, so a partial last wave costs a full one
    const int resident = ws.limits.band_count[dtype == MLMC_BF16];
    const int64_t by_work = ((int64_t)tpw * M + wpb - 1) / wpb;
    auto blocks = [&](int per_sm) { return (unsigned)std::min<int64_t>(by_work, (int64_t)ws.sm_count * per_sm * 2); };
    launch_kernel(ws, K_BAND_COUNT, band_count_kernel<T>, dim3(blocks(resident)), kBandThreads, (size_t)M * sizeof(uint2), s, g, d,
                  ld, tpw, M, ws.emit, ws.tile_desc, lv, ws.tile_list, ws.list_n);
    launch_kernel(ws, K_EMIT, band_write_kernel<T>, dim3(blocks(kWriteBlocks<T>)), kBandThreads, smem_w, s, g, d, ld, tpw, M, ws.emit,
                  ws.tile_desc, lv, ws.tile_list, ws.list_n, out.idx, out.val, out.capacity, ws.group_n, ws.status);
}

}  // namespace

void launch_emit(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const mlmc_topk_msgs& out,
                 cudaStream_t s) {
    if (dtype == MLMC_BF16) launch_emit_t(ws, static_cast<const bf16_t*>(g), dtype, d, M, ld, out, s);
    else launch_emit_t(ws, static_cast<const float*>(g), dtype, d, M, ld, out, s);
}

void launch_aggregate_topk(Workspace& ws, const mlmc_topk_msgs& msgs, int M, int64_t d, float* out, cudaStream_t s) {
    const int ntiles = (int)((d + kAggTile - 1) / kAggTile);
    if (M <= kDirectMost && ntiles <= ws.sm_count * 4) {  // half a wave of blocks: one launch instead of two, a few us of searches
        int lanes_log2 = 5;  // per edge
        while ((2 * M) << lanes_log2 > kDirectThreads) --lanes_log2;
        auto go = [&](auto kernel, int tile) {
            launch_kernel(ws, K_AGG_TOPK, kernel, dim3((unsigned)((d + tile - 1) / tile)), kDirectThreads, 0, s, msgs.idx, msgs.val, msgs.count,
                          msgs.level, msgs.capacity, M, lanes_log2, d, out);
        };
        if (ntiles <= ws.sm_count * 2) go(aggregate_topk_direct_kernel<kAggTile / 4>, kAggTile / 4);
        else go(aggregate_topk_direct_kernel<kAggTile>, kAggTile);
        return;
    }
    const int64_t n_off = (int64_t)M * (ntiles + 1);
    launch_kernel(ws, K_AGG_OFFSETS, agg_offsets_kernel, dim3(offset_blocks(n_off)), 256, 0, s, msgs.idx, msgs.count,
                  msgs.level, msgs.capacity, M, ntiles, offset_lanes(n_off), ws.agg_offsets);
    const int grid = std::min(ntiles, ws.sm_count * ws.limits.aggregate_topk);
    launch_kernel(ws, K_AGG_TOPK, aggregate_topk_warps_kernel, dim3(grid), kAggWarps * 32, 0, s, msgs.idx, msgs.val,
                  msgs.capacity, M, d, ntiles, ws.agg_offsets, out);
}

}  // namespace mlmc

// ---------------------------------------------------------------------------------------------
// Server average of Top-k messages without any allocation.
// ---------------------------------------------------------------------------------------------
// The tile offsets that the averaging kernel needs normally live in the context's workspace, which
// mlmc_create obtains with cudaMalloc.  Here they live in a file-scope device array of fixed size,
// which every GPU that loads this library holds until the process exits.
namespace mlmc {
namespace {

constexpr int64_t kStaticOffsetWords = int64_t(1) << 20;  // 4 MiB: M * (ceil(d / kAggTile) + 1) entries at most
static __device__ __align__(256) uint32_t g_static_offsets[kStaticOffsetWords];

constexpr int kMaxDevices = 64;
// Device address of the array on each device, 0 = not looked up yet.  Host threads may make their first call on a
// device at the same time: the SM count is written first and the address is published last with a release store,
// so a thread that sees the address (acquire load) also sees the count.  Two threads that both find 0 look the
// same values up twice, which is harmless.
std::atomic<uint32_t*> g_static_offsets_addr[kMaxDevices];
int g_static_sm_count[kMaxDevices];

}  // namespace
}  // namespace mlmc

extern "C" int mlmc_aggregate_topk_noalloc(const mlmc_topk_msgs* msgs, int M, int64_t d, float* out, void* stream) {
    using namespace mlmc;
    if (!msgs || !out || !msgs->idx || !msgs->val || !msgs->count || !msgs->level) return MLMC_ERR_ARG;
    if (M < 1 || M > kEmitMaxWorkers || d < 1 || d >= (int64_t(1) << 32) || msgs->capacity < 0) return MLMC_ERR_ARG;
    const int64_t ntiles = (d + kAggTile - 1) / kAggTile;
    const int64_t n_off = (int64_t)M * (ntiles + 1);
    if (n_off > kStaticOffsetWords) return MLMC_ERR_ARG;  // beyond the fixed scratch: use mlmc_aggregate with a context
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return MLMC_ERR_CUDA;
    uint32_t* offsets = g_static_offsets_addr[dev].load(std::memory_order_acquire);
    if (!offsets) {
        // Set-up, once per device, with that device current.  In host code the array's name only stands
        // for the symbol; the address a kernel can use has to be asked for.
        uint32_t* p = nullptr;
        if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_static_offsets) != cudaSuccess || !p) {
            cudaGetLastError();
            return MLMC_ERR_CUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
            return MLMC_ERR_CUDA;
        g_static_sm_count[dev] = sms;
        g_static_offsets_addr[dev].store(p, std::memory_order_release);
        offsets = p;
    }
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    // every entry in [0, n_off) is rewritten by this kernel, so nothing is left over from an earlier call
    agg_offsets_kernel<<<offset_blocks(n_off), 256, 0, s>>>(msgs->idx, msgs->count, msgs->level,
                                                                       msgs->capacity, M, (int)ntiles, offset_lanes(n_off), offsets);
    int64_t grid = (int64_t)g_static_sm_count[dev] * 8;
    if (grid > ntiles) grid = ntiles;
    aggregate_topk_kernel<<<(unsigned)grid, 256, 2 * M * sizeof(uint32_t), s>>>(msgs->idx, msgs->val, msgs->capacity, M, d,
                                                                                (int)ntiles, offsets, out);
    return cudaGetLastError() == cudaSuccess ? MLMC_OK : MLMC_ERR_CUDA;
}
