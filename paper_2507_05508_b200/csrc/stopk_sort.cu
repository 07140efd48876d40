// Radix sort of the rows of an s-Top-k call (fp32, adaptive probabilities, many segments) whose keys do not suit the buckets of
// stopk_segments.cu: most of the row lies in bins with a segment boundary, or one such bin holds a large share of it (rows
// with many zeros or equal magnitudes).  The sort takes the same time whatever the keys are.
//
// Least-significant-digit radix sort of the magnitude keys, 8 bits per pass (equal keys have equal energy, so the order among
// them is irrelevant); the norm of every segment is read off the sorted row.  How many rows are sorted is known on the device
// only: all passes are one cooperative launch as large as the GPU, with a grid barrier between two steps, whose blocks
// stride over the tiles of the rows to be sorted.  (As 13 launches it cost 17 us on calls without such a row, now 3.)
// The steps are bound by latency: a scatter takes 210 us for 4 x 11.7M keys, a count 30; the loads of a tile go out together, while
// the tile before is written (one by one behind the test for the row's end a count took 137).
// 11.7M x 4, L = 100, 95 % zeros: 28.6 ms in buckets, 1.72 sorted; 16 rows with 30 % zeros, three of them at a time: 8.7 and 5.6 ms.
#include <algorithm>

#include <cooperative_groups.h>

#include "stopk_sort.cuh"

namespace mlmc {

namespace {

namespace cg = cooperative_groups;

constexpr int kSortThreads = 512;
constexpr int kSortItems = kSortTile / kSortThreads;        // keys per thread
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kWarpKeys = kSortItems * 32;                  // every warp owns this many consecutive keys of the tile

// The rows to be sorted, in order; called by the whole block.
__device__ __forceinline__ int list_rows(const RowHead* head, int rows, uint16_t* list) {
    __shared__ int sh_n;
    if (threadIdx.x < 32) {
        int n = 0;
        for (int r0 = 0; r0 < rows; r0 += 32) {
            const int r = r0 + (int)threadIdx.x;
            const bool on = r < rows && head[r].sorted != 0u;
            const uint32_t all = __ballot_sync(0xFFFFFFFFu, on);
            if (on) list[n + __popc(all & ((1u << threadIdx.x) - 1u))] = (uint16_t)r;
            n += __popc(all);
        }
        if (threadIdx.x == 0) sh_n = n;
    }
    __syncthreads();
    return sh_n;
}

// The rows of one pass: the gradient, or the sort keys of the pass before.
struct PassInput {
    const uint32_t* rows;
    int64_t stride;
    uint32_t flip;                                           // kSortFlip for the gradient, else 0
    bool by_slot;
    __device__ __forceinline__ uint32_t key(uint32_t x) const { return (x ^ flip) & (flip ? kSortFlip : 0xFFFFFFFFu); }
};

constexpr int kSortSmemWords = kSortTile + 3 * kSortWarps * 256;  // the ordered tile, the warp tables, two mask tables

// The keys of a tile, kSortItems per thread; each warp owns kWarpKeys consecutive ones.
__device__ __forceinline__ void load_tile(const PassInput& in, int slot, int row, int tile, int64_t n, uint32_t (&key)[kSortItems]) {
    const int64_t w0 = (int64_t)tile * kSortTile + (int64_t)(threadIdx.x >> 5) * kWarpKeys + (threadIdx.x & 31);
    const uint32_t* src = in.rows + (int64_t)(in.by_slot ? slot : row) * in.stride + w0;
    if ((int64_t)(tile + 1) * kSortTile <= n) {
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) key[j] = __ldcg(src + j * 32);
    } else {
#pragma unroll
        for (int j = 0; j < kSortItems; ++j) key[j] = (w0 + j * 32 < n) ? __ldcg(src + j * 32) : 0u;
    }
}

// table[digit][tile] of a slot = keys of the tile with that digit.
__device__ __forceinline__ void count_tile(const PassInput& in, const uint32_t (&key)[kSortItems], int slot, int tile, int64_t n, int shift, uint32_t* table, int tiles,
                                           uint32_t* sh_hist /* [warp][256] */) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t w0 = (int64_t)tile * kSortTile + (int64_t)warp * kWarpKeys + lane;
    for (int i = threadIdx.x; i < kSortWarps * 256; i += kSortThreads) sh_hist[i] = 0u;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j)
        if (w0 + j * 32 < n) atomicAdd(&sh_hist[warp * 256 + ((in.key(key[j]) >> shift) & 0xFFu)], 1u);
    __syncthreads();
    if (threadIdx.x < 256) {
        uint32_t tot = 0;
#pragma unroll
        for (int w = 0; w < kSortWarps; ++w) tot += sh_hist[w * 256 + threadIdx.x];
        table[((int64_t)slot * 256 + threadIdx.x) * tiles + tile] = tot;
    }
    __syncthreads();
}

// Exclusive scan, in place, of the tile counts of one digit of one row, by a warp; the digit's total goes to totals[slot][digit].
// The scatter adds the totals of the digits below.
__device__ __forceinline__ void scan_digit(uint32_t* entries, int tiles, uint32_t* total) {
    const int lane = threadIdx.x & 31;
    uint32_t carry = 0;
    for (int i0 = 0; i0 < tiles; i0 += 128) {  // four per lane, consecutive
        uint32_t x[4], sum = 0;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = i0 + lane * 4 + j;
            x[j] = i < tiles ? entries[i] : 0u;
            sum += x[j];
        }
        uint32_t incl = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if (lane >= o) incl += y;
        }
        uint32_t run = carry + incl - sum;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int i = i0 + lane * 4 + j;
            if (i < tiles) entries[i] = run;
            run += x[j];
        }
        carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (lane == 0) *total = carry;
}

// Stable scatter of one pass.  The block first orders its tile by digit in shared memory (a key's place: start of
// its digit in the tile + keys with that digit in the warps before + its rank among its warp's keys with that
// digit, in input order), then writes the tile out so that consecutive threads write consecutive keys of a digit's
// run: the runs are contiguous in the output, from the scanned table.
// Ranks within a warp: the warp takes its keys 32 at a time in input order; the lanes of a step that hold the same
// digit meet in a shared-memory word per digit, into which each ORs its lane bit; the lowest of them advances the
// warp's running count of the digit and clears the word (two mask tables alternate, so that a step never meets the
// clearing of the step before).
// The next tile's keys are asked for (load_next) when this tile's have left their registers.
template <typename F>
__device__ __forceinline__ void scatter_tile(const PassInput& in, uint32_t (&key)[kSortItems], F&& load_next, int slot, int tile, uint32_t* out_row,
                                             int64_t n, int shift, const uint32_t* tables, const uint32_t* totals, int tiles, uint32_t* sh_dyn) {
    uint32_t* sh_key = sh_dyn;                            // [kSortTile]
    uint32_t* sh_hist = sh_dyn + kSortTile;               // [warp][256]
    uint32_t* sh_mask = sh_hist + kSortWarps * 256;       // [2][warp][256]
    __shared__ uint32_t sh_shift[256];  // position in the output - position in the ordered tile, per digit (mod 2^32)
    __shared__ uint32_t sh_wsum[8], sh_gsum[8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < 3 * kSortWarps * 256; i += kSortThreads) sh_hist[i] = 0u;
    const int64_t tile0 = (int64_t)tile * kSortTile;
    const int64_t w0 = tile0 + (int64_t)warp * kWarpKeys + lane;
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) key[j] = in.key(key[j]);
    __syncthreads();
    uint32_t* my_hist = sh_hist + warp * 256;
    uint32_t* my_mask = sh_mask + warp * 256;
    const uint32_t lane_bit = 1u << lane, lanes_below = lane_bit - 1u;
    uint32_t rank2[kSortItems / 2];  // two 16-bit ranks per word
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const bool live = w0 + j * 32 < n;
        const uint32_t digit = (key[j] >> shift) & 0xFFu;
        uint32_t* mask = my_mask + (j & 1) * (kSortWarps * 256) + digit;
        if (live) atomicOr(mask, lane_bit);
        __syncwarp();
        uint32_t peers = 0u, base = 0u;
        if (live) {
            peers = *mask;
            base = my_hist[digit];
        }
        __syncwarp();
        if (live && (peers & lanes_below) == 0u) {
            my_hist[digit] = base + __popc(peers);
            *mask = 0u;
        }
        const uint32_t rank = base + __popc(peers & lanes_below);
        if (j & 1)
            rank2[j >> 1] |= rank << 16;
        else
            rank2[j >> 1] = rank;
    }
    __syncthreads();
    {  // per digit: the tile-local start of every warp's keys, and the shift from the tile order to the output
        uint32_t total = 0, gtotal = 0;  // keys with this digit: in the tile, in the row
        if (threadIdx.x < 256) {
#pragma unroll
            for (int w = 0; w < kSortWarps; ++w) total += sh_hist[w * 256 + threadIdx.x];
            gtotal = __ldcg(&totals[slot * 256 + threadIdx.x]);
        }
        uint32_t incl = total, gincl = gtotal;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            const uint32_t gy = __shfl_up_sync(0xFFFFFFFFu, gincl, o);
            if (lane >= o) {
                incl += y;
                gincl += gy;
            }
        }
        if (threadIdx.x < 256 && lane == 31) {
            sh_wsum[warp] = incl;
            sh_gsum[warp] = gincl;
        }
        __syncthreads();
        if (threadIdx.x < 256) {
            uint32_t start = incl - total, gstart = gincl - gtotal;
            for (int w = 0; w < warp; ++w) {
                start += sh_wsum[w];
                gstart += sh_gsum[w];
            }
            sh_shift[threadIdx.x] = gstart + __ldcg(&tables[((int64_t)slot * 256 + threadIdx.x) * tiles + tile]) - start;
            uint32_t run = start;
#pragma unroll
            for (int w = 0; w < kSortWarps; ++w) {
                const uint32_t c = sh_hist[w * 256 + threadIdx.x];
                sh_hist[w * 256 + threadIdx.x] = run;
                run += c;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        if (w0 + j * 32 < n) {
            const uint32_t rank = (j & 1) ? (rank2[j >> 1] >> 16) : (rank2[j >> 1] & 0xFFFFu);
            sh_key[my_hist[(key[j] >> shift) & 0xFFu] + rank] = key[j];
        }
    }
    __syncthreads();
    load_next();
    const int tile_n = (int)((n - tile0 < (int64_t)kSortTile) ? (n - tile0) : (int64_t)kSortTile);
#pragma unroll
    for (int j = 0; j < kSortItems; ++j) {
        const int pos = j * kSortThreads + threadIdx.x;
        if (pos < tile_n) {
            const uint32_t k = sh_key[pos];
            out_row[(uint32_t)pos + sh_shift[(k >> shift) & 0xFFu]] = k;  // mod 2^32
        }
    }
    __syncthreads();  // the tables are cleared for the next tile
}

// Energy of keys begin .. end - 1 of a sorted row in fp64, in a fixed order, by a warp.
__device__ __forceinline__ double segment_energy(const uint32_t* keys, int64_t begin, int64_t end) {
    double e0 = 0.0, e1 = 0.0;
    int64_t i = begin + (threadIdx.x & 31);
    for (; i + 7 * 32 < end; i += 8 * 32) {
        uint32_t k[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) k[j] = __ldcg(keys + i + j * 32);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const double x = (double)__uint_as_float(kSortFlip - k[j]);
            if (j & 1) e1 = fma(x, x, e1);
            else e0 = fma(x, x, e0);
        }
    }
    for (; i < end; i += 32) {
        const double x = (double)__uint_as_float(kSortFlip - __ldcg(keys + i));
        e0 = fma(x, x, e0);
    }
    e0 += e1;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e0 += __shfl_xor_sync(0xFFFFFFFFu, e0, o);
    return e0;
}

// A warp adds up a segment, or kNormChunk keys of a longer one; the sums of those wait in the room of the digit table, two words each
// (at most 2 d / 4096 of them a row, in 256 words per 8192 keys).
constexpr int kNormChunk = 4096;

// No block leaves before the last barrier unless all do (the same flags decide in every block).
__global__ void __launch_bounds__(kSortThreads, 2)
sort_rows_kernel(const uint32_t* g, int64_t d, int64_t ld, int rows, const RowHead* head, SortBuffers buf, int tiles, uint32_t s_len, uint32_t L,
                 double* delta, int64_t seg_cap) {
    extern __shared__ __align__(16) uint32_t sh_dyn[];
    __shared__ uint16_t sh_list[kEmitMaxWorkers];
    pdl_enter();
    const int listed = list_rows(head, rows, sh_list);
    if (listed == 0) return;
    cg::grid_group grid = cg::this_grid();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t warps = gridDim.x * kSortWarps, first = blockIdx.x * kSortWarps + warp;
    // the block's tiles: every gridDim.x-th of all rows that are sorted at a time
    struct Place {
        int i, tile;   // the slot of the row
    };
    auto settle = [&](Place at) -> Place {
        while (at.tile >= tiles) {
            at.tile -= tiles;
            ++at.i;
        }
        return at;
    };
    const Place start = settle({0, (int)blockIdx.x});
#pragma unroll 1
    for (int r0 = 0; r0 < listed; r0 += buf.slots) {
        const int n_rows = min(buf.slots, listed - r0);
        const uint16_t* list = sh_list + r0;
        PassInput in = {g, ld, kSortFlip, false};
#pragma unroll 1
        for (int p = 0; p < 4; ++p) {  // 31-bit keys: from the gradient to b, to a, to b, to a
            const int shift = 8 * p;
            uint32_t key[kSortItems], next[kSortItems];
            auto load = [&](const Place& at, uint32_t (&k)[kSortItems]) {
                if (at.i < n_rows) load_tile(in, at.i, list[at.i], at.tile, d, k);
            };
            load(start, key);
#pragma unroll 1
            for (Place at = start; at.i < n_rows;) {
                const Place then = settle({at.i, at.tile + (int)gridDim.x});
                load(then, next);
                count_tile(in, key, at.i, at.tile, d, shift, buf.table, tiles, sh_dyn);
#pragma unroll
                for (int j = 0; j < kSortItems; ++j) key[j] = next[j];
                at = then;
            }
            grid.sync();
            for (uint32_t i = first; i < (uint32_t)n_rows * 256u; i += warps) scan_digit(buf.table + (int64_t)i * tiles, tiles, &buf.totals[i]);
            grid.sync();
            load(start, key);
#pragma unroll 1
            for (Place at = start; at.i < n_rows;) {
                const Place then = settle({at.i, at.tile + (int)gridDim.x});
                uint32_t* out_row = (p & 1) ? buf.a + (int64_t)list[at.i] * buf.stride : buf.b + (int64_t)at.i * buf.stride;
                scatter_tile(in, key, [&]() { load(then, key); }, at.i, at.tile, out_row, d, shift, buf.table, buf.totals, tiles, sh_dyn);
                at = then;
            }
            grid.sync();
            in = {(p & 1) ? buf.a : buf.b, buf.stride, 0u, (p & 1) == 0};
        }
        const uint32_t cps = (s_len + kNormChunk - 1) / kNormChunk;
        const int64_t items = (int64_t)L * cps;
        double* partial = reinterpret_cast<double*>(buf.table);
        for (int i = 0; i < n_rows; ++i) {
            const uint32_t* keys = buf.a + (int64_t)list[i] * buf.stride;
            for (int64_t at = first; at < items; at += warps) {
                const int64_t l = at / cps, begin = l * s_len + (at - l * cps) * kNormChunk;
                const int64_t end = min(min(begin + kNormChunk, (l + 1) * (int64_t)s_len), d);
                const double e = segment_energy(keys, begin, end);
                if (lane == 0) {
                    if (cps == 1) delta[(int64_t)list[i] * seg_cap + l] = sqrt(e);
                    else partial[(int64_t)i * 128 * tiles + at] = e;
                }
            }
        }
        if (cps == 1) continue;  // the next rows' counts do not touch what is read here
        grid.sync();
        for (int64_t at = (int64_t)first * 32 + lane; at < (int64_t)n_rows * L; at += (int64_t)warps * 32) {
            const int i = (int)(at / L);
            const double* part = partial + (int64_t)i * 128 * tiles + (at % L) * cps;
            double e = 0.0;
            for (uint32_t c = 0; c < cps; ++c) e += __ldcg(part + c);
            delta[(int64_t)list[i] * seg_cap + at % L] = sqrt(e);
        }
        grid.sync();  // the sums have been read: the table takes the next rows' counts
    }
}

}  // namespace

constexpr size_t kSortSmem = kSortSmemWords * sizeof(uint32_t);  // the tile and the tables pass 48 KB

int configure_sort_kernels() {
    return cudaFuncSetAttribute(sort_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSortSmem) == cudaSuccess ? MLMC_OK : MLMC_ERR_CUDA;
}

void sort_limits(KernelLimits* limits) { limits->sort_rows = resident_blocks(sort_rows_kernel, kSortThreads, kSortSmem); }

void launch_sorted_rows(Workspace& ws, const float* g, int64_t d, int rows, int64_t ld, const RowHead* head, const SortBuffers& buf,
                        uint32_t s_len, uint32_t L, double* delta, int64_t seg_cap, cudaStream_t s) {
    const int tiles = (int)sort_tiles(d);
    const int blocks = (int)std::min<int64_t>((int64_t)tiles * buf.slots, (int64_t)ws.sm_count * ws.limits.sort_rows);  // all of them run at a time
    launch_kernel_grid(ws, K_SORT_ROWS, sort_rows_kernel, dim3((unsigned)blocks), kSortThreads, kSortSmem, s,
                       reinterpret_cast<const uint32_t*>(g), d, ld, rows, head, buf, tiles, s_len, L, delta, seg_cap);
}

}  // namespace mlmc
