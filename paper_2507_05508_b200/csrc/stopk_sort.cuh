// Rows of an s-Top-k call that are sorted instead of split into buckets (stopk_sort.cu; the rule is in stopk_segments.cu).
#pragma once

#include "common.cuh"

namespace mlmc {

// What the first kernel of the segment norms finds out about a row.
struct RowHead {
    uint32_t buckets, cells;
    uint32_t sorted;         // the row takes the radix sort
    uint32_t pad;
};

constexpr int kSortTile = 8192;                              // keys per block and trip
constexpr uint32_t kSortFlip = 0x7FFFFFFFu;                  // sort key = flip - magnitude key: ascending sort, descending magnitude

inline int64_t sort_tiles(int64_t d) { return (d + kSortTile - 1) / kSortTile; }

// Rows that are sorted at a time: as many as keep the GPU busy (32M keys), so that all but the first buffer stay small.
inline int sort_slots(int64_t d, int rows) {
    const int64_t n = ((int64_t(1) << 25) + d - 1) / d;
    return n < rows ? (int)n : rows;
}

struct SortBuffers {
    uint32_t* a;             // [rows][stride]   the sorted row
    uint32_t* b;             // [slots][stride]
    uint32_t* table;         // [slots][256][tiles]
    uint32_t* totals;        // [slots][256]
    int64_t stride;
    int slots;
};

int configure_sort_kernels();
void sort_limits(KernelLimits* limits);
// Sorts the rows with head.sorted and writes the norms of their segments to delta[rows][seg_cap].
void launch_sorted_rows(Workspace& ws, const float* g, int64_t d, int rows, int64_t ld, const RowHead* head, const SortBuffers& buf,
                        uint32_t s_len, uint32_t L, double* delta, int64_t seg_cap, cudaStream_t s);

}  // namespace mlmc
