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

struct SortBuffers {
    uint32_t* a;             // [rows][stride]
    uint32_t* b;             // [rows][stride]  the sorted row
    uint32_t* table;         // [rows][256][tiles]
    uint32_t* totals;        // [rows][256]
    int64_t stride;
};

int configure_sort_kernels();
void sort_limits(KernelLimits* limits);
// Sorts the rows with head.sorted and writes the norms of their segments to delta[rows][seg_cap].
void launch_sorted_rows(Workspace& ws, const float* g, int64_t d, int rows, int64_t ld, const RowHead* head, const SortBuffers& buf,
                        uint32_t s_len, uint32_t L, double* delta, int64_t seg_cap, cudaStream_t s);

}  // namespace mlmc
