// Bit planes of 1024 consecutive entries by one warp: a lane owns 32 consecutive entries, that is one word of every plane.
#pragma once

#include "common.cuh"

namespace mlmc {
namespace {

template <typename T>
constexpr int kGroupChunks = 32 * (int)sizeof(T) / 16;   // 16-byte chunks of a lane's entries: 8 or 4
template <typename T>
constexpr int kGroupSlot = 1024 * (int)sizeof(T) / 4;    // 32-bit words of a group

// Where chunk c of lane l is kept in a group's shared-memory slot: XOR-ed with the lane's number, so that the lanes' reads
// of their c-th chunks fall into different banks (bf16: a lane's chunks are 64 bytes, so every second lane).
template <typename T>
__device__ __forceinline__ int group_place(int l, int c) {
    constexpr int n = kGroupChunks<T>;
    return l * n * 4 + ((c ^ ((n == 8 ? l : l >> 1) & (n - 1))) << 2);
}

// Starts the copy of group `grp` of a row into a warp's slot (16-byte asynchronous copies; the ragged end of the row by
// plain stores, entries past d read as +0) and commits it.
template <typename T>
__device__ __forceinline__ void fetch_group(const T* __restrict__ row, int64_t d, int64_t grp, int64_t ngroups, uint32_t* slot) {
    constexpr int n = kGroupChunks<T>;
    const int lane = threadIdx.x & 31;
    if (grp < ngroups) {
        const int64_t e0 = grp * 1024;
        if (e0 + 1024 <= d) {
            const uint4* src = reinterpret_cast<const uint4*>(row + e0);
#pragma unroll
            for (int j = 0; j < n; ++j) {
                const int i = j * 32 + lane;  // chunk of the group
                cp_async_16(slot + group_place<T>(i / n, i % n), src + i);
            }
        } else {
            for (int i = lane; i < kGroupSlot<T>; i += 32) {
                uint32_t v = 0u;
                if constexpr (sizeof(T) == 4) {
                    if (e0 + i < d) v = reinterpret_cast<const uint32_t*>(row)[e0 + i];
                } else {
                    const uint16_t* h = reinterpret_cast<const uint16_t*>(row) + e0;
                    if (e0 + 2 * i < d) v = h[2 * i];
                    if (e0 + 2 * i + 1 < d) v |= (uint32_t)h[2 * i + 1] << 16;
                }
                slot[group_place<T>(i / (n * 4), (i % (n * 4)) / 4) + (i & 3)] = v;
            }
        }
    }
    cp_async_commit();
}

// 32 x 32 bit transpose: on return bit t of x[b] is bit b of the former x[t].
__device__ __forceinline__ void transpose_bits(uint32_t (&x)[32]) {
#pragma unroll
    for (int k = 0; k < 16; ++k) {
        const uint32_t a = x[k], b = x[k + 16];
        x[k] = __byte_perm(a, b, 0x5410);
        x[k + 16] = __byte_perm(a, b, 0x7632);
    }
#pragma unroll
    for (int k = 0; k < 32; ++k) {
        if (k & 8) continue;
        const uint32_t a = x[k], b = x[k + 8];
        x[k] = __byte_perm(a, b, 0x6240);
        x[k + 8] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
    for (int j = 4; j > 0; j >>= 1) {
        const uint32_t mask = j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int k = 0; k < 32; ++k) {
            if (k & j) continue;
            const uint32_t t = ((x[k] >> j) ^ x[k + j]) & mask;
            x[k + j] ^= t;
            x[k] ^= t << j;
        }
    }
}

}  // namespace
}  // namespace mlmc
