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

// ---- averages of plane messages: a thread adds up one word (32 entries) of every worker's planes, worker after worker.  Its
// words come through a ring of kAvgSlots shared-memory slots, thread by thread: the next three workers' are in flight.  (In
// registers there was room for one worker and one plane of it: 20 KB in flight per SM, half of what HBM needs.)
constexpr int kAvgThreads = 256;
constexpr int kAvgSlots = 4;
constexpr int kAvgStage = 32 * 33;   // words of a warp's output rows; they take the place of its ring
constexpr int kAvgPlanes = 8;       // magnitude planes in the ring; the fields of wider levels are read as they are used

__device__ __forceinline__ void cp_async_4(void* smem_dst, const void* gmem_src) {
    const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(gmem_src) : "memory");
}

// fb[k] holds bit k of 32 fields of at most 8 bits; afterwards byte t >> 3 of fb[t & 7] is the field of entry t.
__device__ __forceinline__ void fields_to_bytes(uint32_t (&fb)[8]) {
#pragma unroll
    for (int j = 4; j > 0; j >>= 1) {
        const uint32_t mask = j == 4 ? 0x0F0F0F0Fu : j == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (k & j) continue;
            const uint32_t x = ((fb[k] >> j) ^ fb[k + j]) & mask;
            fb[k + j] ^= x;
            fb[k] ^= x << j;
        }
    }
}

// f unit for the field f of entry t, rounded once: a byte below the bits of 2^23 is 2^23 + f, and offset = -2^23 unit.
__device__ __forceinline__ float field_times(const uint32_t (&fb)[8], int t, float unit, float offset) {
    return fmaf(__uint_as_float(__byte_perm(fb[t & 7], 0x4B000000u, 0x7650u + (uint32_t)(t >> 3))), unit, offset);
}

// Fields of any width, plane by plane, the words of AHEAD planes in flight.
template <int AHEAD>
__device__ __forceinline__ void gather_fields(const uint32_t* __restrict__ plane1, int64_t words, int w, uint32_t (&f)[32]) {
#pragma unroll
    for (int t = 0; t < 32; ++t) f[t] = 0u;
    for (int j0 = 0; j0 < w; j0 += AHEAD) {
        uint32_t pw[AHEAD];
#pragma unroll
        for (int j = 0; j < AHEAD; ++j) pw[j] = j0 + j < w ? __ldg(plane1 + (int64_t)(j0 + j) * words) : 0u;
#pragma unroll
        for (int j = 0; j < AHEAD; ++j) {
            if (j0 + j >= w) break;
#pragma unroll
            for (int t = 0; t < 32; ++t) f[t] = (f[t] << 1) | ((pw[j] >> t) & 1u);
        }
    }
}

// The 32 sums of every lane of a warp, whose words are word0 + lane, leave as rows of 128 bytes.  stage: 32 x 33 words.
__device__ __forceinline__ void store_words(uint32_t* stage_words, const float (&acc)[32], float factor, int64_t word0, int64_t d,
                                            float* __restrict__ out) {
    float (*stage)[33] = reinterpret_cast<float (*)[33]>(stage_words);
    const int lane = threadIdx.x & 31;
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 32; ++t) stage[lane][t] = acc[t] * factor;
    __syncwarp();
#pragma unroll 4
    for (int r = 0; r < 32; ++r) {
        const int64_t i = (word0 + r) * 32 + lane;
        if (i < d) out[i] = stage[r][lane];
    }
    __syncwarp();
}

}  // namespace
}  // namespace mlmc
