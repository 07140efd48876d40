// The band of ranks (k_{l-1}, k_l] on the words of a gradient row: membership, counts and ordered output of one batch.
#pragma once

#include "common.cuh"

namespace mlmc {
namespace {

constexpr int kBatchWords = kEmitRows * 32;     // words a warp holds in registers at a time
static_assert(kEmitTile / kBatchWords == kEmitGroups, "a tile is kEmitGroups batches");

// How a 32-bit word of the gradient row maps to elements: one fp32 element, or two bf16 elements
// (low half first).  A word past the end of the row reads as kPad, whose keys lie above every
// threshold the kernels use (thresholds are clamped to kCap, the key of +Inf), so padded elements
// are never inside the band.
template <typename T>
struct EmitWord;

template <>
struct EmitWord<float> {
    static constexpr int S = 1;
    static constexpr uint32_t kPad = 0x7FFFFFFFu;
    static constexpr uint32_t kCap = 0x7F800000u;
    __device__ static __forceinline__ uint32_t key(uint32_t w, int) { return w & 0x7FFFFFFFu; }
    __device__ static __forceinline__ float value(uint32_t w, int) { return __uint_as_float(w); }
};

template <>
struct EmitWord<bf16_t> {
    static constexpr int S = 2;
    static constexpr uint32_t kPad = 0x7FFF7FFFu;
    static constexpr uint32_t kCap = 0x7F80u;
    __device__ static __forceinline__ uint32_t key(uint32_t w, int s) { return s ? ((w >> 16) & 0x7FFFu) : (w & 0x7FFFu); }
    __device__ static __forceinline__ float value(uint32_t w, int s) {
        return __uint_as_float(s ? (w & 0xFFFF0000u) : (w << 16));
    }
};

// Number of band entries among a prefix of the row that holds C closed-range keys, A keys equal to Ta
// and B keys equal to Tb: the first min(A, ra) ties of Ta belong to Top-k_{l-1} (not to the band), and
// only the first min(B, rb) ties of Tb belong to Top-k_l.
__device__ __forceinline__ uint32_t band_prefix(uint32_t C, uint32_t A, uint32_t B, uint32_t ra, uint32_t rb) {
    return C - B + min(B, rb) - min(A, ra);
}

// Lane `lane` of a warp loads word i * 32 + lane (i < kEmitRows) of batch `batch` of tile `tile`: every row
// is one coalesced 128-byte request.  Words past the end of the row read as kPad.
template <typename T>
__device__ __forceinline__ void load_batch(const T* __restrict__ row, int64_t d, int64_t tile, int batch, int lane,
                                           uint32_t (&w)[kEmitRows]) {
    using EW = EmitWord<T>;
    const int64_t w0 = tile * kEmitTile + (int64_t)batch * kBatchWords + lane;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(row) + w0;
    if ((w0 - lane + kBatchWords) * EW::S <= d) {
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i) w[i] = __ldg(words + i * 32);
    } else {
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i) {
            const int64_t wi = w0 + i * 32;
            uint32_t v = EW::kPad;
            if ((wi + 1) * EW::S <= d) {
                v = __ldg(words + i * 32);
            } else if (EW::S == 2 && wi * 2 < d) {  // odd bf16 tail: only the low half exists
                v = (uint32_t)reinterpret_cast<const uint16_t*>(row)[wi * 2] | 0x7FFF0000u;
            }
            w[i] = v;
        }
    }
}

// The write pass gives every lane 16 consecutive words of a batch (four 16-byte chunks), so that the order of the
// lanes is the order of the coordinates.  Chunk c = 4 * lane + j of the batch is kept at position swz(c) of the
// warp's shared-memory slot: with the two low bits of the chunk number XOR-ed with bits 3..4, the eight lanes of a
// quarter warp read their j-th chunks (128-bit loads, 64 bytes apart before the swizzle) from eight different
// 16-byte bank groups.
__device__ __forceinline__ int swz(int c) { return (c & ~3) | ((c ^ (c >> 3)) & 3); }

// Starts the copy of batch `batch` of tile `tile` into a warp's shared-memory slot (kBatchWords words in the
// swizzled chunk order above): 16-byte asynchronous copies, or plain padded stores for the ragged end of the row.
template <typename T>
__device__ __forceinline__ void copy_batch_async(const T* __restrict__ row, int64_t d, int64_t tile, int batch, int lane,
                                                 uint32_t* slot) {
    using EW = EmitWord<T>;
    const int64_t w0 = tile * kEmitTile + (int64_t)batch * kBatchWords;
    const uint32_t* words = reinterpret_cast<const uint32_t*>(row) + w0;
    if ((w0 + kBatchWords) * EW::S <= d) {
#pragma unroll
        for (int c = lane; c < kBatchWords / 4; c += 32) cp_async_16(slot + swz(c) * 4, words + c * 4);
    } else {
        for (int i = lane; i < kBatchWords; i += 32) {
            const int64_t wi = w0 + i;
            uint32_t v = EW::kPad;
            if ((wi + 1) * EW::S <= d) {
                v = __ldg(words + i);
            } else if (EW::S == 2 && wi * 2 < d) {  // odd bf16 tail: only the low half exists
                v = (uint32_t)reinterpret_cast<const uint16_t*>(row)[wi * 2] | 0x7FFF0000u;
            }
            slot[swz(i >> 2) * 4 + (i & 3)] = v;
        }
    }
}

// Closed-range flags of one batch and, per lane, its counts.  flags: bit i (fp32) or bits i and 16 + i
// (bf16 low / high half) = word i of this lane holds a key with Tb <= key <= Ta.  cA / cB: this lane's keys
// equal to Ta / Tb (looked for only when the warp has a closed-range key at all; ties are closed-range keys).
template <typename T>
__device__ __forceinline__ uint32_t batch_flags(const uint32_t (&w)[kEmitRows], uint32_t Tb, uint32_t Ta, uint32_t* cA,
                                                uint32_t* cB) {
    uint32_t flags = 0, a = 0, b = 0;
    if constexpr (EmitWord<T>::S == 1) {
        const uint32_t W = Ta - Tb;
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i)
            if (((w[i] & 0x7FFFFFFFu) - Tb) <= W) flags |= 1u << i;
        if (__any_sync(0xFFFFFFFFu, flags != 0u)) {
#pragma unroll
            for (int i = 0; i < kEmitRows; ++i) {
                const uint32_t tk = (w[i] & 0x7FFFFFFFu) - Tb;
                a += (tk == W) ? 1u : 0u;
                b += (tk == 0u) ? 1u : 0u;
            }
        }
    } else {
        // two 15-bit keys per word; bit 15 of each half is free, so both halves are compared at
        // once: (key + 0x8000 - T) has bit 15 set iff key >= T, (T + 0x8000 - key) iff key <= T
        const uint32_t hi = 0x80008000u;
        const uint32_t geB = hi - Tb * 0x10001u, geB1 = hi - (Tb + 1u) * 0x10001u;
        const uint32_t leA = hi + Ta * 0x10001u, leA1 = hi + (Ta ? Ta - 1u : 0u) * 0x10001u;
        const uint32_t keepA1 = Ta ? 0xFFFFFFFFu : 0u;  // Ta = 0: every closed key equals Ta
        uint32_t acc = 0;
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i) {
            const uint32_t k2 = w[i] & 0x7FFF7FFFu;
            flags |= ((k2 + geB) & (leA - k2) & hi) >> (15 - i);
        }
        if (__any_sync(0xFFFFFFFFu, flags != 0u)) {
#pragma unroll
            for (int i = 0; i < kEmitRows; ++i) {
                const uint32_t k2 = w[i] & 0x7FFF7FFFu;
                const uint32_t f = (k2 + geB) & (leA - k2) & hi;
                const uint32_t fB = f & ~(k2 + geB1);
                const uint32_t fA = f & ~((leA1 - k2) & keepA1);
                acc += (fA >> 15) + (fB >> 7);  // 5-bit counters: A at bits 0 / 16, B at bits 8 / 24
            }
        }
        a = (acc & 0x1Fu) + ((acc >> 16) & 0x1Fu);
        b = ((acc >> 8) & 0x1Fu) + ((acc >> 24) & 0x1Fu);
    }
    *cA = a;
    *cB = b;
    return flags;
}

// The same flags for the write pass, with the ties as masks instead of counts: bit i (fp32) or bits i and 16 + i
// (bf16 low / high half) of mA / mB = word i of this lane holds a key equal to Ta / Tb.
template <typename T>
__device__ __forceinline__ uint32_t batch_masks(const uint32_t (&w)[kEmitRows], uint32_t Tb, uint32_t Ta, bool ties,
                                                uint32_t* mA, uint32_t* mB) {
    uint32_t flags = 0, a = 0, b = 0;  // ties = false: the tile holds no key equal to a threshold, the masks stay empty
    if constexpr (EmitWord<T>::S == 1) {
        const uint32_t W = Ta - Tb;
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i)
            if (((w[i] & 0x7FFFFFFFu) - Tb) <= W) flags |= 1u << i;
        if (ties && __any_sync(0xFFFFFFFFu, flags != 0u)) {
#pragma unroll
            for (int i = 0; i < kEmitRows; ++i) {
                const uint32_t tk = (w[i] & 0x7FFFFFFFu) - Tb;
                a |= (tk == W) ? (1u << i) : 0u;
                b |= (tk == 0u) ? (1u << i) : 0u;
            }
        }
    } else {
        const uint32_t hi = 0x80008000u;
        const uint32_t geB = hi - Tb * 0x10001u, geB1 = hi - (Tb + 1u) * 0x10001u;
        const uint32_t leA = hi + Ta * 0x10001u, leA1 = hi + (Ta ? Ta - 1u : 0u) * 0x10001u;
        const uint32_t keepA1 = Ta ? 0xFFFFFFFFu : 0u;  // Ta = 0: every closed key equals Ta
#pragma unroll
        for (int i = 0; i < kEmitRows; ++i) {
            const uint32_t k2 = w[i] & 0x7FFF7FFFu;
            flags |= ((k2 + geB) & (leA - k2) & hi) >> (15 - i);
        }
        if (ties && __any_sync(0xFFFFFFFFu, flags != 0u)) {
#pragma unroll
            for (int i = 0; i < kEmitRows; ++i) {
                const uint32_t k2 = w[i] & 0x7FFF7FFFu;
                const uint32_t f = (k2 + geB) & (leA - k2) & hi;
                b |= (f & ~(k2 + geB1)) >> (15 - i);
                a |= (f & ~((leA1 - k2) & keepA1)) >> (15 - i);
            }
        }
    }
    *mA = a;
    *mB = b;
    return flags;
}

// The band of one worker as the emission needs it.
struct Band {
    uint32_t Tb, Ta;     // clamped thresholds, W = Ta - Tb
    uint32_t ra, rb;
    float inv_p;
};

// Writes the band entries of one batch, by a warp.  slot: the batch's words in shared memory, in the swizzled chunk order;
// e0: coordinate of the batch's first entry; run: {C, A, B} before the batch, advanced past it.
// A lane owns 16 consecutive words of the batch, so the order of the lanes is the order of the coordinates: the
// position of a lane's first entry is the batch's base plus the entries of the lanes before it (one warp scan).
// Few entries: every lane writes its own, one after the other.  From kStagedEntries on, the lanes leave the offsets of their
// entries in `stage` (kBatchWords * S half words; null: never) and the warp writes the whole run, consecutive lanes to consecutive places:
// a store of scattered words costs a 32-byte packet to L2 per entry, a coalesced one an eighth of that (32 x 25.6M bf16
// entries: write pass 441 -> 291 us).
constexpr uint32_t kStagedEntries = 64;
template <typename T>
__device__ __forceinline__ void emit_batch(const uint32_t* slot, uint16_t* stage, const Band& band, bool tile_ties, uint32_t e0,
                                           uint3& run, uint32_t* __restrict__ idx_w, float* __restrict__ val_w, int64_t capacity) {
    using EW = EmitWord<T>;
    constexpr int S = EW::S;
    static_assert(kEmitRows == 16, "a lane owns four 16-byte chunks of a batch");
    const int lane = threadIdx.x & 31;
    // where this lane's words sit in a slot: word r at own + (r ^ own_xor), i.e. chunk q at swz(4 * lane + q)
    const int own = lane * kEmitRows, own_xor = ((lane >> 1) & 3) << 2;
    const uint32_t W = band.Ta - band.Tb;
    uint32_t cur[kEmitRows];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 x = *reinterpret_cast<const uint4*>(slot + own + ((4 * q) ^ own_xor));
        cur[4 * q + 0] = x.x; cur[4 * q + 1] = x.y; cur[4 * q + 2] = x.z; cur[4 * q + 3] = x.w;
    }
    uint32_t mA, mB;
    uint32_t member = batch_masks<T>(cur, band.Tb, band.Ta, tile_ties, &mA, &mB);
    if (!__any_sync(0xFFFFFFFFu, member != 0u)) return;  // no closed-range key in the batch: nothing to count either
    const uint32_t nC = __popc(member), nA = __popc(mA), nB = __popc(mB);
    const uint32_t totCA = __reduce_add_sync(0xFFFFFFFFu, nC | (nA << 16));
    const uint32_t myB = __reduce_add_sync(0xFFFFFFFFu, nB);
    const uint32_t myC = totCA & 0xFFFFu, myA = totCA >> 16;
    const uint32_t base = band_prefix(run.x, run.y, run.z, band.ra, band.rb);
    if ((myA | myB) != 0u) {  // warp-uniform
        // Ties in this batch.  Unless the cut rank of a threshold falls among them, all of them are on one
        // side of it: the ties of Ta all outside Top-k_{l-1} (in the band) or all inside (dropped), the ties
        // of Tb all inside Top-k_l (in the band) or all outside (dropped).  Only a batch that holds a cut
        // ranks its ties one by one.
        const bool dropA = myA != 0u && run.y + myA <= band.ra, keepA = myA == 0u || run.y >= band.ra;
        const bool dropB = myB != 0u && run.z >= band.rb, keepB = myB == 0u || run.z + myB <= band.rb;
        const bool ranked = !((keepA || dropA) && (keepB || dropB)) || W == 0u;
        if (!ranked) {
            if (dropA) member &= ~mA;
            if (dropB) member &= ~mB;
        } else {
            // index-ordered tie ranks (0-based): the ties of the lanes before this one, then this lane's in order
            uint32_t iA = nA, iB = nB;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t yA = __shfl_up_sync(0xFFFFFFFFu, iA, o), yB = __shfl_up_sync(0xFFFFFFFFu, iB, o);
                if (lane >= o) { iA += yA; iB += yB; }
            }
            uint32_t tA = run.y + iA - nA, tB = run.z + iB - nB;
            const uint32_t t = mA | mB;
            uint32_t rows = (S == 1) ? t : ((t | (t >> 16)) & 0xFFFFu);
            while (rows) {
                const int r = __ffs(rows) - 1;
                rows &= rows - 1u;
#pragma unroll
                for (int s = 0; s < S; ++s) {
                    const uint32_t bit = 1u << (r + 16 * s);
                    if (mA & bit) {
                        if (tA < band.ra) member &= ~bit;   // still inside Top-k_{l-1}
                        ++tA;
                    }
                    if (mB & bit) {
                        if (tB >= band.rb) member &= ~bit;  // already outside Top-k_l
                        ++tB;
                    }
                }
            }
        }
    }
    // positions: the batch's base plus the entries of the lanes before this one
    const uint32_t cnt = __popc(member);
    uint32_t incl = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    run.x += myC; run.y += myA; run.z += myB;
    const uint32_t total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    if (stage && total >= kStagedEntries) {
        uint32_t x = member;  // bit i: entry i of this lane's S * 16
        if (S == 2) {         // bits i and 16 + i -> 2 i and 2 i + 1
            uint32_t t;
            t = (x ^ (x >> 8)) & 0x0000FF00u; x ^= t ^ (t << 8);
            t = (x ^ (x >> 4)) & 0x00F000F0u; x ^= t ^ (t << 4);
            t = (x ^ (x >> 2)) & 0x0C0C0C0Cu; x ^= t ^ (t << 2);
            t = (x ^ (x >> 1)) & 0x22222222u; x ^= t ^ (t << 1);
        }
        uint16_t* to = stage + (incl - cnt);
        const uint32_t mine = (uint32_t)(lane * kEmitRows * S);
        while (x) {
            *to++ = (uint16_t)(mine + (uint32_t)__ffs(x) - 1u);
            x &= x - 1u;
        }
        __syncwarp();
        const uint32_t n = (int64_t)base + total <= capacity ? total : (int64_t)base < capacity ? (uint32_t)(capacity - base) : 0u;
#pragma unroll 2
        for (uint32_t i = lane; i < n; i += 32) {
            const uint32_t o = stage[i], w = S == 2 ? o >> 1 : o;
            const uint32_t v = slot[(w & ~12u) | (((w >> 2) ^ (w >> 5)) & 3u) << 2];  // word w in the swizzled slot
            idx_w[base + i] = e0 + o;
            val_w[base + i] = (S == 2 ? __uint_as_float((o & 1u) ? v & 0xFFFF0000u : v << 16) : __uint_as_float(v)) * band.inv_p;
        }
        return;  // the next batch's stage is written after the caller's __syncwarp
    }
    uint32_t pos = base + incl - cnt;
    const uint32_t lane_e0 = e0 + (uint32_t)(lane * kEmitRows * S);
    uint32_t rows = (S == 1) ? member : ((member | (member >> 16)) & 0xFFFFu);
    while (rows) {  // this lane's words that hold an entry, in ascending order
        const int r = __ffs(rows) - 1;
        rows &= rows - 1u;
        const uint32_t w = slot[own + (r ^ own_xor)];  // word r of this lane in the swizzled slot
#pragma unroll
        for (int s = 0; s < S; ++s) {
            if ((member >> (r + 16 * s)) & 1u) {
                if ((int64_t)pos < capacity) {
                    idx_w[pos] = lane_e0 + (uint32_t)(r * S + s);
                    val_w[pos] = EW::value(w, s) * band.inv_p;
                }
                ++pos;
            }
        }
    }
}

}  // namespace
}  // namespace mlmc
