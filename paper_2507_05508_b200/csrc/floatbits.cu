// MLMC with the floating-point bit-wise compressor (Sec. 2.2 "Floating-point compressors", App. B).
//
// An entry is e = (-1)^S 2^(E - bias) (1 + sum_j m_j 2^-j).  C^l keeps sign, exponent and the first mb_l mantissa
// digits; the residual C^l - C^{l-1} is the field of digits mb_{l-1}+1 .. mb_l, worth f 2^-mb_l 2^(E - bias).  Sign
// and exponent are sent with every message (App. B counts 1 + exponent + 1 bits per entry), and they are the base
// g^0 = sign 2^(E - bias) of the estimate g^0 + (1/p^l)(C^l - C^{l-1}).  The level draw does not depend on the data
// (App. B's lemma gives fixed probabilities), so one sweep over the gradient writes the whole message.
#include <algorithm>

#include "bitplanes.cuh"

namespace mlmc {

namespace {

constexpr int kFloatThreads = 256;
template <typename T>
constexpr int kFloatBlocks = sizeof(T) == 4 ? 4 : 3;  // of the message kernel, per SM

struct MantissaSchedule {
    int L;
    int lo[kMaxLevels];  // mb_{l-1}
    int hi[kMaxLevels];  // mb_l
};

MantissaSchedule make_mantissa_schedule(const int32_t* mb, int L) {
    MantissaSchedule sc = {};
    sc.L = L;
    for (int l = 0; l < L; ++l) {
        sc.lo[l] = l ? mb[l - 1] : 0;
        sc.hi[l] = mb[l];
    }
    return sc;
}

// Bits 0..15 of x to the even bit positions.
__device__ __forceinline__ uint32_t spread_bits(uint32_t x) {
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}

// Word of bit `bit` of a lane's 32 entries.  fp32: one funnel shift collects the top bit of each (shifted) entry.
// bf16: the words hold two entries; the bits of the low and the high halves are collected apart and interleaved.
template <typename T>
__device__ __forceinline__ uint32_t plane_word(const uint32_t* x, int bit) {
    uint32_t w = 0;
    if constexpr (sizeof(T) == 4) {
#pragma unroll
        for (int t = 31; t >= 0; --t) w = __funnelshift_l(x[t] << (31 - bit), w, 1);
        return w;
    } else {
        uint32_t h = 0;  // bit = position in the 16-bit encoding
#pragma unroll
        for (int t = 15; t >= 0; --t) {
            h = __funnelshift_l(x[t] << (15 - bit), h, 1);
            w = __funnelshift_l(x[t] << (31 - bit), w, 1);
        }
        return spread_bits(w) | (spread_bits(h) << 1);
    }
}

// A warp turns 1024 consecutive entries into 32 words of the sign plane and of each mantissa plane and into 1024 exponent
// bytes.  A lane owns 32 consecutive entries, so every word is collected in the lane's own registers (2 instructions
// per entry and plane; from 6 planes on one bit transpose for all of them is cheaper).  The entries come through a
// slot of shared memory per warp filled by 16-byte asynchronous copies: the next group's copy starts when this group's words are in
// registers.  The 16-byte chunks of a lane are XOR-ed with its number so that the lanes' reads fall into different banks.
// The draw does not depend on the data (it is the host's); the worker's last block writes the header.
// Bound by HBM (reads 4 or 2 bytes, writes 1 byte and 1 + w bits per entry).  8 x 1M fp32 entries: 29.4 us per step with two slots and
// three blocks per SM, now 27.5 with one and four (8 x 124M: the same); bf16 rows are 1 % slower with four blocks.
// Prefetching the group after the next one into L2: 8 x 12M fp32 163.8 -> 147.6 us per step, bf16 127 -> 120, 8 x 124M fp32 message 946 -> 897;
// one more group ahead 165 and 8 x 124M 1.56 ms instead of 1.42 for the step.  Ballots over rows of 32 entries took 1.14 ms
// for 8 x 124M fp32 entries (0.72 of the copy rate).
template <typename T>
__global__ void __launch_bounds__(kFloatThreads, kFloatBlocks<T>)
float_pack_kernel(const T* __restrict__ g, int64_t d, int64_t ld, MantissaSchedule sc, const __grid_constant__ DrawnLevels drawn,
                  uint8_t* __restrict__ expo, uint32_t* __restrict__ planes, int w_max, int64_t words,
                  int32_t* out_level, double* out_p_sel, uint32_t* acc, uint32_t* done, int* status) {
    constexpr int kChunks = kGroupChunks<T>;
    constexpr int kSlot = kGroupSlot<T>;
    constexpr int kMantBits = sizeof(T) == 4 ? 23 : 7;
    extern __shared__ __align__(16) uint32_t sh_ring[];  // [warps][kSlot]
    const int m = blockIdx.y;
    const int level = drawn.level[m];
    pdl_enter();
    if (sc.hi[level] - sc.lo[level] > w_max) {  // the field does not fit the message buffer
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            set_status(status, MLMC_ERR_CAPACITY);
            out_level[m] = -1;
            out_p_sel[m] = 0.0;
        }
        return;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int lo = sc.lo[level], w = sc.hi[level] - lo;
    const T* row = g + (int64_t)m * ld;
    uint32_t* out = planes + (int64_t)m * (1 + w_max) * words;
    uint8_t* ex = expo + (int64_t)m * words * 32;
    uint32_t* ring = sh_ring + warp * kSlot;
    const int64_t ngroups = (words + 31) / 32;
    const int64_t stride = (int64_t)gridDim.x * (blockDim.x / 32);
    auto fetch = [&](int64_t grp, uint32_t* slot) { fetch_group<T>(row, d, grp, ngroups, slot); };
    const bool wide_store = (reinterpret_cast<uintptr_t>(expo) & 31) == 0;
    uint32_t top = 0;  // largest exponent field seen, at the top of the word
    int64_t grp = (int64_t)blockIdx.x * (blockDim.x / 32) + warp;
    fetch(grp, ring);
    for (; grp < ngroups; grp += stride) {
        cp_async_wait<0>();
        __syncwarp();
        uint32_t x[32];
#pragma unroll
        for (int c = 0; c < kChunks; ++c) {
            const uint4 q = *reinterpret_cast<const uint4*>(ring + group_place<T>(lane, c));
            x[4 * c] = q.x; x[4 * c + 1] = q.y; x[4 * c + 2] = q.z; x[4 * c + 3] = q.w;
        }
        __syncwarp();  // the slot has been read by every lane: the next copy may land in it
        fetch(grp + stride, ring);
        // and the group after it as far as L2
        if (lane < kChunks * 4 && (grp + 2 * stride + 1) * 1024 <= d) prefetch_line(reinterpret_cast<const uint4*>(row + (grp + 2 * stride) * 1024) + lane * 8);
        const int64_t word = grp * 32 + lane;
        const bool live = word < words;
        uint32_t e[8];  // the lane's exponent bytes
        if constexpr (sizeof(T) == 4) {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t a = x[4 * q] << 1, b = x[4 * q + 1] << 1, c = x[4 * q + 2] << 1, f = x[4 * q + 3] << 1;
                top = max(top, max(max(a, b), max(c, f)));
                e[q] = __byte_perm(__byte_perm(a, b, 0x0073), __byte_perm(c, f, 0x0073), 0x5410);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t a = x[2 * q] << 1, b = x[2 * q + 1] << 1;  // a bit of the low half reaches bit 16: not part of a field
                e[q] = __byte_perm(a, b, 0x7531);
                top = max(top, max(max(a, a << 16), max(b, b << 16)));
            }
        }
        if (live) {
            uint8_t* dst = ex + word * 32;
            if (wide_store) {
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(e[0]), "r"(e[1]), "r"(e[2]),
                             "r"(e[3]), "r"(e[4]), "r"(e[5]), "r"(e[6]), "r"(e[7])
                             : "memory");
            } else {
                reinterpret_cast<uint4*>(dst)[0] = make_uint4(e[0], e[1], e[2], e[3]);
                reinterpret_cast<uint4*>(dst)[1] = make_uint4(e[4], e[5], e[6], e[7]);
            }
        }
        const uint32_t sign_w = plane_word<T>(x, sizeof(T) == 4 ? 31 : 15);
        if (live) out[word] = sign_w;
        if (sizeof(T) == 2 || w < 6) {
            for (int j = 1; j <= w; ++j) {  // mantissa digit lo + j
                const uint32_t pw = plane_word<T>(x, kMantBits - (lo + j));
                if (live) out[(int64_t)j * words + word] = pw;
            }
        } else {
            transpose_bits(x);
#pragma unroll
            for (int bit = 22; bit >= 0; --bit) {
                const int j = kMantBits - bit - lo;
                if (live && j >= 1 && j <= w) out[(int64_t)j * words + word] = x[bit];
            }
        }
    }
    cp_async_wait<0>();
    if (top >= 0xFF000000u) atomicOr(&acc[m], 1u);
    if (!last_block(&done[m], gridDim.x) || threadIdx.x != 0) return;
    const bool any_bad = __ldcg(&acc[m]) != 0u;  // NaN or Inf: the worker's message is void
    acc[m] = 0u;
    if (any_bad) set_status(status, MLMC_ERR_NONFINITE);
    out_level[m] = any_bad ? -1 : level;
    out_p_sel[m] = drawn.p[level];
}

// Server average: thread = one word (32 entries); terms are added in worker order in fp32.
// A term is +-2^(E - 127) (1 + f 2^-mb_l / p): the power of two times a multiplier, added by one fused multiply-add (the
// product with a power of two is exact, so this is the sum of the rounded term).  An exponent field 0 has no leading one
// and the scale of exponent field 1; a word that holds one takes the general form.
// Bound by issue: 8 to 12 instructions per entry and worker.  8 x 124M entries: 0.88 ms with the general form for every entry,
// 0.55 with one worker in flight and fields wider than a bit gathered bit by bit, now 0.48 (10M x 8, wider fields: 161 -> 74 us).
constexpr int kAvgFloatRows = 8 + 1 + kAvgPlanes;  // words of a thread: 32 exponents, signs, planes
constexpr int kAvgFloatWords = kAvgSlots * kAvgFloatRows * 32 > kAvgStage ? kAvgSlots * kAvgFloatRows * 32 : kAvgStage;  // per warp
constexpr size_t kAvgFloatSmem = (size_t)kAvgFloatWords * (kAvgThreads / 32) * 4;

__global__ void __launch_bounds__(kAvgThreads)
aggregate_float_kernel(const uint8_t* __restrict__ expo, const uint32_t* __restrict__ planes, const int32_t* level,
                       const double* p_sel, const __grid_constant__ MantissaSchedule sc, int w_max, int64_t words, int M, int64_t d,
                       float* __restrict__ out) {
    // [warps][kAvgSlots][32 x two vectors of exponents, then rows of signs and planes][32], units and levels
    extern __shared__ __align__(16) uint32_t sh_ring[];
    float* sh_unit = reinterpret_cast<float*>(sh_ring + kAvgThreads / 32 * kAvgFloatWords);  // 2^-mb_l / p_l
    int* sh_level = reinterpret_cast<int*>(sh_unit + M);
    pdl_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* ring = sh_ring + warp * kAvgFloatWords;
    const float inv_M = 1.0f / (float)M;
    const int64_t nblk = (words + kAvgThreads - 1) / kAvgThreads;
    for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        const int64_t word = blk * kAvgThreads + threadIdx.x, at = min(word, words - 1);  // lanes past the end repeat the last word
        float acc[32];
#pragma unroll
        for (int t = 0; t < 32; ++t) acc[t] = 0.0f;
        auto slot = [&](int m) { return ring + (m & (kAvgSlots - 1)) * kAvgFloatRows * 32; };
        auto fetch = [&](int m) {  // the sign word to row 0, bit k of the fields (plane w - k) to row 1 + k
            const int lv = m < M ? __ldg(&level[m]) : -1;
            if (lv >= 0) {
                const int w = sc.hi[lv] - sc.lo[lv];
                const uint32_t* from = planes + (int64_t)m * (1 + w_max) * words + at;
                const uint8_t* e = expo + ((int64_t)m * words + at) * 32;
                uint32_t* to = slot(m);
                cp_async_16(to + lane * 4, e);
                cp_async_16(to + (32 + lane) * 4, e + 16);
                to += 8 * 32 + lane;
                cp_async_4(to, from);
                if (w <= kAvgPlanes)
                    for (int k = 0; k < w; ++k) cp_async_4(to + (1 + k) * 32, from + (int64_t)(w - k) * words);
            }
            cp_async_commit();
        };
#pragma unroll
        for (int m = 0; m < kAvgSlots - 1; ++m) fetch(m);
        if (blk == blockIdx.x) {  // while the first words are on their way
            for (int m = threadIdx.x; m < M; m += kAvgThreads) {
                const int lv = level[m];
                sh_level[m] = lv;
                sh_unit[m] = lv >= 0 ? (float)(ldexp(1.0, -sc.hi[lv]) / p_sel[m]) : 0.0f;
            }
            __syncthreads();
        }
        for (int m = 0; m < M; ++m) {  // fixed worker order
            fetch(m + kAvgSlots - 1);
            cp_async_wait<kAvgSlots - 1>();
            const int lv = sh_level[m];
            if (lv < 0) continue;
            const int w = sc.hi[lv] - sc.lo[lv];
            const float c = sh_unit[m];
            const uint32_t* from = slot(m);
            const uint4 ea = reinterpret_cast<const uint4*>(from)[lane], eb = reinterpret_cast<const uint4*>(from)[32 + lane];
            from += 8 * 32 + lane;
            const uint32_t sgn = from[0];
            const uint32_t e4[8] = {ea.x, ea.y, ea.z, ea.w, eb.x, eb.y, eb.z, eb.w};
            uint32_t zero = 0;  // some exponent byte is 0
#pragma unroll
            for (int q = 0; q < 8; ++q) zero |= (e4[q] - 0x01010101u) & ~e4[q] & 0x80808080u;
            // 2^(E - 127) of entry t
            auto base = [&](int t) {
                return __uint_as_float((t & 3) == 3 ? ((e4[t >> 2] >> 1) & 0x7F800000u) : ((e4[t >> 2] << (23 - 8 * (t & 3))) & 0x7F800000u));
            };
            if (zero == 0u && w == 1) {
                const uint32_t pw1 = from[32], m1 = __float_as_uint(1.0f + c);
#pragma unroll
                for (int t = 0; t < 32; ++t) {
                    const uint32_t mag = (pw1 & (1u << t)) ? m1 : 0x3F800000u;
                    acc[t] = fmaf(base(t), __uint_as_float(mag ^ ((sgn << (31 - t)) & 0x80000000u)), acc[t]);
                }
            } else if (zero == 0u && w <= kAvgPlanes && c < 0x1p100f) {
                uint32_t fb[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) fb[k] = k < w ? from[(1 + k) * 32] : 0u;
                fields_to_bytes(fb);
                const float offset = -8388608.0f * c;
#pragma unroll
                for (int t = 0; t < 32; ++t) {  // (1 + f c) 2^(E - 127): the power of two is exact
                    const uint32_t mag = __float_as_uint(1.0f + field_times(fb, t, c, offset));
                    acc[t] = fmaf(base(t), __uint_as_float(mag ^ ((sgn << (31 - t)) & 0x80000000u)), acc[t]);
                }
            } else {
                uint32_t f[32];
                gather_fields<4>(planes + ((int64_t)m * (1 + w_max) + 1) * words + at, words, w, f);
#pragma unroll
                for (int t = 0; t < 32; ++t) {
                    const uint32_t E = (e4[t >> 2] >> (8 * (t & 3))) & 0xFFu;
                    const float low = __uint_as_float(E << 23);                    // 2^(E - 127), or 0
                    const float scale = __uint_as_float(max(E, 1u) << 23);         // 2^(max(E, 1) - 127)
                    const float ff = __uint_as_float(0x4B000000u | f[t]) - 8388608.0f;  // exact integer-to-float
                    const float v = fmaf(ff * c, scale, low);  // the power of two last: ff c is a normal number
                    acc[t] += __uint_as_float(__float_as_uint(v) ^ ((sgn << (31 - t)) & 0x80000000u));
                }
            }
        }
        cp_async_wait<0>();
        store_words(ring, acc, inv_M, blk * kAvgThreads + warp * 32, d, out);
    }
}

size_t float_pack_smem(size_t elem, int warps) { return (size_t)warps * 1024 * elem; }

}  // namespace

int configure_float_kernels() {
    const bool ok = cudaFuncSetAttribute(aggregate_float_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kAvgFloatSmem + kEmitMaxWorkers * 8) == cudaSuccess &&
                    cudaFuncSetAttribute(float_pack_kernel<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)float_pack_smem(4, kFloatThreads / 32)) == cudaSuccess;
    return ok ? MLMC_OK : MLMC_ERR_CUDA;
}

void float_limits(KernelLimits* limits) { limits->aggregate_float = resident_blocks(aggregate_float_kernel, kAvgThreads, kAvgFloatSmem + 64); }

void launch_compress_floatbits(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* mb,
                               int L, const double* p, uint64_t seed, uint64_t step, const mlmc_float_msgs& out,
                               cudaStream_t s) {
    const MantissaSchedule sc = make_mantissa_schedule(mb, L);
    const int64_t words = (d + 31) / 32;
    const int64_t ngroups = (words + 31) / 32;
    const int warps = (int)std::min<int64_t>(ngroups, kFloatThreads / 32);  // of short rows as many blocks as possible fit an SM
    const int64_t by_work = (ngroups + warps - 1) / warps;
    int64_t nb = ((int64_t)ws.sm_count * (dtype == MLMC_BF16 ? kFloatBlocks<bf16_t> : kFloatBlocks<float>)) / M;  // persistent: one wave, rounded down
    if (nb > by_work) nb = by_work;
    if (nb < 1) nb = 1;
    const DrawnLevels drawn = draw_levels(p, L, seed, step, M);
    auto go = [&](auto kernel, auto* row) {
        launch_kernel(ws, K_FLOAT_PACK, kernel, dim3((unsigned)nb, M), warps * 32, float_pack_smem(sizeof(*row), warps), s, row, d, ld, sc, drawn, out.expo, out.planes, out.w_max, words, out.level, out.p_sel, ws.acc_word, ws.done, ws.status);
    };
    if (dtype == MLMC_BF16) go(float_pack_kernel<bf16_t>, static_cast<const bf16_t*>(g));
    else go(float_pack_kernel<float>, static_cast<const float*>(g));
}

void launch_aggregate_floatbits(Workspace& ws, const mlmc_float_msgs& msgs, const int32_t* mb, int L, int M, int64_t d,
                                float* out, cudaStream_t s) {
    const MantissaSchedule sc = make_mantissa_schedule(mb, L);
    const int64_t words = (d + 31) / 32;
    const size_t smem = kAvgFloatSmem + (size_t)M * 8;
    const int64_t nb = std::min((words + kAvgThreads - 1) / kAvgThreads, (int64_t)ws.sm_count * ws.limits.aggregate_float * 2);
    launch_kernel(ws, K_AGG_FLOAT, aggregate_float_kernel, dim3((unsigned)nb), kAvgThreads, smem, s, msgs.expo, msgs.planes,
                  msgs.level, msgs.p_sel, sc, msgs.w_max, words, M, d, out);
}

}  // namespace mlmc
