// MLMC with the fixed-point bit-wise compressor (Sec. 3.1).
//
// Entries are divided by the largest magnitude of the worker's gradient and written as a sign plus
// B fractional bits (Eq. 6 with B = b_{L-1} <= 23 instead of 63, since the input is fp32/bf16):
//   e = fl32(|g| / gmax),  q = min(floor(e 2^B), 2^B - 1).
// Level l keeps the top b_l bits of q; the residual C^l - C^{l-1} is the field
//   f_l = (q >> (B - b_l)) & (2^{w_l} - 1),  w_l = b_l - b_{l-1},  worth  sign f_l 2^{-b_l} gmax,
// sent as one sign plane and w_l magnitude planes.  Adaptive probabilities (Lemma 3.4) use the exact
// integer field energies S_l = sum_i f_l^2:  Delta_l = gmax 2^{-b_l} sqrt(S_l).
#include "dense_cluster.cuh"

namespace mlmc {

namespace {

constexpr int kBitThreads = 256;

struct BitSchedule {
    int L;
    int B;
    int shift[kMaxLevels];      // B - b_l
    int width[kMaxLevels];      // w_l
    int bits[kMaxLevels];       // b_l
    // levels of at most 8 bits in runs of at most 8 bits together
    uint32_t run_up[kMaxLevels];  // moves the run to the top byte of the code: 2^(24 - B + b of its last level)
    int in_run[kMaxLevels];       // the last level's b - b_l: where the field sits in the byte
    uint32_t mask4[kMaxLevels];   // the field's bits, in every byte
};

// The code of an entry at b bits, min(trunc(e 2^b), 2^b - 1) with the IEEE-rounded fp32 quotient e = fl32(|g| / gmax).  (The
// top bits of a longer code are the shorter code: both truncate the same e.)
// The divisor is fixed, so the quotient comes from its correctly rounded reciprocal by two correction steps (Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor", 1990: with the reciprocal correctly rounded
// and a quotient within one ulp, one step of remainder and correction rounds like the division).  The truncation is the
// addition of 2^23 with rounding toward zero.  (The fp64 product and conversions used before took two slots of the conversion
// unit.)  The remainders must not underflow and the reciprocal must be normal: where gmax lies
// outside [2^-60, 2^100], numerator and divisor are moved by a power of two.  (That is exact, except for numerators whose
// quotient lies far below 2^-23: their code is 0 either way.)
// The operations are done on pairs of entries (packed fp32 instructions round like the single ones): they are what binds the kernels,
// by issue.  Only |g| = gmax has the quotient 1, so that the limit is taken where a group's largest entry says so.
struct Quantiser {
    float gmax, inv, move;
    int top;  // bits of the largest magnitude
    __device__ __forceinline__ explicit Quantiser(float g) {
        top = __float_as_int(g);
        gmax = g > 0.0f ? g : 1.0f;
        move = gmax < 0x1.0p-60f ? 0x1.0p100f : gmax > 0x1.0p100f ? 0x1.0p-64f : 1.0f;
        gmax *= move;
        inv = __frcp_rn(gmax);
    }
    // The codes of N entries at b bits (scale 2^b, b <= 23): in the low 23 bits, the bits of 2^23 above.  limit: gmax may be among them.
    template <int N>
    __device__ __forceinline__ void codes(const float (&v)[N], float scale, bool limit, uint32_t (&q)[N]) const {
        static_assert(N % 2 == 0, "pairs");
        if (move != 1.0f) {
            float x[N];
#pragma unroll
            for (int i = 0; i < N; ++i) x[i] = v[i] * move;
            quotients(x, scale, q);
        } else {
            quotients(v, scale, q);
        }
        if (limit) {  // e = 1 has no b-bit fraction: the largest e below it has the code 2^b - 1
            const uint32_t most = __float_as_uint(8388608.0f + scale) - 1u;
#pragma unroll
            for (int i = 0; i < N; ++i) q[i] = min(q[i], most);
        }
    }
    template <int N>
    __device__ __forceinline__ void quotients(const float (&v)[N], float scale, uint32_t (&q)[N]) const {
        const uint64_t inv2 = pair(inv, inv), minus2 = pair(-gmax, -gmax), scale2 = pair(scale, scale), one2 = pair(8388608.0f, 8388608.0f);
#pragma unroll
        for (int i = 0; i < N; i += 2) {
            const uint64_t x = pair(fabsf(v[i]), fabsf(v[i + 1]));
            uint64_t e = mul_pair(x, inv2);
            e = fma_pair(fma_pair(e, minus2, x), inv2, e);
            e = fma_pair(fma_pair(e, minus2, x), inv2, e);
            e = fma_pair_toward_zero(e, scale2, one2);
            q[i] = (uint32_t)e;
            q[i + 1] = (uint32_t)(e >> 32);
        }
    }
};

// An entry below gmax 2^-b (1 - 2^-20) has fl32(|g| / gmax) < 2^-b: its code at b bits is 0.
__device__ __forceinline__ int zero_code_below(float gmax, int b) {
    return gmax > 0.0f ? __float_as_int(gmax * ldexpf(1.0f - 0x1.0p-20f, -b)) : 0x7FFFFFFF;
}

// The sign words of a batch (four vectors per lane): from the nibble (bf16: byte) of signs of every vector, in the word's order.
// Lanes that hold pieces of one word hold pieces of the words of all four vectors; they exchange them so that every lane
// is left with one word (fp32: every second quartet of lanes holds a copy).
template <typename T>
__device__ __forceinline__ void write_signs(const uint4 (&q)[4], uint32_t* __restrict__ out) {
    const int lane = threadIdx.x & 31;
    uint32_t x[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t s = 0;
        if constexpr (sizeof(T) == 4) {
            s = __funnelshift_l(q[j].w, s, 1);
            s = __funnelshift_l(q[j].z, s, 1);
            s = __funnelshift_l(q[j].y, s, 1);
            s = __funnelshift_l(q[j].x, s, 1);
            x[j] = s << (4 * (lane & 7));
        } else {
            auto two = [](uint32_t w) { return ((w >> 15) & 1u) | ((w >> 30) & 2u); };
            s = two(q[j].x) | two(q[j].y) << 2 | two(q[j].z) << 4 | two(q[j].w) << 6;
            x[j] = s << (8 * (lane & 3));
        }
    }
    const bool odd = lane & 1, high = lane & 2;
    uint32_t a = odd ? x[1] : x[0], b = odd ? x[3] : x[2];
    a |= __shfl_xor_sync(0xFFFFFFFFu, odd ? x[0] : x[1], 1);
    b |= __shfl_xor_sync(0xFFFFFFFFu, odd ? x[2] : x[3], 1);
    uint32_t w = high ? b : a;
    w |= __shfl_xor_sync(0xFFFFFFFFu, high ? a : b, 2);
    const int j = lane & 3;  // of vector j
    if constexpr (sizeof(T) == 4) {
        w |= __shfl_xor_sync(0xFFFFFFFFu, w, 4);
        if (!(lane & 4)) out[4 * j + (lane >> 3)] = w;
    } else {
        out[8 * j + (lane >> 2)] = w;
    }
}

// ---- per-worker max |g| as an integer max over magnitude keys; flags NaN / Inf.  With given probabilities (draw != 0)
// the worker's last block also draws the level and writes the message header.
// KEEP 1: the smallest of the batches' largest keys too, behind the workers' largest keys in gmax_bits (a row of one scale has no batch
// that rounds to 0 at any level, and its message is written without a look at them).
// KEEP 1 and 2: the largest key of every batch (kEmitGroupVecs vectors, a warp's share of a trip) is kept, and the kernels that write
// the message do not read the batches that round to 0 at the drawn level.  KEEP 2: what they would miss of those, the sign plane
// of a bit-plane message, is written here too.  8 x 124M fp32 entries: 560, 566 and 620 us; what it saves the message kernels is
// beside them.  KEEP 0, for calls that L2 holds (8 x 1M entries, bit planes: 32.2 us per step, with 2 33.4).
template <typename T, int KEEP>
__global__ void __launch_bounds__(kSweepThreads, 3)
absmax_kernel(const T* __restrict__ g, int64_t d, int64_t ld, uint32_t* gmax_bits, uint32_t* acc, uint32_t* done,
              uint32_t* __restrict__ batch_max, int batches_per_worker, uint32_t* __restrict__ planes, int64_t plane_row,
              const __grid_constant__ DrawPlan pl, const __grid_constant__ DrawnLevels drawn, int draw, int* status, int* worker_err) {
    using Tr = ElemTraits<T>;
    __shared__ uint32_t sh_max[kSweepThreads / 32], sh_min[kSweepThreads / 32];
    pdl_enter();
    const int m = blockIdx.y, lane = threadIdx.x & 31;
    const T* row = g + (int64_t)m * ld;
    uint32_t mx = 0, mn = 0xFFFFFFFFu;
    const int64_t nvec = (d + Tr::kVec - 1) / Tr::kVec, full_end = d / Tr::kVec;  // vectors of the row, and those wholly inside it
    if constexpr (KEEP == 0) {
        // Chunks of kBatch vectors per thread, all in flight before any is used, dealt round-robin to the blocks of the worker.
        // (One contiguous range per block ran between 0.75 and 1.0 of the copy rate, depending on the row length.)
        constexpr int kBatch = 4;
        for (int64_t base = (int64_t)blockIdx.x * kBatch * kSweepThreads; base < nvec; base += (int64_t)gridDim.x * kBatch * kSweepThreads) {
            const int64_t v = base + threadIdx.x;
            if (base + kBatch * kSweepThreads > full_end) {  // the row's last chunk
                for (int64_t u = v; u < nvec; u += kSweepThreads)
                    for_each_in_vector<T>(row, u, d, [&](int64_t, uint32_t bits) { mx = max(mx, Tr::key(bits)); });
                break;
            }
            uint4 q[kBatch];
#pragma unroll
            for (int j = 0; j < kBatch; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + v + j * kSweepThreads);
#pragma unroll
            for (int j = 0; j < kBatch; ++j) {
                if constexpr (Tr::kVec == 4) {
                    mx = max(max(mx, q[j].x & 0x7FFFFFFFu), max(q[j].y & 0x7FFFFFFFu, max(q[j].z & 0x7FFFFFFFu, q[j].w & 0x7FFFFFFFu)));
                } else {
                    const uint32_t a = __vmaxu2(__vmaxu2(q[j].x & 0x7FFF7FFFu, q[j].y & 0x7FFF7FFFu),
                                                __vmaxu2(q[j].z & 0x7FFF7FFFu, q[j].w & 0x7FFF7FFFu));
                    mx = max(mx, max(a & 0xFFFFu, a >> 16));
                }
            }
        }
    } else {
        // A batch per warp and trip, all four vectors in flight before any is used, dealt round-robin to the blocks of the worker.
        uint32_t* bmax = batch_max + (int64_t)m * batches_per_worker;
        const int64_t nbatch = (nvec + kEmitGroupVecs - 1) / kEmitGroupVecs, stride = (int64_t)gridDim.x * (kSweepThreads / 32);
        for (int64_t b = (int64_t)blockIdx.x * (kSweepThreads / 32) + (threadIdx.x >> 5); b < nbatch; b += stride) {
            const int64_t v = b * kEmitGroupVecs + lane;
            uint32_t vm = 0;
            if ((b + 1) * kEmitGroupVecs > full_end) {  // the row's last batch; its signs are left to the message kernel
                for (int64_t u = v; u < nvec; u += 32)
                    for_each_in_vector<T>(row, u, d, [&](int64_t, uint32_t bits) { vm = max(vm, Tr::key(bits)); });
            } else {
                uint4 q[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + v + j * 32);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    if constexpr (Tr::kVec == 4) {
                        vm = max(max(vm, q[j].x & 0x7FFFFFFFu), max(q[j].y & 0x7FFFFFFFu, max(q[j].z & 0x7FFFFFFFu, q[j].w & 0x7FFFFFFFu)));
                    } else {
                        const uint32_t a = __vmaxu2(__vmaxu2(q[j].x & 0x7FFF7FFFu, q[j].y & 0x7FFF7FFFu),
                                                    __vmaxu2(q[j].z & 0x7FFF7FFFu, q[j].w & 0x7FFF7FFFu));
                        vm = max(vm, max(a & 0xFFFFu, a >> 16));
                    }
                }
                if (KEEP == 2) write_signs<T>(q, planes + (int64_t)m * plane_row + b * (kEmitGroupVecs * Tr::kVec / 32));
            }
            vm = __reduce_max_sync(0xFFFFFFFFu, vm);
            if (lane == 0) bmax[b] = Tr::kVec == 8 ? vm << 16 : vm;  // as the bits of an fp32 magnitude
            mx = max(mx, vm);
            if (KEEP == 1) mn = min(mn, vm);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if ((threadIdx.x & 31) == 0) {
        sh_max[threadIdx.x >> 5] = mx;
        if (KEEP == 1) sh_min[threadIdx.x >> 5] = mn;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < kSweepThreads / 32; ++w) mx = max(mx, sh_max[w]);
        atomicMax(&acc[m], mx);
        if (KEEP == 1) {
            for (int w = 1; w < kSweepThreads / 32; ++w) mn = min(mn, sh_min[w]);
            atomicMax(&acc[gridDim.y + m], ~mn);
        }
    }
    if (!last_block(&done[m], gridDim.x) || threadIdx.x != 0) return;
    mx = __ldcg(&acc[m]);
    acc[m] = 0u;
    const uint32_t as_f32 = (Tr::kVec == 8) ? (mx << 16) : mx;
    gmax_bits[m] = as_f32;
    if (KEEP == 1) {
        mn = ~__ldcg(&acc[gridDim.y + m]);
        acc[gridDim.y + m] = 0u;
        gmax_bits[gridDim.y + m] = (Tr::kVec == 8) ? (mn << 16) : mn;
    }
    if (mx >= Tr::kInfKey) {
        worker_err[m] = MLMC_ERR_NONFINITE;
        set_status(status, MLMC_ERR_NONFINITE);
        void_header(pl, m);
    } else {
        worker_err[m] = 0;
        if (draw) write_header(pl, m, drawn.level[m], drawn.p[drawn.level[m]], __uint_as_float(as_f32), status, worker_err);
    }
}

// ---- adaptive only: exact field energies S_l = sum_i f_l^2 for every level in one sweep; the worker's last block turns
// them into probabilities, draws the level and writes the message header.
// Acc = uint32_t when every field is at most 8 bits wide and a thread sees fewer than 2^16 entries (f^2 < 2^16,
// so the sum fits 32 bits), else unsigned long long.  Fields come from the prefix codes P_l = q >> (B - b_l):
// f_l = P_l - (P_{l-1} << w_l), one shift and one multiply-add per level.
// A warp takes its entries level by level, kBitHeld per lane, from the first level at which the largest of them has a code
// above 0 (the coarse levels of a gradient with per-layer scales are nearly all zero).  Fields of at most 8 bits are summed
// four entries per instruction: levels that share a byte (1, 1, 2 and 4 bits, say) are packed into words of four entries
// once, then a level is a mask and a byte product.  Shifts are multiplications where they can be: the shifter and the logic
// share a pipe of half the rate, which bound the kernel.  8 x 124M fp32 entries, six
// levels: 1.0 ms with every entry taken through every level and the fp64 quotient, 0.82 field by field, 0.70 with single quotients, now
// 0.66 (0.62 is the first sweep of the same row; bf16 codes of 36M x 16: 0.55 -> 0.37).
constexpr int kBitHeld = 8;

template <typename T, int LMAX, typename Acc>
__device__ __forceinline__ void take_fields(const float (&v)[kBitHeld], const Quantiser& qz, float scale, const int (&zero_below)[LMAX],
                                            const BitSchedule& sc, Acc (&acc)[LMAX]) {
    float top = 0.0f;
#pragma unroll
    for (int e = 0; e < kBitHeld; ++e) top = fmaxf(top, fabsf(v[e]));
    const int mx = __reduce_max_sync(0xFFFFFFFFu, __float_as_int(top));
    if (mx < zero_below[LMAX - 1]) return;  // the thresholds fall with the level; those past L repeat the last
    if constexpr (sizeof(Acc) == 4) {
        uint32_t q[kBitHeld], w[kBitHeld / 4];
        uint32_t run = 0u;
        qz.codes(v, scale, mx == qz.top, q);
#pragma unroll
        for (int l = 0; l < LMAX; ++l) {
            if (l >= sc.L) break;
            if (mx < zero_below[l]) continue;
            if (sc.run_up[l] != run) {  // the byte of the run of every entry, four per word
                run = sc.run_up[l];
#pragma unroll
                for (int e = 0; e < kBitHeld; e += 4)
                    w[e / 4] = __byte_perm(__byte_perm(q[e] * run, q[e + 1] * run, 0x0073),
                                           __byte_perm(q[e + 2] * run, q[e + 3] * run, 0x0073), 0x5410);
            }
#pragma unroll
            for (int e = 0; e < kBitHeld / 4; ++e) {  // the field stays where it is: its square counts 2^(2 in_run)
                const uint32_t f = w[e] & sc.mask4[l];
                acc[l] = __dp4a(f, f, acc[l]);
            }
        }
    } else {
        uint32_t q[kBitHeld], prev[kBitHeld];
        qz.codes(v, scale, mx == qz.top, q);
#pragma unroll
        for (int e = 0; e < kBitHeld; ++e) {
            q[e] -= 0x4B000000u;
            prev[e] = 0u;
        }
#pragma unroll
        for (int l = 0; l < LMAX; ++l) {
            if (l >= sc.L) break;
            if (mx < zero_below[l]) continue;
            const int shift = sc.shift[l];
            const uint32_t neg_pow = 0u - (1u << sc.width[l]);
#pragma unroll
            for (int e = 0; e < kBitHeld; ++e) {
                const uint32_t P = q[e] >> shift, f = prev[e] * neg_pow + P;
                acc[l] += (Acc)f * f;
                prev[e] = P;
            }
        }
    }
}

template <typename T>
__device__ __forceinline__ void expand_vectors(const uint4* q, float (&v)[kBitHeld]) {  // kBitHeld entries
#pragma unroll
    for (int j = 0; j < kBitHeld / ElemTraits<T>::kVec; ++j) {
        const uint32_t w[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (ElemTraits<T>::kVec == 4) {
                v[4 * j + i] = __uint_as_float(w[i]);
            } else {
                v[8 * j + 2 * i] = __uint_as_float(w[i] << 16);
                v[8 * j + 2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
            }
        }
    }
}

template <typename T, int LMAX, typename Acc>
__global__ void __launch_bounds__(kSweepThreads, LMAX <= 8 ? 2 : 1)
bit_stats_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const uint32_t* gmax_bits, const __grid_constant__ BitSchedule sc,
                 unsigned long long* S_partial, int stat_ctas, uint32_t* done, const __grid_constant__ DrawPlan pl, int* status, int* worker_err) {
    using Tr = ElemTraits<T>;
    __shared__ unsigned long long sh_red[LMAX][kSweepThreads / 32];
    __shared__ double sh_delta[kMaxLevels];
    pdl_enter();
    const int m = blockIdx.y;
    if (worker_err[m]) return;
    const float gmax = __uint_as_float(gmax_bits[m]);
    const Quantiser qz(gmax);
    const float scale = (float)(1u << sc.B);
    Acc acc[LMAX];
    int zero_below[LMAX];
#pragma unroll
    for (int l = 0; l < LMAX; ++l) {
        acc[l] = 0;
        zero_below[l] = zero_code_below(gmax, sc.bits[min(l, sc.L - 1)]);
    }
    if (gmax > 0.0f) {
        const T* row = g + (int64_t)m * ld;
        constexpr int kVecs = kBitHeld / Tr::kVec;  // 16-byte vectors per lane and trip; the next trip's are in flight
        constexpr int kTrip = kSweepThreads * kVecs;
        const int64_t trips = d / Tr::kVec / kTrip;
        uint4 nxt[kVecs];
        auto load = [&](int64_t trip) {
            if (trip >= trips) return;
#pragma unroll
            for (int j = 0; j < kVecs; ++j)
                nxt[j] = __ldg(reinterpret_cast<const uint4*>(row) + trip * kTrip + j * kSweepThreads + threadIdx.x);
        };
        load(blockIdx.x);
        for (int64_t trip = blockIdx.x; trip < trips; trip += gridDim.x) {
            float v[kBitHeld];
            expand_vectors<T>(nxt, v);
            load(trip + gridDim.x);
            take_fields<T, LMAX, Acc>(v, qz, scale, zero_below, sc, acc);
        }
        if (blockIdx.x == gridDim.x - 1) {  // the rest of the row; entries past it read as 0, which adds nothing
            for (int64_t i0 = trips * kTrip * Tr::kVec; i0 < d; i0 += (int64_t)kSweepThreads * kBitHeld) {
                float v[kBitHeld];
#pragma unroll
                for (int e = 0; e < kBitHeld; ++e) {
                    const int64_t i = i0 + e * kSweepThreads + threadIdx.x;
                    v[e] = 0.0f;
                    if (i < d) {
                        if constexpr (Tr::kVec == 4) v[e] = reinterpret_cast<const float*>(row)[i];
                        else v[e] = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(row)[i] << 16);
                    }
                }
                take_fields<T, LMAX, Acc>(v, qz, scale, zero_below, sc, acc);
            }
        }
    }
#pragma unroll
    for (int l = 0; l < LMAX; ++l) {
        if (l >= sc.L) break;
        unsigned long long x = (unsigned long long)(sizeof(Acc) == 4 ? acc[l] >> (2 * sc.in_run[l]) : acc[l]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
        if ((threadIdx.x & 31) == 0) sh_red[l][threadIdx.x >> 5] = x;
    }
    __syncthreads();
    if (threadIdx.x < sc.L) {
        unsigned long long s = 0;
#pragma unroll
        for (int w = 0; w < kSweepThreads / 32; ++w) s += sh_red[threadIdx.x][w];
        S_partial[((int64_t)m * stat_ctas + blockIdx.x) * kMaxLevels + threadIdx.x] = s;
    }
    if (!last_block(&done[m], gridDim.x)) return;
    // exact 128-bit sums of the per-block partials (integer adds: any order), rounded once to fp64; a warp per level
    const int lane = threadIdx.x & 31;
    for (int l = threadIdx.x >> 5; l < sc.L; l += kSweepThreads / 32) {
        unsigned __int128 S = 0;
        for (int c = lane; c < (int)gridDim.x; c += 32) S += __ldcg(&S_partial[((int64_t)m * stat_ctas + c) * kMaxLevels + l]);
        unsigned long long lo = (unsigned long long)S, hi = (unsigned long long)(S >> 64);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long lo2 = __shfl_xor_sync(0xFFFFFFFFu, lo, o), hi2 = __shfl_xor_sync(0xFFFFFFFFu, hi, o);
            const unsigned __int128 t = (((unsigned __int128)hi << 64) | lo) + (((unsigned __int128)hi2 << 64) | lo2);
            lo = (unsigned long long)t;
            hi = (unsigned long long)(t >> 64);
        }
        if (lane == 0) sh_delta[l] = (double)gmax * ldexp(1.0, -sc.bits[l]) * sqrt((double)hi * 0x1.0p64 + (double)lo);
    }
    __syncthreads();
    finish_levels(pl, m, sh_delta, gmax, status, worker_err);
}

// ---- pack: a warp turns 1024 consecutive entries into 32 words of each plane, a lane owning 32 consecutive entries (one
// word per plane).  The entries come through one or two slots of shared memory per warp: a slot takes its next group's copy when the
// group before it is in registers, and the copy is in flight while that is coded.  A plane's word is collected by one shift and one
// funnel shift per entry, from 6 planes on by one bit transpose for all of them.  A group whose largest entry has the code 0 at the drawn
// level's bits is not coded: its magnitude planes are zero.  The groups of which the sweep before knows that are not even read (8 x 124M
// fp32 entries with layers: 782 -> 424 us).  Calls that read everything have three blocks per SM and one slot per warp (8 x 3M 53.6 us
// per step, 55.5 with four blocks); for the others see launch_bit_pack_t.
// Bound by HBM.  Rows of 32 entries across the lanes with a ballot each took 1.04 ms for 8 x 124M fp32 entries.
// after_read: called when the lane has its entries of the group in registers.
template <typename T, typename F>
__device__ __forceinline__ void pack_group(const uint32_t* slot, const Quantiser& qz, float scale, int zero_below, int w, int64_t word,
                                           int64_t words, uint32_t* __restrict__ out, bool signs, F&& after_read) {
    const int lane = threadIdx.x & 31;
    const bool live = word < words;
    float x[32];
#pragma unroll
    for (int c = 0; c < kGroupChunks<T>; ++c) {
        const uint4 q = *reinterpret_cast<const uint4*>(slot + group_place<T>(lane, c));
        const uint32_t u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if constexpr (sizeof(T) == 4) {
                x[4 * c + i] = __uint_as_float(u[i]);
            } else {
                x[8 * c + 2 * i] = __uint_as_float(u[i] << 16);
                x[8 * c + 2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
            }
        }
    }
    after_read();
    uint32_t sign_w = 0;
    float mx = 0.0f;
#pragma unroll
    for (int t = 31; t >= 0; --t) {
        sign_w = __funnelshift_l(__float_as_uint(x[t]), sign_w, 1);
        mx = fmaxf(mx, fabsf(x[t]));
    }
    if (live && signs) out[word] = sign_w;
    if (!__any_sync(0xFFFFFFFFu, __float_as_int(mx) >= zero_below)) {
        if (live)
            for (int j = 1; j <= w; ++j) out[(int64_t)j * words + word] = 0u;
        return;
    }
    uint32_t q[32];
    // the bits above a field leave with the shifts, or are planes that are not written
    qz.codes(x, scale, __any_sync(0xFFFFFFFFu, __float_as_int(mx) == qz.top), q);
    if (w < 6) {
        for (int j = 1; j <= w; ++j) {
            const int up = 31 - (w - j);
            uint32_t pw = 0;
#pragma unroll
            for (int t = 31; t >= 0; --t) pw = __funnelshift_l(q[t] << up, pw, 1);
            if (live) out[(int64_t)j * words + word] = pw;
        }
    } else {
        transpose_bits(q);
#pragma unroll
        for (int bit = 22; bit >= 0; --bit)
            if (live && bit < w) out[(int64_t)(w - bit) * words + word] = q[bit];
    }
}

template <typename T, bool SKIP, int BLOCKS>
constexpr int kPackSlots = SKIP && (BLOCKS == 3 || sizeof(T) == 2) ? 2 : 1;  // groups in flight per warp; four blocks of fp32 have room for one

template <typename T, bool SKIP, int BLOCKS>  // BLOCKS: per SM
__global__ void __launch_bounds__(kBitThreads, BLOCKS)
bit_pack_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const uint32_t* gmax_bits, BitSchedule sc,
                const int32_t* bit_level, const uint32_t* batch_max, int batches_per_worker, uint32_t* __restrict__ planes, int w_max,
                int64_t words) {
    extern __shared__ __align__(16) uint32_t sh_ring[];  // [warps][SLOTS][kGroupSlot]
    pdl_enter();
    const int m = blockIdx.y;
    const int level = bit_level[m];
    if (level < 0) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ngroups = (words + 31) / 32;
    const float gmax = __uint_as_float(gmax_bits[m]);
    const Quantiser qz(gmax);
    const int w = sc.width[level], bits = sc.bits[level];
    const int zero_below = zero_code_below(gmax, bits);
    const float scale = (float)(1u << bits);
    const T* row = g + (int64_t)m * ld;
    uint32_t* out = planes + (int64_t)m * (1 + w_max) * words;
    constexpr int SLOTS = kPackSlots<T, SKIP, BLOCKS>;
    uint32_t* ring = sh_ring + warp * SLOTS * kGroupSlot<T>;
    const int64_t stride = (int64_t)gridDim.x * (blockDim.x / 32);
    if constexpr (!SKIP) {
        int64_t grp = (int64_t)blockIdx.x * (blockDim.x / 32) + warp;
        fetch_group<T>(row, d, grp, ngroups, ring);
        for (; grp < ngroups; grp += stride) {
            cp_async_wait<0>();
            __syncwarp();
            pack_group<T>(ring, qz, scale, zero_below, w, grp * 32 + lane, words, out, true, [&]() {
                __syncwarp();  // the slot has been read by every lane
                fetch_group<T>(row, d, grp + stride, ngroups, ring);
            });
        }
    } else {
        constexpr int kPer = 2 * (int)sizeof(T) / 4;  // batches of a group: 2 or 1
        const uint32_t* bmax = batch_max + (int64_t)m * batches_per_worker;
        // A lane looks at the largest key of one of the warp's next 32 groups.
        for (int64_t base = (int64_t)blockIdx.x * (blockDim.x / 32) + warp; base < ngroups; base += 32 * stride) {
            const int64_t own = base + lane * stride;
            bool coded = false;
            if (own < ngroups) {
                coded = (own + 1) * 1024 > d;  // the ragged end: its signs are not written yet
                if (!coded) {
                    uint32_t mx = bmax[own * kPer];
                    if (kPer == 2) mx = max(mx, bmax[own * kPer + 1]);
                    coded = (int)mx >= zero_below;
                }
            }
            uint32_t todo = __ballot_sync(0xFFFFFFFFu, coded), zero = __ballot_sync(0xFFFFFFFFu, own < ngroups && !coded);
            auto next = [&]() -> int64_t {
                if (!todo) return ngroups;
                const int64_t grp = base + (__ffs(todo) - 1) * stride;
                todo &= todo - 1u;
                return grp;
            };
            int64_t grp[SLOTS];
#pragma unroll
            for (int i = 0; i < SLOTS; ++i) {
                grp[i] = next();
                fetch_group<T>(row, d, grp[i], ngroups, ring + i * kGroupSlot<T>);
            }
            for (; zero; zero &= zero - 1u) {  // magnitude planes of zeros, while the first group is on its way
                uint32_t* to = out + (base + (__ffs(zero) - 1) * stride) * 32 + lane;
                for (int j = 1; j <= w; ++j) to[(int64_t)j * words] = 0u;
            }
            for (int at = 0; grp[0] < ngroups; at = SLOTS == 1 ? 0 : at ^ kGroupSlot<T>) {
                const int64_t after = next();
                cp_async_wait<SLOTS - 1>();
                __syncwarp();
                pack_group<T>(ring + at, qz, scale, zero_below, w, grp[0] * 32 + lane, words, out, (grp[0] + 1) * 1024 > d, [&]() {
                    __syncwarp();  // the slot has been read by every lane
                    fetch_group<T>(row, d, after, ngroups, ring + at);
                });
                if (SLOTS == 2) grp[0] = grp[SLOTS - 1];
                grp[SLOTS - 1] = after;
            }
        }
    }
    cp_async_wait<0>();
}

// ---- short rows: all of the above in one launch (dense_cluster.cuh).  Fields of at most 8 bits, at most kDenseLevels levels.
// 6 x 400,003 bf16 entries, six levels, adaptive: 22 us for the three kernels above, 15 for this one, now 13.5.
constexpr int kBitDenseWarps = 32;

template <typename T>
__global__ void __launch_bounds__(kBitDenseWarps * 32, 1)
bit_cluster_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const __grid_constant__ BitSchedule sc,
                   const __grid_constant__ DrawPlan pl, const __grid_constant__ DrawnLevels drawn, int adaptive, int per_block,
                   uint32_t* __restrict__ planes, int w_max, int64_t words, int* status, int* worker_err) {
    using Tr = ElemTraits<T>;
    extern __shared__ __align__(16) uint32_t sh_slots[];
    __shared__ DenseShared<kBitDenseWarps, unsigned long long> sh;
    __shared__ int sh_below[kDenseLevels];
    cg::cluster_group cluster = cg::this_cluster();
    pdl_enter();
    const int rank = (int)cluster.block_rank(), m = blockIdx.x / (int)cluster.num_blocks();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t ngroups = (words + 31) / 32, g0 = (int64_t)rank * per_block;
    const int n = (int)max((int64_t)0, min((int64_t)per_block, ngroups - g0));
    const uint32_t top = dense_load<T>(cluster, g + (int64_t)m * ld, d, g0, n, sh_slots, sh);
    const bool bad = top >= Tr::kInfKey, first = rank == 0;
    if (first && threadIdx.x == 0) {
        worker_err[m] = bad ? MLMC_ERR_NONFINITE : 0;
        if (bad) {
            set_status(status, MLMC_ERR_NONFINITE);
            void_header(pl, m);
        }
    }
    if (bad) return;  // the same in every block
    const float gmax = __uint_as_float(Tr::kVec == 8 ? top << 16 : top);
    const Quantiser qz(gmax);
    double delta = 0.0;
    if (adaptive) {
        if (threadIdx.x < kDenseLevels) sh_below[threadIdx.x] = zero_code_below(gmax, sc.bits[min((int)threadIdx.x, sc.L - 1)]);
        __syncthreads();
        uint32_t acc[kDenseLevels];
        int zero_below[kDenseLevels];
#pragma unroll
        for (int l = 0; l < kDenseLevels; ++l) {
            acc[l] = 0u;
            zero_below[l] = sh_below[l];
        }
        if (gmax > 0.0f) {
            constexpr int kVecs = kBitHeld / Tr::kVec;  // a warp takes a quarter of a group
#pragma unroll 1
            for (int u = warp; u < 4 * n; u += kBitDenseWarps) {
                const uint4* x = reinterpret_cast<const uint4*>(sh_slots + (u >> 2) * kGroupSlot<T>) + (u & 3) * kVecs * 32 + lane;
                uint4 q[kVecs];
#pragma unroll
                for (int j = 0; j < kVecs; ++j) q[j] = x[j * 32];
                float v[kBitHeld];
                expand_vectors<T>(q, v);
                take_fields<T, kDenseLevels, uint32_t>(v, qz, (float)(1u << sc.B), zero_below, sc, acc);
            }
        }
#pragma unroll
        for (int l = 0; l < kDenseLevels; ++l) acc[l] >>= 2 * sc.in_run[l];
        const unsigned long long S = dense_sums(cluster, acc, sh);
        if (threadIdx.x < sc.L) delta = (double)gmax * ldexp(1.0, -sc.bits[threadIdx.x]) * sqrt((double)S);
    }
    double p;
    const int level = dense_level(pl, drawn, adaptive, m, first, delta, gmax, sh, &p, status, worker_err);
    if (sc.width[level] > w_max) return;  // reported with the header
    const float scale = (float)(1u << sc.bits[level]);
    const int zero_below = zero_code_below(gmax, sc.bits[level]);
    uint32_t* out = planes + (int64_t)m * (1 + w_max) * words;
    for (int i = warp; i < n; i += kBitDenseWarps)
        pack_group<T>(sh_slots + i * kGroupSlot<T>, qz, scale, zero_below, sc.width[level], (g0 + i) * 32 + lane, words, out, true, []() {});
}

// ---- server average of bit-plane messages.  8 x 124M entries, six levels: 372 us with one worker in flight, now 250.
constexpr int kAvgBitRows = 1 + kAvgPlanes;
constexpr int kAvgBitWords = kAvgSlots * kAvgBitRows * 32 > kAvgStage ? kAvgSlots * kAvgBitRows * 32 : kAvgStage;  // per warp
constexpr size_t kAvgBitSmem = (size_t)kAvgBitWords * (kAvgThreads / 32) * 4;

__global__ void __launch_bounds__(kAvgThreads)
aggregate_bitwise_kernel(const uint32_t* __restrict__ planes, const float* gmax, const int32_t* level, const double* p_sel,
                         const __grid_constant__ BitSchedule sc, int w_max, int64_t words, int M, int64_t d, float* __restrict__ out) {
    extern __shared__ __align__(16) uint32_t sh_ring[];  // [warps][kAvgSlots][kAvgBitRows][32], units and levels
    float* sh_unit = reinterpret_cast<float*>(sh_ring + kAvgThreads / 32 * kAvgBitWords);  // value of one unit of the field: 2^{-b_l} gmax / p_l
    int* sh_level = reinterpret_cast<int*>(sh_unit + M);
    pdl_enter();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t* ring = sh_ring + warp * kAvgBitWords;
    const float inv_M = 1.0f / (float)M;
    const int64_t nblk = (words + kAvgThreads - 1) / kAvgThreads;
    for (int64_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        const int64_t word = blk * kAvgThreads + threadIdx.x, at = min(word, words - 1);  // lanes past the end repeat the last word
        float acc[32];
#pragma unroll
        for (int t = 0; t < 32; ++t) acc[t] = 0.0f;
        auto fetch = [&](int m) {  // the sign word to row 0, bit k of the fields (plane w - k) to row 1 + k
            const int lv = m < M ? __ldg(&level[m]) : -1;
            if (lv >= 0) {
                const int w = sc.width[lv];
                const uint32_t* from = planes + (int64_t)m * (1 + w_max) * words + at;
                uint32_t* to = ring + (m & (kAvgSlots - 1)) * kAvgBitRows * 32 + lane;
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
                sh_unit[m] = lv >= 0 ? (float)(ldexp((double)gmax[m], -sc.bits[lv]) / p_sel[m]) : 0.0f;
            }
            __syncthreads();
        }
        for (int m = 0; m < M; ++m) {  // fixed worker order
            fetch(m + kAvgSlots - 1);
            cp_async_wait<kAvgSlots - 1>();
            const int lv = sh_level[m];
            if (lv < 0) continue;
            const int w = sc.width[lv];
            const float unit = sh_unit[m];
            const uint32_t* from = ring + (m & (kAvgSlots - 1)) * kAvgBitRows * 32 + lane;
            const uint32_t sgn = from[0];
            if (w <= kAvgPlanes && fabsf(unit) < 0x1p100f) {
                uint32_t fb[8], any = 0u;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    fb[k] = k < w ? from[(1 + k) * 32] : 0u;
                    any |= fb[k];
                }
                // A word whose fields are all zero adds +-0 to every entry, which changes nothing.  The high levels of a
                // heavy-tailed gradient are almost all zero, so whole warps skip.
                if (any != 0u) {
                    fields_to_bytes(fb);
                    const float offset = -8388608.0f * unit;
#pragma unroll
                    for (int t = 0; t < 32; ++t)
                        acc[t] += __uint_as_float(__float_as_uint(field_times(fb, t, unit, offset)) ^ ((sgn << (31 - t)) & 0x80000000u));
                }
            } else {
                uint32_t f[32];
                gather_fields<1>(planes + ((int64_t)m * (1 + w_max) + 1) * words + at, words, w, f);
#pragma unroll
                for (int t = 0; t < 32; ++t) {
                    const float ff = __uint_as_float(0x4B000000u | f[t]) - 8388608.0f;  // f < 2^23: exact
                    acc[t] += __uint_as_float(__float_as_uint(ff * unit) ^ ((sgn << (31 - t)) & 0x80000000u));
                }
            }
        }
        cp_async_wait<0>();
        store_words(ring, acc, inv_M, blk * kAvgThreads + warp * 32, d, out);
    }
}


BitSchedule make_schedule(const int32_t* b, int L) {
    BitSchedule sc = {};
    sc.L = L;
    sc.B = b[L - 1];
    for (int l = 0; l < L; ++l) {
        const int w = b[l] - (l ? b[l - 1] : 0);
        sc.bits[l] = b[l];
        sc.width[l] = w;
        sc.shift[l] = sc.B - b[l];
    }
    for (int l = 0, end; l < L; l = end) {
        for (end = l + 1; end < L && b[end] - (l ? b[l - 1] : 0) <= 8;) ++end;
        for (int i = l; i < end; ++i) {
            sc.run_up[i] = 1u << (24 - sc.B + b[end - 1]);
            sc.in_run[i] = b[end - 1] - b[i];
            sc.mask4[i] = ((((1u << sc.width[i]) - 1u) << sc.in_run[i]) & 0xFFu) * 0x01010101u;
        }
    }
    return sc;
}

int bit_blocks(const Workspace& ws, int64_t d, int vec, int M, int waves) {
    const int64_t nvec = (d + vec - 1) / vec;
    const int64_t by_work = (nvec + (int64_t)kSweepThreads * 4 - 1) / ((int64_t)kSweepThreads * 4);
    int64_t by_sm = ((int64_t)ws.sm_count * waves) / M;  // rounded down: one block too many per worker costs a whole extra wave
    int64_t nb = by_work < by_sm ? by_work : by_sm;
    return (int)(nb < 1 ? 1 : nb);
}

size_t bit_pack_smem(size_t elem, int warps, int slots) { return (size_t)warps * slots * 1024 * elem; }

}  // namespace

int configure_bit_kernels() {
    const bool ok = cudaFuncSetAttribute(aggregate_bitwise_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kAvgBitSmem + kEmitMaxWorkers * 8) == cudaSuccess &&
                    configure_dense_cluster(bit_cluster_kernel<float>) && configure_dense_cluster(bit_cluster_kernel<bf16_t>) &&
                    cudaFuncSetAttribute(bit_pack_kernel<float, true, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bit_pack_smem(4, kBitThreads / 32, kPackSlots<float, true, 3>)) == cudaSuccess;
    return ok ? MLMC_OK : MLMC_ERR_CUDA;
}

void bit_limits(KernelLimits* limits) {
    clusters_that_fit(bit_cluster_kernel<float>, kBitDenseWarps * 32, kDenseBytes, limits->dense_fit);
    limits->aggregate_bitwise = resident_blocks(aggregate_bitwise_kernel, kAvgThreads, kAvgBitSmem + 64);
}

DrawPlan bit_draw_plan(Workspace& ws, const int32_t* b, int L, uint64_t seed, uint64_t step, const mlmc_bit_msgs* out) {
    DrawPlan pl = {};
    pl.L = L;
    for (int l = 0; l < L; ++l) pl.width[l] = b[l] - (l ? b[l - 1] : 0);
    pl.seed = seed;
    pl.step = step;
    pl.bit_level = ws.bit_level;
    pl.p_all = ws.p_all;
    pl.delta_all = ws.delta_all;
    if (out) {
        pl.w_max = out->w_max;
        pl.out_scale = out->gmax;
        pl.out_level = out->level;
        pl.out_p_sel = out->p_sel;
    }
    return pl;
}

void launch_absmax(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const DrawPlan& plan, const double* p,
                   const mlmc_bit_msgs* signs, cudaStream_t s) {
    const DrawnLevels drawn = draw_levels(p, plan.L, plan.seed, plan.step, M);
    const int nb = bit_blocks(ws, d, dtype == MLMC_BF16 ? 8 : 4, M, 8);
    uint32_t* planes = signs ? signs->planes : nullptr;
    const int64_t plane_row = signs ? (1 + (int64_t)signs->w_max) * ((d + 31) / 32) : 0;
    auto go = [&](auto kernel, auto* row) {
        launch_kernel(ws, K_ABSMAX, kernel, dim3(nb, M), kSweepThreads, 0, s, row, d, ld, ws.gmax_bits, ws.acc_word, ws.done, ws.tile_max,
                      emit_tiles_per_worker(d, dtype) * kEmitGroups, planes, plane_row, plan, drawn, p ? 1 : 0, ws.status, ws.worker_err);
    };
    const int keep = !zero_batches(ws) ? 0 : signs ? 2 : 1;
    if (dtype == MLMC_BF16)
        go(keep == 2 ? absmax_kernel<bf16_t, 2> : keep ? absmax_kernel<bf16_t, 1> : absmax_kernel<bf16_t, 0>, static_cast<const bf16_t*>(g));
    else
        go(keep == 2 ? absmax_kernel<float, 2> : keep ? absmax_kernel<float, 1> : absmax_kernel<float, 0>, static_cast<const float*>(g));
}

template <typename T, typename Acc>
static void launch_bit_stats_t(Workspace& ws, const T* g, int64_t d, int M, int64_t ld, const BitSchedule& sc, int nb,
                               const DrawPlan& plan, cudaStream_t s) {
    auto kernel = sc.L <= 4 ? bit_stats_kernel<T, 4, Acc> : sc.L <= 6 ? bit_stats_kernel<T, 6, Acc> : sc.L <= 8 ? bit_stats_kernel<T, 8, Acc>
                : sc.L <= 16 ? bit_stats_kernel<T, 16, Acc> : bit_stats_kernel<T, 23, Acc>;
    launch_kernel(ws, K_BIT_STATS, kernel, dim3(nb, M), kSweepThreads, 0, s, g, d, ld, ws.gmax_bits, sc, ws.S_partial,
                  ws.stat_ctas, ws.done, plan, ws.status, ws.worker_err);
}

void launch_bit_stats(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b, int L,
                      const DrawPlan& plan, cudaStream_t s) {
    const BitSchedule sc = make_schedule(b, L);
    int nb = bit_blocks(ws, d, dtype == MLMC_BF16 ? 8 : 4, M, 4);
    if (nb > ws.stat_ctas) nb = ws.stat_ctas;
    // 32-bit sums are exact while f^2 < 2^16 and a thread adds fewer than 2^16 of them
    const int64_t trips = d / (kSweepThreads * kBitHeld);
    const int64_t per_thread = ((trips + nb - 1) / nb + 2) * kBitHeld;
    int w_top = 0;
    for (int l = 0; l < L; ++l) w_top = sc.width[l] > w_top ? sc.width[l] : w_top;
    const bool narrow = w_top <= 8 && per_thread < 65536;
    if (dtype == MLMC_BF16) {
        if (narrow) launch_bit_stats_t<bf16_t, uint32_t>(ws, static_cast<const bf16_t*>(g), d, M, ld, sc, nb, plan, s);
        else launch_bit_stats_t<bf16_t, unsigned long long>(ws, static_cast<const bf16_t*>(g), d, M, ld, sc, nb, plan, s);
    } else {
        if (narrow) launch_bit_stats_t<float, uint32_t>(ws, static_cast<const float*>(g), d, M, ld, sc, nb, plan, s);
        else launch_bit_stats_t<float, unsigned long long>(ws, static_cast<const float*>(g), d, M, ld, sc, nb, plan, s);
    }
}

// The whole message of short rows in one launch; false: the row is not for it.
bool launch_bit_cluster(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b, int L,
                        const DrawPlan& plan, const double* p, const mlmc_bit_msgs& out, cudaStream_t s) {
    const BitSchedule sc = make_schedule(b, L);
    int w_top = 0;
    for (int l = 0; l < L; ++l) w_top = std::max(w_top, sc.width[l]);
    const int cl = dense_cluster_blocks(ws, d, M);
    if (cl == 0 || (!p && (L > kDenseLevels || w_top > 8))) return false;
    const DrawnLevels drawn = draw_levels(p, L, plan.seed, plan.step, M);
    const int64_t words = (d + 31) / 32;
    const int per = (int)(((words + 31) / 32 + cl - 1) / cl);
    auto go = [&](auto kernel, auto* row, size_t elem) {
        launch_kernel_cluster(ws, K_BIT_CLUSTER, cl, kernel, dim3(M * cl), kBitDenseWarps * 32, per * 1024 * elem, s, row, d, ld, sc, plan,
                              drawn, p ? 0 : 1, per, out.planes, out.w_max, words, ws.status, ws.worker_err);
    };
    if (dtype == MLMC_BF16) go(bit_cluster_kernel<bf16_t>, static_cast<const bf16_t*>(g), 2);
    else go(bit_cluster_kernel<float>, static_cast<const float*>(g), 4);
    return true;
}

template <typename T>
static void launch_bit_pack_t(Workspace& ws, const T* g, int64_t d, int M, int64_t ld, const BitSchedule& sc,
                              const mlmc_bit_msgs& out, cudaStream_t s) {
    const int64_t words = (d + 31) / 32;
    const int64_t ngroups = (words + 31) / 32;
    const int warps = (int)std::min<int64_t>(ngroups, kBitThreads / 32);  // of short rows as many blocks as possible fit an SM
    const int64_t by_work = (ngroups + warps - 1) / warps;
    auto blocks = [&](int per_sm) {  // persistent: one wave, rounded down
        return std::max<int64_t>(1, std::min(by_work, (int64_t)ws.sm_count * per_sm / M));
    };
    auto go = [&](auto kernel, int per_sm, int slots) {
        launch_kernel(ws, K_BIT_PACK, kernel, dim3((unsigned)blocks(per_sm), M), warps * 32, bit_pack_smem(sizeof(T), warps, slots), s, g, d, ld,
                      ws.gmax_bits, sc, ws.bit_level, zero_batches(ws), emit_tiles_per_worker(d, sizeof(T) == 2 ? MLMC_BF16 : MLMC_F32) * kEmitGroups,
                      out.planes, out.w_max, words);
    };
    if (!zero_batches(ws)) {
        go(bit_pack_kernel<T, false, 3>, 3, kPackSlots<T, false, 3>);
        return;
    }
    // The groups that are left to read lie where the layers are large: some warps have far more of them than others.  Where a warp has
    // few groups the call lasts as long as the longest such chain, and three blocks per SM with registers to spare and two copies in
    // flight are the faster way; with many, four blocks (64 registers: the bf16 kernel spills some, and is the faster one all the same).
    // us per step, adaptive p, three / four: fp32 8 x 3.3M 92 / 100, 8 x 6.6M 154 / 154, 8 x 12.5M 266 / 267, 8 x 20M 392 / 390,
    // 8 x 62M 1041 / 1023; bf16 8 x 7M 131 / 136, 8 x 11M 198 / 199, 8 x 15M 254 / 254, 8 x 18M 303 / 297, 32 x 25.6M 1491 / 1445.
    // Earlier where whole blocks per worker leave more than 5 % of three blocks per SM idle (given p): fp32 32 x 2M 126 / 123,
    // bf16 32 x 2.1M 103 / 102, 32 x 1.7M 74.5 / 75.9.
    constexpr int64_t kManyGroups = 24, kManyGroupsIdle = 12;
    const int64_t per_warp = (ngroups + blocks(4) * warps - 1) / (blocks(4) * warps);
    const bool idle = ws.sm_count * 3 / M * M * 20 < ws.sm_count * 3 * 19;
    if (per_warp > (idle ? kManyGroupsIdle : kManyGroups)) go(bit_pack_kernel<T, true, 4>, 4, kPackSlots<T, true, 4>);
    else go(bit_pack_kernel<T, true, 3>, 3, kPackSlots<T, true, 3>);
}

void launch_bit_pack(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b, int L,
                     const mlmc_bit_msgs& out, cudaStream_t s) {
    const BitSchedule sc = make_schedule(b, L);
    if (dtype == MLMC_BF16)
        launch_bit_pack_t<bf16_t>(ws, static_cast<const bf16_t*>(g), d, M, ld, sc, out, s);
    else
        launch_bit_pack_t<float>(ws, static_cast<const float*>(g), d, M, ld, sc, out, s);
}

void launch_aggregate_bitwise(Workspace& ws, const mlmc_bit_msgs& msgs, const int32_t* b, int L, int M, int64_t d,
                              float* out, cudaStream_t s) {
    const BitSchedule sc = make_schedule(b, L);
    const int64_t words = (d + 31) / 32;
    const size_t smem = kAvgBitSmem + (size_t)M * 8;
    // whole waves only: every block does the same number of iterations, so a partial last wave costs a full one
    const int64_t nb = std::min((words + kAvgThreads - 1) / kAvgThreads, (int64_t)ws.sm_count * ws.limits.aggregate_bitwise * 2);
    launch_kernel(ws, K_AGG_BIT, aggregate_bitwise_kernel, dim3((unsigned)nb), kAvgThreads, smem, s, msgs.planes, msgs.gmax,
                  msgs.level, msgs.p_sel, sc, msgs.w_max, words, M, d, out);
}

}  // namespace mlmc
