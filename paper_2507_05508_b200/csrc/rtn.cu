// MLMC with round-to-nearest levels (Sec. 3.2 end, App. G).
//
//   C^l(v) = clip(delta^l round(v / delta^l), -c, c),  delta^l = 2c / (2^{r_l} - 1),  c = max_i |v_i|;
// the top level is the identity (Def. 3.1) and C^{-1} = 0.  The residual C^l - C^{l-1} is dense and has no band or
// bit-plane structure, so the adaptive probabilities (Lemma 3.4, Alg. 3) need ||C^l - C^{l-1}|| of every level from
// one sweep: every thread keeps one fp64 accumulator per level in registers.  Then the draw, and a sweep that writes the
// dense message.
//
// The rounding decides an integer, so its arithmetic is fixed (the same on the host checker): with
// inv = fl32((2^r - 1) / (2c)) and delta = fl32(2c / (2^r - 1)), t = fl32(v inv), k = t rounded to nearest, ties to
// even, C = clip(fl32(k delta), -c, c).  Residuals, norms and the scaling by 1/p are fp64.
#include <algorithm>
#include <type_traits>

#include "dense_cluster.cuh"

namespace mlmc {

namespace {

constexpr int kRtnThreads = 256;
constexpr int kRtnMaxLevels = 17;  // widths 1..16 strictly increasing, plus the identity

struct RtnSchedule {
    int L;                  // levels, the last one is the identity
    int r[kRtnMaxLevels];   // widths of levels 0..L-2
};

struct RtnGrid {
    float inv, delta;
};

__device__ __forceinline__ RtnGrid rtn_grid(float c, int r) {
    const double steps = (double)((1u << r) - 1u);
    RtnGrid gq;
    gq.inv = (float)(steps / (2.0 * (double)c));
    gq.delta = (float)(2.0 * (double)c / steps);
    return gq;
}

__device__ __forceinline__ float rtn_value(float v, float c, RtnGrid gq) {
    const float t = __fmul_rn(v, gq.inv);
    // to nearest, ties to even: |t| <= 2^15 (r <= 16), so adding and subtracting 1.5 * 2^23 rounds t to an integer in
    // the adder, with the default rounding mode, without the conversion unit
    const float k = __fadd_rn(__fadd_rn(t, 12582912.0f), -12582912.0f);
    return fminf(fmaxf(__fmul_rn(k, gq.delta), -c), c);
}

// What the statistics need to know of a level: its grid, the largest magnitude that rounds to 0 and the largest one that
// the clipping cannot touch (both as bits of a magnitude, so that they compare as integers).
struct RtnLevel {
    float inv, delta;
    int zero_upto, free_upto;  // -1: none
};

__device__ RtnLevel rtn_level(float c, int r) {
    const RtnGrid gq = rtn_grid(c, r);
    RtnLevel v;
    v.inv = gq.inv;
    v.delta = gq.delta;
    // t = fl32(m inv) does not fall as m grows, and t <= 1/2 rounds to 0 (ties to even)
    v.zero_upto = v.free_upto = -1;
    // c below the normal range: 1 / delta overflows, and 0 inv is not a number; one bit, c at the end of the range: delta overflows
    if (!(gq.inv <= 3.0e38f && gq.delta <= 3.0e38f)) return v;
    uint32_t z = min(__float_as_uint(0.5f / gq.inv), 0x7F7FFFFFu);
    while (z > 0u && __fmul_rn(__uint_as_float(z), gq.inv) > 0.5f) --z;
    while (z < 0x7F7FFFFFu && __fmul_rn(__uint_as_float(z + 1u), gq.inv) <= 0.5f) ++z;
    v.zero_upto = (int)z;
    const float f = c - gq.delta;  // |k delta| <= |v| + delta / 2 (1 + 2^-20)
    if (f > 0.0f) v.free_upto = __float_as_int(f);
    return v;
}

// C^l(-v) = -C^l(v) for every entry of the row and every level?  The first level has the largest delta, the last one the largest 1 / delta.
__device__ __forceinline__ bool odd_levels(const RtnLevel* levels, int L) {
    return L < 2 || (levels[0].zero_upto >= 0 && levels[L - 2].zero_upto >= 0);
}

// Residual energies of every level: partial[m][block][l] = sum over the block's entries of (C^l - C^{l-1})^2.
// A warp takes the entries level by level, kRtnHeld per lane.  The levels whose grid is so coarse that the largest of the
// warp's entries rounds to 0 contribute nothing and are skipped: the clipping value is the row's largest magnitude, and
// in a gradient with per-layer scales most entries are small beside it.  The first level that is left has C^{l-1} = 0, so
// its residual is its value.  The differences and sums are fp64 (a difference of two fp32 values is exact); what bounds the
// kernel where nothing is skipped is issue: a value per entry and level is found, widened to fp64, subtracted, squared and added.
// 8 x 124M fp32 entries, L = 5: 2.29 ms with every entry taken through every level; 1.02 with one trip in flight and one and
// a half waves of blocks, 0.85 with every value through the conversion unit, 0.79 with single instructions for the grid values, now 0.74
// (0.57 is the first sweep of the same row).
constexpr int kRtnHeld = 8;

template <typename T>
__device__ __forceinline__ void rtn_expand(const uint4* q, float (&v)[kRtnHeld]) {
#pragma unroll
    for (int j = 0; j < kRtnHeld / ElemTraits<T>::kVec; ++j) {
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

// The conversion unit takes 16 numbers per clock and SM, a quarter of what the fp64 unit adds up.  So every second number (x >= 0; one
// of four or three of four are within 1 %) goes another way: its bits moved to the places of a double are x 2^-896, zero and the numbers
// below the normal range included, and the product with 2^896 is exact.
__device__ __forceinline__ double widen(float x, bool by_product) {
    if (!by_product) return (double)x;
    const uint32_t b = __float_as_uint(x);
    return __hiloint2double((int)(b >> 3), (int)(b << 29)) * 0x1p896;
}

// One trip of a warp: kRtnHeld entries per lane.  Magnitudes: C^l(-v) = -C^l(v), except in rows with a level whose 1 / delta or delta
// overflows: the product 0 Inf is not a number and comes out of the clipping as -c (with delta = 0 that of every entry).  Those rows
// go entry by entry.  The grid values of two entries are found together, by packed instructions.  one = 1, an argument: the compiler
// merges a packed product and the addition after it into one rounding, also where both say that they round, and the rounding of
// t = fl32(v inv) decides ties.  So the addition is a multiply-add of t with one.
template <int LMAX>
__device__ __forceinline__ void take_levels(const float (&signed_v)[kRtnHeld], float c, const RtnLevel* levels, int L, float one, double (&acc)[LMAX]) {
    float v[kRtnHeld];
    int mx = 0;
#pragma unroll
    for (int e = 0; e < kRtnHeld; ++e) {
        v[e] = fabsf(signed_v[e]);
        mx = max(mx, __float_as_int(v[e]));
    }
    mx = __reduce_max_sync(0xFFFFFFFFu, mx);
    double prev[kRtnHeld];  // C^{l-1}
    bool first = true;      // C^{l-1} = 0 for every entry of the warp (warp-uniform)
#pragma unroll
    for (int l = 0; l < LMAX; ++l) {
        if (l > L - 1) break;
        if (l == L - 1) {  // the identity
            if (first) {
#pragma unroll
                for (int e = 0; e < kRtnHeld; ++e) prev[e] = 0.0;
            }
            double odd = 0.0;  // two chains of additions
#pragma unroll
            for (int e = 0; e < kRtnHeld; ++e) {
                const double res = widen(v[e], e & 1) - prev[e];
                if (e & 1) odd = fma(res, res, odd);
                else acc[l] = fma(res, res, acc[l]);
            }
            acc[l] += odd;
            break;
        }
        const RtnLevel lv = levels[l];
        if (mx <= lv.zero_upto) continue;  // the grids get finer: once a level is not skipped, none after it is
        float x[kRtnHeld];
        const uint64_t inv2 = pair(lv.inv, lv.inv), delta2 = pair(lv.delta, lv.delta), up2 = pair(12582912.0f, 12582912.0f),
                       down2 = pair(-12582912.0f, -12582912.0f), one2 = pair(one, one);
#pragma unroll
        for (int e = 0; e < kRtnHeld; e += 2) {
            const uint64_t k = add_pair(fma_pair(mul_pair(pair(v[e], v[e + 1]), inv2), one2, up2), down2);
            const uint64_t y = mul_pair(k, delta2);
            x[e] = __uint_as_float((uint32_t)y);
            x[e + 1] = __uint_as_float((uint32_t)(y >> 32));
        }
        if (mx > lv.free_upto) {
#pragma unroll
            for (int e = 0; e < kRtnHeld; ++e) x[e] = fminf(x[e], c);
        }
        double odd = 0.0;
        if (first) {
#pragma unroll
            for (int e = 0; e < kRtnHeld; ++e) {
                prev[e] = widen(x[e], e & 1);
                if (e & 1) odd = fma(prev[e], prev[e], odd);
                else acc[l] = fma(prev[e], prev[e], acc[l]);
            }
            first = false;
        } else {
#pragma unroll
            for (int e = 0; e < kRtnHeld; ++e) {
                const double cur = widen(x[e], e & 1), res = cur - prev[e];
                if (e & 1) odd = fma(res, res, odd);
                else acc[l] = fma(res, res, acc[l]);
                prev[e] = cur;
            }
        }
        acc[l] += odd;
    }
}

template <int LMAX>
__device__ __forceinline__ void take_entry(float v, float c, const RtnLevel* levels, int L, double (&acc)[LMAX]) {
    double prev = 0.0;
#pragma unroll
    for (int l = 0; l < LMAX; ++l) {
        if (l > L - 1) break;
        const double cur = (l < L - 1) ? (double)rtn_value(v, c, {levels[l].inv, levels[l].delta}) : (double)v;
        acc[l] = fma(cur - prev, cur - prev, acc[l]);
        prev = cur;
    }
}

template <typename T, int LMAX>
__global__ void __launch_bounds__(kRtnThreads, LMAX <= 6 ? 4 : 3)
rtn_stats_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const uint32_t* gmax_bits, const __grid_constant__ RtnSchedule sc, double* partial,
                 int rtn_ctas, uint32_t* done, const __grid_constant__ DrawPlan pl, int* status, int* worker_err, float one) {
    using Tr = ElemTraits<T>;
    extern __shared__ __align__(16) uint4 sh_vectors[];  // [4][vectors per trip][kRtnThreads]
    __shared__ double sh_red[LMAX][kRtnThreads / 32];
    __shared__ double sh_delta[kMaxLevels];
    __shared__ RtnLevel sh_lv[kRtnMaxLevels];
    pdl_enter();
    const int m = blockIdx.y;
    if (worker_err[m]) return;
    const float c = __uint_as_float(gmax_bits[m]);
    if (threadIdx.x < sc.L - 1) sh_lv[threadIdx.x] = rtn_level(c > 0.0f ? c : 1.0f, sc.r[threadIdx.x]);
    __syncthreads();
    double acc[LMAX];
#pragma unroll
    for (int l = 0; l < LMAX; ++l) acc[l] = 0.0;
    if (c > 0.0f) {
        const T* row = g + (int64_t)m * ld;
        constexpr int kVecs = kRtnHeld / Tr::kVec;  // 16-byte vectors per lane and trip
        constexpr int kTrip = kRtnThreads * kVecs;
        const int64_t full_end = d / Tr::kVec;
        const bool odd = odd_levels(sh_lv, sc.L);
        const int64_t trips = odd ? full_end / kTrip : 0;
        stream_trips<kVecs, kRtnThreads>(reinterpret_cast<const uint4*>(row), blockIdx.x, gridDim.x, trips, sh_vectors, [&](const uint4 (&q)[kVecs]) {
            float v[kRtnHeld];
            rtn_expand<T>(q, v);
            take_levels<LMAX>(v, c, sh_lv, sc.L, one, acc);
        });
        // the rest of the row, one by one: fewer than kTrip + 1 vectors for the last block, or everything for all blocks
        if (!odd || blockIdx.x == gridDim.x - 1) {
            const int64_t step = odd ? kRtnThreads : (int64_t)gridDim.x * kRtnThreads;
            for (int64_t i = trips * kTrip * Tr::kVec + (odd ? 0 : (int64_t)blockIdx.x * kRtnThreads) + threadIdx.x; i < d; i += step) {
                float v;
                if constexpr (Tr::kVec == 4) v = reinterpret_cast<const float*>(row)[i];
                else v = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(row)[i] << 16);
                take_entry<LMAX>(v, c, sh_lv, sc.L, acc);
            }
        }
    }
    // fixed-order reduction: shuffle tree per warp, then the warp sums in warp order
#pragma unroll
    for (int l = 0; l < LMAX; ++l) {
        if (l >= sc.L) break;
        double x = acc[l];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
        if ((threadIdx.x & 31) == 0) sh_red[l][threadIdx.x >> 5] = x;
    }
    __syncthreads();
    if (threadIdx.x < sc.L) {
        double s = 0.0;
#pragma unroll
        for (int w = 0; w < kRtnThreads / 32; ++w) s += sh_red[threadIdx.x][w];
        partial[((int64_t)m * rtn_ctas + blockIdx.x) * kMaxLevels + threadIdx.x] = s;
    }
    if (!last_block(&done[m], gridDim.x)) return;
    // the per-block partials, a warp per level in a fixed order; then p, the draw and the header
    const int lane = threadIdx.x & 31;
    for (int l = threadIdx.x >> 5; l < sc.L; l += kRtnThreads / 32) {
        double e = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) e += __ldcg(&partial[((int64_t)m * rtn_ctas + b) * kMaxLevels + l]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xFFFFFFFFu, e, o);
        if (lane == 0) sh_delta[l] = sqrt(e);
    }
    __syncthreads();
    finish_levels(pl, m, sh_delta, c, status, worker_err);
}

// val_i of the drawn level's message.
template <typename T>
struct Residual {
    double inv_p;
    float c;
    bool top, first, flat;  // flat: a small entry leaves nothing (not so where delta overflows and 0 delta is not a number)
    RtnGrid hi, lo;
    __device__ __forceinline__ Residual(float c_, const RtnSchedule& sc, int level, double p)
        : inv_p(p > 0.0 ? 1.0 / p : 0.0), c(c_), top(level == sc.L - 1), first(level == 0) {
        hi = rtn_grid(c > 0.0f ? c : 1.0f, top ? 1 : sc.r[level]);
        lo = rtn_grid(c > 0.0f ? c : 1.0f, first ? 1 : sc.r[level - 1]);
        flat = !top && (first ? hi : lo).delta <= 3.0e38f;
    }
    __device__ __forceinline__ float operator()(uint32_t bits) const {
        const float v = ElemTraits<T>::value(bits);
        if (!(c > 0.0f)) return 0.0f;
        const double h = top ? (double)v : (double)rtn_value(v, c, hi);
        const double l = first ? 0.0 : (double)rtn_value(v, c, lo);
        return (float)((h - l) * inv_p);
    }
    // Nothing up to this magnitude leaves anything: fl32(m inv) does not fall as m grows, 1/2 rounds to 0 (ties to even), and the
    // level before has the coarser grid.
    __device__ __forceinline__ bool rounds_to_zero(uint32_t magnitude) const {
        return !(c > 0.0f) || (flat && __fmul_rn(__uint_as_float(magnitude), hi.inv) <= 0.5f);
    }
    __device__ __forceinline__ void vector(const uint4& q, float* __restrict__ out) const {  // a vector's entries, out 16-byte aligned
        if constexpr (sizeof(T) == 4) {
            reinterpret_cast<float4*>(out)[0] = make_float4((*this)(q.x), (*this)(q.y), (*this)(q.z), (*this)(q.w));
        } else {
            reinterpret_cast<float4*>(out)[0] =
                make_float4((*this)(q.x & 0xFFFFu), (*this)(q.x >> 16), (*this)(q.y & 0xFFFFu), (*this)(q.y >> 16));
            reinterpret_cast<float4*>(out)[1] =
                make_float4((*this)(q.z & 0xFFFFu), (*this)(q.z >> 16), (*this)(q.w & 0xFFFFu), (*this)(q.w >> 16));
        }
    }
};

// The dense message of the drawn level: val_i = (C^l - C^{l-1})_i / p_l, rounded to fp32 once.  A warp takes a batch (four 16-byte
// vectors per lane) at a time.  The batches whose largest key (recorded by the first sweep) rounds to 0 at the drawn level do so
// at the coarser level before it too: they are written, and not read.  With clipping at the row's largest magnitude that is
// most of a row wherever its layers differ in scale (8 x 124M fp32 entries: 1290 -> 748 us).  Calls that L2 holds read everything,
// and so do fp32 rows of which no batch rounds to 0 (the smallest of the largest keys says so): there the looks only cost.  8 x 3.3M
// entries of one scale 43.6 us with the looks, 37.8 without; 8 x 31M 327, 320; 8 x 124M 1300, 1293.  bf16 rows look always, at
// the next 32 batches while 32 are written: both ways in one kernel cost them more registers than the looks cost time (8 x 62M of one
// scale: everything read 687, both ways 700, looks 702; 8 x 25M 277, 279, 277; 8 x 6.6M 74.4, 72.4, 74.7).  fp32 with the looks ahead:
// 8 x 124M in layers 838, 8 x 31M of one scale 324.
template <typename T, bool SKIP>
__global__ void __launch_bounds__(kRtnThreads)
rtn_emit_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const uint32_t* gmax_bits, RtnSchedule sc,
                const int32_t* bit_level, const double* p_all, const uint32_t* batch_max, int batches_per_worker, float* __restrict__ val,
                int64_t ldv) {
    using Tr = ElemTraits<T>;
    pdl_enter();
    const int m = blockIdx.y;
    const int level = bit_level[m];
    if (level < 0) return;
    const float c = __uint_as_float(gmax_bits[m]);
    const Residual<T> residual(c, sc, level, p_all[m * kMaxLevels + level]);
    const T* row = g + (int64_t)m * ld;
    float* out = val + (int64_t)m * ldv;
    const int64_t nvec = (d + Tr::kVec - 1) / Tr::kVec, full_end = (ldv % 4 == 0) ? d / Tr::kVec : 0;
    if (!SKIP || (sizeof(T) == 4 && !residual.rounds_to_zero(gmax_bits[gridDim.y + m]))) {  // no batch is skipped
        // Chunks of kBatch vectors per thread, all in flight before the first is used.
        constexpr int kBatch = 4;
        for (int64_t base = (int64_t)blockIdx.x * kBatch * kRtnThreads; base < nvec; base += (int64_t)gridDim.x * kBatch * kRtnThreads) {
            const int64_t v = base + threadIdx.x;
            if (base + kBatch * kRtnThreads <= full_end) {
                uint4 q[kBatch];
#pragma unroll
                for (int j = 0; j < kBatch; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + v + j * kRtnThreads);
#pragma unroll
                for (int j = 0; j < kBatch; ++j) residual.vector(q[j], out + (v + j * kRtnThreads) * Tr::kVec);
            } else {
                for (int64_t u = v; u < min(nvec, base + kBatch * kRtnThreads); u += kRtnThreads) {
                    if (u < full_end) residual.vector(__ldg(reinterpret_cast<const uint4*>(row) + u), out + u * Tr::kVec);
                    else for_each_in_vector<T>(row, u, d, [&](int64_t i, uint32_t bits) { out[i] = residual(bits); });
                }
            }
        }
    } else {
        const int lane = threadIdx.x & 31;
        const uint32_t* bmax = batch_max + (int64_t)m * batches_per_worker;
        const int64_t nbatch = (nvec + kEmitGroupVecs - 1) / kEmitGroupVecs, stride = (int64_t)gridDim.x * (kRtnThreads / 32);
        // a lane looks at the largest key of one of the warp's next 32 batches (bf16: while the 32 before are written)
        int64_t own = (int64_t)blockIdx.x * (kRtnThreads / 32) + (threadIdx.x >> 5) + lane * stride;
        uint32_t ahead = sizeof(T) == 2 && own < nbatch ? bmax[own] : 0u;
        for (; own - lane * stride < nbatch; own += 32 * stride) {
            const int64_t base = own - lane * stride;
            const bool inside = own < nbatch && (own + 1) * kEmitGroupVecs <= full_end;
            const bool zero = inside && residual.rounds_to_zero(sizeof(T) == 2 ? ahead : bmax[own]);
            if (sizeof(T) == 2) ahead = own + 32 * stride < nbatch ? bmax[own + 32 * stride] : 0u;
            uint32_t todo = __ballot_sync(0xFFFFFFFFu, own < nbatch);
            const uint32_t zeros = __ballot_sync(0xFFFFFFFFu, zero);
            for (; todo; todo &= todo - 1u) {
                const int i = __ffs(todo) - 1;
                const int64_t b = base + i * stride, v = b * kEmitGroupVecs + lane;
                if ((zeros >> i) & 1u) {
                    float4* to = reinterpret_cast<float4*>(out + (v - lane) * Tr::kVec) + lane;
#pragma unroll
                    for (int j = 0; j < Tr::kVec; ++j) to[j * 32] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                } else if ((b + 1) * kEmitGroupVecs <= full_end) {
                    uint4 q[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) q[j] = __ldg(reinterpret_cast<const uint4*>(row) + v + j * 32);
#pragma unroll
                    for (int j = 0; j < 4; ++j) residual.vector(q[j], out + (v + j * 32) * Tr::kVec);
                } else {
                    for (int64_t u = v; u < min(nvec, (b + 1) * kEmitGroupVecs); u += 32) {
                        if (u < full_end) residual.vector(__ldg(reinterpret_cast<const uint4*>(row) + u), out + u * Tr::kVec);
                        else for_each_in_vector<T>(row, u, d, [&](int64_t e, uint32_t bits) { out[e] = residual(bits); });
                    }
                }
            }
        }
    }
}

// Short rows: all of the above in one launch (dense_cluster.cuh); with adaptive probabilities at most kRtnDenseLevels levels.
// 4 x 50,000 bf16 entries, adaptive: 19 us for the three kernels above, 14 for this one.
constexpr int kRtnDenseLevels = 6;
constexpr int kRtnDenseWarps = 16;  // the fp64 statistics need the registers

template <typename T>
__global__ void __launch_bounds__(kRtnDenseWarps * 32, 1)
rtn_cluster_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const __grid_constant__ RtnSchedule sc,
                   const __grid_constant__ DrawPlan pl, const __grid_constant__ DrawnLevels drawn, int adaptive, int per_block,
                   float* __restrict__ val, int64_t ldv, int* status, int* worker_err, float one) {
    using Tr = ElemTraits<T>;
    extern __shared__ __align__(16) uint32_t sh_slots[];
    __shared__ DenseShared<kRtnDenseWarps, double> sh;
    __shared__ RtnLevel sh_lv[kRtnDenseLevels];
    cg::cluster_group cluster = cg::this_cluster();
    pdl_enter();
    const int rank = (int)cluster.block_rank(), m = blockIdx.x / (int)cluster.num_blocks();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t g0 = (int64_t)rank * per_block;
    const int n = (int)max((int64_t)0, min((int64_t)per_block, (d + 1023) / 1024 - g0));
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
    const float c = __uint_as_float(Tr::kVec == 8 ? top << 16 : top);
    auto entry = [&](int i, int e) -> uint32_t {  // entry e of group i
        const uint32_t w = sh_slots[i * kGroupSlot<T> + group_place<T>(e / 32, (e % 32) / Tr::kVec) + (e % Tr::kVec) * (int)sizeof(T) / 4];
        return sizeof(T) == 4 ? w : (e & 1) ? w >> 16 : w & 0xFFFFu;
    };
    double delta = 0.0;
    if (adaptive) {
        if (threadIdx.x < sc.L - 1) sh_lv[threadIdx.x] = rtn_level(c > 0.0f ? c : 1.0f, sc.r[threadIdx.x]);
        __syncthreads();
        double acc[kRtnDenseLevels];
#pragma unroll
        for (int l = 0; l < kRtnDenseLevels; ++l) acc[l] = 0.0;
        if (c > 0.0f) {
            constexpr int kVecs = kRtnHeld / Tr::kVec;  // a warp takes a quarter of a group
            const bool odd = odd_levels(sh_lv, sc.L);
#pragma unroll 1
            for (int u = warp; u < 4 * n; u += kRtnDenseWarps) {
                const int64_t e0 = (g0 + (u >> 2)) * 1024;
                if (odd && e0 + 1024 <= d) {
                    const uint4* x = reinterpret_cast<const uint4*>(sh_slots + (u >> 2) * kGroupSlot<T>) + (u & 3) * kVecs * 32 + lane;
                    uint4 q[kVecs];
#pragma unroll
                    for (int j = 0; j < kVecs; ++j) q[j] = x[j * 32];
                    float v[kRtnHeld];
                    rtn_expand<T>(q, v);
                    take_levels<kRtnDenseLevels>(v, c, sh_lv, sc.L, one, acc);
                } else {  // one by one; entries past the row's end are not entries
                    for (int e = (u & 3) * 256 + lane; e < (u & 3) * 256 + 256 && e0 + e < d; e += 32)
                        take_entry<kRtnDenseLevels>(Tr::value(entry(u >> 2, e)), c, sh_lv, sc.L, acc);
                }
            }
        }
        double all[kDenseLevels];
#pragma unroll
        for (int l = 0; l < kDenseLevels; ++l) all[l] = l < kRtnDenseLevels ? acc[min(l, kRtnDenseLevels - 1)] : 0.0;
        delta = sqrt(dense_sums(cluster, all, sh));
        if (threadIdx.x >= sc.L) delta = 0.0;
    }
    double p;
    const int level = dense_level(pl, drawn, adaptive, m, first, delta, c, sh, &p, status, worker_err);
    const Residual<T> residual(c, sc, level, p);
    float* out = val + (int64_t)m * ldv;
    const bool vec_ok = (ldv % 4 == 0);
    for (int u = warp; u < 4 * n; u += kRtnDenseWarps) {  // a quarter of a group
        const int i = u >> 2;
        const int64_t e0 = (g0 + i) * 1024;
        if (e0 + 1024 <= d && vec_ok) {
            constexpr int kQuarter = kGroupChunks<T> * 8;
#pragma unroll
            for (int k = (u & 3) * kQuarter + lane, j = 0; j < kQuarter / 32; ++j, k += 32)
                residual.vector(*reinterpret_cast<const uint4*>(sh_slots + i * kGroupSlot<T> + group_place<T>(k / kGroupChunks<T>, k % kGroupChunks<T>)),
                                out + e0 + k * Tr::kVec);
        } else {
            for (int e = (u & 3) * 256 + lane; e < (u & 3) * 256 + 256 && e0 + e < d; e += 32) out[e0 + e] = residual(entry(i, e));
        }
    }
}

// Server average of dense messages: out[i] = (1/M) sum_m val[m][i] in worker order, four workers' entries in flight.  (With one
// and its level before it, 200 workers of 3000 entries took 34 us, 64 of 200,000 12.8.)
constexpr int kAvgTogether = 4;

__global__ void __launch_bounds__(kRtnThreads)
aggregate_dense_kernel(const float* __restrict__ val, const int32_t* level, int M, int64_t d, int64_t ldv,
                       float* __restrict__ out) {
    pdl_enter();
    const float inv_M = 1.0f / (float)M;
    const bool aligned = ldv % 4 == 0 && ((reinterpret_cast<uintptr_t>(val) | reinterpret_cast<uintptr_t>(out)) & 15) == 0;
    const int64_t n4 = aligned ? d / 4 : 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n4; v += (int64_t)gridDim.x * blockDim.x) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int m0 = 0; m0 < M; m0 += kAvgTogether) {
            float4 x[kAvgTogether];
            bool on[kAvgTogether];
#pragma unroll
            for (int j = 0; j < kAvgTogether; ++j) on[j] = m0 + j < M && level[m0 + j] >= 0;
#pragma unroll
            for (int j = 0; j < kAvgTogether; ++j)
                if (on[j]) x[j] = __ldg(reinterpret_cast<const float4*>(val + (int64_t)(m0 + j) * ldv) + v);
#pragma unroll
            for (int j = 0; j < kAvgTogether; ++j)
                if (on[j]) {
                    a.x += x[j].x; a.y += x[j].y; a.z += x[j].z; a.w += x[j].w;
                }
        }
        a.x *= inv_M; a.y *= inv_M; a.z *= inv_M; a.w *= inv_M;
        reinterpret_cast<float4*>(out)[v] = a;
    }
    for (int64_t i = n4 * 4 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
        float a = 0.f;
        for (int m = 0; m < M; ++m)
            if (level[m] >= 0) a += val[(int64_t)m * ldv + i];
        out[i] = a * inv_M;
    }
}

RtnSchedule make_rtn_schedule(const int32_t* r, int L) {
    RtnSchedule sc = {};
    sc.L = L;
    for (int l = 0; l + 1 < L; ++l) sc.r[l] = r[l];
    return sc;
}

int rtn_blocks(const Workspace& ws, int64_t d, int vec, int M, int per_sm) {
    const int64_t nvec = (d + vec - 1) / vec;
    const int64_t by_work = (nvec + (int64_t)kRtnThreads * 4 - 1) / ((int64_t)kRtnThreads * 4);
    int64_t by_sm = ((int64_t)ws.sm_count * per_sm) / M;
    int64_t nb = by_work < by_sm ? by_work : by_sm;
    return (int)(nb < 1 ? 1 : nb);
}

}  // namespace

DrawPlan rtn_draw_plan(Workspace& ws, int L, uint64_t seed, uint64_t step, const mlmc_rtn_msgs* out) {
    DrawPlan pl = {};
    pl.L = L;
    pl.seed = seed;
    pl.step = step;
    pl.bit_level = ws.bit_level;
    pl.p_all = ws.p_all;
    pl.delta_all = ws.delta_all;
    if (out) {
        pl.out_scale = out->c;
        pl.out_level = out->level;
        pl.out_p_sel = out->p_sel;
    }
    return pl;
}

namespace {
size_t rtn_stats_smem(size_t elem) { return (size_t)4 * kRtnThreads * kRtnHeld * elem; }

template <typename T, int LMAX>
void launch_rtn_stats_t(Workspace& ws, const T* g, int64_t d, int M, int64_t ld, const RtnSchedule& sc, const DrawPlan& plan,
                        cudaStream_t s) {
    const size_t smem = rtn_stats_smem(sizeof(T));
    const int resident = ws.limits.rtn_stats[sizeof(T) == 2][LMAX == kRtnMaxLevels];
    // whole waves (a partial last one costs a full one), four of them: how much a block skips differs (one: 910 us, two: 897,
    // four: 866 for 8 x 124M entries)
    const int nb = std::min(rtn_blocks(ws, d, ElemTraits<T>::kVec, M, 4 * resident), ws.rtn_ctas);
    launch_kernel(ws, K_RTN_STATS, rtn_stats_kernel<T, LMAX>, dim3(nb, M), kRtnThreads, smem, s, g, d, ld, ws.gmax_bits, sc,
                  ws.rtn_partial, ws.rtn_ctas, ws.done, plan, ws.status, ws.worker_err, 1.0f);
}
}  // namespace

void launch_rtn_stats(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                      const DrawPlan& plan, cudaStream_t s) {
    const RtnSchedule sc = make_rtn_schedule(r, L);
    auto go = [&](auto* row) {
        if (L <= 6) launch_rtn_stats_t<std::remove_const_t<std::remove_pointer_t<decltype(row)>>, 6>(ws, row, d, M, ld, sc, plan, s);
        else launch_rtn_stats_t<std::remove_const_t<std::remove_pointer_t<decltype(row)>>, kRtnMaxLevels>(ws, row, d, M, ld, sc, plan, s);
    };
    if (dtype == MLMC_BF16) go(static_cast<const bf16_t*>(g));
    else go(static_cast<const float*>(g));
}

// The whole message of short rows in one launch; false: the row is not for it.
bool launch_rtn_cluster(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                        const DrawPlan& plan, const double* p, const mlmc_rtn_msgs& out, cudaStream_t s) {
    const int cl = dense_cluster_blocks(ws, d, M);
    if (cl == 0 || (!p && L > kRtnDenseLevels)) return false;
    const RtnSchedule sc = make_rtn_schedule(r, L);
    const DrawnLevels drawn = draw_levels(p, L, plan.seed, plan.step, M);
    const int per = (int)(((d + 1023) / 1024 + cl - 1) / cl);
    auto go = [&](auto kernel, auto* row, size_t elem) {
        launch_kernel_cluster(ws, K_RTN_CLUSTER, cl, kernel, dim3(M * cl), kRtnDenseWarps * 32, per * 1024 * elem, s, row, d, ld, sc, plan,
                              drawn, p ? 0 : 1, per, out.val, out.ldv, ws.status, ws.worker_err, 1.0f);
    };
    if (dtype == MLMC_BF16) go(rtn_cluster_kernel<bf16_t>, static_cast<const bf16_t*>(g), 2);
    else go(rtn_cluster_kernel<float>, static_cast<const float*>(g), 4);
    return true;
}

int configure_rtn_kernels() {
    return configure_dense_cluster(rtn_cluster_kernel<float>) && configure_dense_cluster(rtn_cluster_kernel<bf16_t>) ? MLMC_OK : MLMC_ERR_CUDA;
}

void rtn_limits(KernelLimits* limits) {
    limits->rtn_stats[0][0] = resident_blocks(rtn_stats_kernel<float, 6>, kRtnThreads, rtn_stats_smem(4));
    limits->rtn_stats[0][1] = resident_blocks(rtn_stats_kernel<float, kRtnMaxLevels>, kRtnThreads, rtn_stats_smem(4));
    limits->rtn_stats[1][0] = resident_blocks(rtn_stats_kernel<bf16_t, 6>, kRtnThreads, rtn_stats_smem(2));
    limits->rtn_stats[1][1] = resident_blocks(rtn_stats_kernel<bf16_t, kRtnMaxLevels>, kRtnThreads, rtn_stats_smem(2));
}

void launch_rtn_emit(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                     const mlmc_rtn_msgs& out, cudaStream_t s) {
    const RtnSchedule sc = make_rtn_schedule(r, L);
    const int nb = rtn_blocks(ws, d, dtype == MLMC_BF16 ? 8 : 4, M, 16);
    auto go = [&](auto kernel, auto* row) {
        launch_kernel(ws, K_RTN_EMIT, kernel, dim3(nb, M), kRtnThreads, 0, s, row, d, ld, ws.gmax_bits, sc, ws.bit_level,
                      ws.p_all, zero_batches(ws), emit_tiles_per_worker(d, dtype) * kEmitGroups, out.val, out.ldv);
    };
    const bool skip = zero_batches(ws) != nullptr;
    if (dtype == MLMC_BF16) go(skip ? rtn_emit_kernel<bf16_t, true> : rtn_emit_kernel<bf16_t, false>, static_cast<const bf16_t*>(g));
    else go(skip ? rtn_emit_kernel<float, true> : rtn_emit_kernel<float, false>, static_cast<const float*>(g));
}

void launch_aggregate_dense(Workspace& ws, const float* val, const int32_t* level, int M, int64_t d, int64_t ldv,
                            float* out, cudaStream_t s) {
    int64_t nb = (d / 4 + kRtnThreads - 1) / kRtnThreads;
    const int64_t cap = (int64_t)ws.sm_count * 16;
    if (nb > cap) nb = cap;
    if (nb < 1) nb = 1;
    launch_kernel(ws, K_AGG_DENSE, aggregate_dense_kernel, dim3((unsigned)nb), kRtnThreads, 0, s, val, level, M, d, ldv, out);
}

}  // namespace mlmc
