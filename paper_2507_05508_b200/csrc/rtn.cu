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

#include "common.cuh"

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
    if (!(gq.inv <= 3.0e38f)) return v;  // c below the normal range: 1 / delta overflows, and 0 inv is not a number
    uint32_t z = min(__float_as_uint(0.5f / gq.inv), 0x7F7FFFFFu);
    while (z > 0u && __fmul_rn(__uint_as_float(z), gq.inv) > 0.5f) --z;
    while (z < 0x7F7FFFFFu && __fmul_rn(__uint_as_float(z + 1u), gq.inv) <= 0.5f) ++z;
    v.zero_upto = (int)z;
    const float f = c - gq.delta;  // |k delta| <= |v| + delta / 2 (1 + 2^-20)
    if (f > 0.0f) v.free_upto = __float_as_int(f);
    return v;
}

// Residual energies of every level: partial[m][block][l] = sum over the block's entries of (C^l - C^{l-1})^2.
// A warp takes the entries level by level, kRtnHeld per lane.  The levels whose grid is so coarse that the largest of the
// warp's entries rounds to 0 contribute nothing and are skipped: the clipping value is the row's largest magnitude, and
// in a gradient with per-layer scales most entries are small beside it.  The first level that is left has C^{l-1} = 0, so
// its residual is its value.  The differences and sums are fp64 (a difference of two fp32 values is exact); what bounds the
// kernel where nothing is skipped is the conversion of one fp32 value to fp64 per entry and level (16 per clock and SM).
// 8 x 124M fp32 entries, L = 5: 2.29 ms with every entry taken through every level; 1.02 with one trip in flight and one and
// a half waves of blocks, now 0.87.
constexpr int kRtnHeld = 8;

template <typename T, int LMAX>
__global__ void __launch_bounds__(kRtnThreads, LMAX <= 6 ? 4 : 3)
rtn_stats_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const uint32_t* gmax_bits, const __grid_constant__ RtnSchedule sc, double* partial,
                 int rtn_ctas, uint32_t* done, const __grid_constant__ DrawPlan pl, int* status, int* worker_err) {
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
    auto take = [&](const float (&v)[kRtnHeld]) {
        int mx = 0;
#pragma unroll
        for (int e = 0; e < kRtnHeld; ++e) mx = max(mx, __float_as_int(v[e]) & 0x7FFFFFFF);
        mx = __reduce_max_sync(0xFFFFFFFFu, mx);
        double prev[kRtnHeld];  // C^{l-1}
        bool first = true;      // C^{l-1} = 0 for every entry of the warp (warp-uniform)
#pragma unroll
        for (int l = 0; l < LMAX; ++l) {
            if (l > sc.L - 1) break;
            if (l == sc.L - 1) {  // the identity
#pragma unroll
                for (int e = 0; e < kRtnHeld; ++e) {
                    const double res = first ? (double)v[e] : (double)v[e] - prev[e];
                    acc[l] = fma(res, res, acc[l]);
                }
                break;
            }
            const RtnLevel lv = sh_lv[l];
            if (mx <= lv.zero_upto) continue;  // the grids get finer: once a level is not skipped, none after it is
            float x[kRtnHeld];
#pragma unroll
            for (int e = 0; e < kRtnHeld; ++e) {
                const float k = __fadd_rn(__fadd_rn(__fmul_rn(v[e], lv.inv), 12582912.0f), -12582912.0f);
                x[e] = __fmul_rn(k, lv.delta);
            }
            if (mx > lv.free_upto) {
#pragma unroll
                for (int e = 0; e < kRtnHeld; ++e) x[e] = fminf(fmaxf(x[e], -c), c);
            }
            if (first) {
#pragma unroll
                for (int e = 0; e < kRtnHeld; ++e) {
                    prev[e] = (double)x[e];
                    acc[l] = fma(prev[e], prev[e], acc[l]);
                }
                first = false;
            } else {
#pragma unroll
                for (int e = 0; e < kRtnHeld; ++e) {
                    const double cur = (double)x[e], res = cur - prev[e];
                    acc[l] = fma(res, res, acc[l]);
                    prev[e] = cur;
                }
            }
        }
    };
    if (c > 0.0f) {
        const T* row = g + (int64_t)m * ld;
        constexpr int kVecs = kRtnHeld / Tr::kVec;  // 16-byte vectors per lane and trip
        constexpr int kTrip = kRtnThreads * kVecs;
        const int64_t full_end = d / Tr::kVec;
        const int64_t trips = full_end / kTrip;
        auto expand = [&](const uint4 (&q)[kVecs], float (&v)[kRtnHeld]) {
#pragma unroll
            for (int j = 0; j < kVecs; ++j) {
                const uint32_t w[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    if constexpr (Tr::kVec == 4) {
                        v[4 * j + i] = __uint_as_float(w[i]);
                    } else {
                        v[8 * j + 2 * i] = __uint_as_float(w[i] << 16);
                        v[8 * j + 2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u);
                    }
                }
            }
        };
        stream_trips<kVecs, kRtnThreads>(reinterpret_cast<const uint4*>(row), blockIdx.x, gridDim.x, trips, sh_vectors, [&](const uint4 (&q)[kVecs]) {
            float v[kRtnHeld];
            expand(q, v);
            take(v);
        });
        if (blockIdx.x == gridDim.x - 1) {  // the rest of the row, fewer than kTrip + 1 vectors, one by one
            for (int64_t i = trips * kTrip * Tr::kVec + threadIdx.x; i < d; i += kRtnThreads) {
                float v;
                if constexpr (Tr::kVec == 4) v = reinterpret_cast<const float*>(row)[i];
                else v = __uint_as_float((uint32_t)reinterpret_cast<const uint16_t*>(row)[i] << 16);
                double prev = 0.0;
#pragma unroll
                for (int l = 0; l < LMAX; ++l) {
                    if (l > sc.L - 1) break;
                    const double cur = (l < sc.L - 1) ? (double)rtn_value(v, c, {sh_lv[l].inv, sh_lv[l].delta}) : (double)v;
                    acc[l] = fma(cur - prev, cur - prev, acc[l]);
                    prev = cur;
                }
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

// The dense message of the drawn level: val_i = (C^l - C^{l-1})_i / p_l, rounded to fp32 once.
template <typename T>
__global__ void __launch_bounds__(kRtnThreads)
rtn_emit_kernel(const T* __restrict__ g, int64_t d, int64_t ld, const uint32_t* gmax_bits, RtnSchedule sc,
                const int32_t* bit_level, const double* p_all, float* __restrict__ val, int64_t ldv) {
    using Tr = ElemTraits<T>;
    pdl_enter();
    const int m = blockIdx.y;
    const int level = bit_level[m];
    if (level < 0) return;
    const float c = __uint_as_float(gmax_bits[m]);
    const double p = p_all[m * kMaxLevels + level];
    const double inv_p = p > 0.0 ? 1.0 / p : 0.0;
    const bool top = level == sc.L - 1, first = level == 0;
    const RtnGrid g_hi = rtn_grid(c > 0.0f ? c : 1.0f, top ? 1 : sc.r[level]);
    const RtnGrid g_lo = rtn_grid(c > 0.0f ? c : 1.0f, first ? 1 : sc.r[level - 1]);
    const T* row = g + (int64_t)m * ld;
    float* out = val + (int64_t)m * ldv;
    auto residual = [&](uint32_t bits) -> float {
        const float v = Tr::value(bits);
        if (!(c > 0.0f)) return 0.0f;
        const double hi = top ? (double)v : (double)rtn_value(v, c, g_hi);
        const double lo = first ? 0.0 : (double)rtn_value(v, c, g_lo);
        return (float)((hi - lo) * inv_p);
    };
    const int64_t nvec = (d + Tr::kVec - 1) / Tr::kVec;
    const bool vec_ok = (ldv % 4 == 0);
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < nvec; v += (int64_t)gridDim.x * blockDim.x) {
        const int64_t base = v * Tr::kVec;
        if (base + Tr::kVec <= d && vec_ok) {
            const uint4 q = __ldg(reinterpret_cast<const uint4*>(row) + v);
            if constexpr (Tr::kVec == 4) {
                reinterpret_cast<float4*>(out + base)[0] = make_float4(residual(q.x), residual(q.y), residual(q.z), residual(q.w));
            } else {
                reinterpret_cast<float4*>(out + base)[0] =
                    make_float4(residual(q.x & 0xFFFFu), residual(q.x >> 16), residual(q.y & 0xFFFFu), residual(q.y >> 16));
                reinterpret_cast<float4*>(out + base)[1] =
                    make_float4(residual(q.z & 0xFFFFu), residual(q.z >> 16), residual(q.w & 0xFFFFu), residual(q.w >> 16));
            }
        } else {
            for_each_in_vector<T>(row, v, d, [&](int64_t i, uint32_t bits) { out[i] = residual(bits); });
        }
    }
}

// Server average of dense messages: out[i] = (1/M) sum_m val[m][i] in worker order.
__global__ void __launch_bounds__(kRtnThreads)
aggregate_dense_kernel(const float* __restrict__ val, const int32_t* level, int M, int64_t d, int64_t ldv,
                       float* __restrict__ out) {
    pdl_enter();
    const float inv_M = 1.0f / (float)M;
    const bool vec_ok = (ldv % 4 == 0) && (d % 4 == 0);
    if (vec_ok) {
        const int64_t n4 = d / 4;
        for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n4; v += (int64_t)gridDim.x * blockDim.x) {
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int m = 0; m < M; ++m) {
                if (level[m] < 0) continue;
                const float4 x = __ldg(reinterpret_cast<const float4*>(val + (int64_t)m * ldv) + v);
                a.x += x.x; a.y += x.y; a.z += x.z; a.w += x.w;
            }
            a.x *= inv_M; a.y *= inv_M; a.z *= inv_M; a.w *= inv_M;
            reinterpret_cast<float4*>(out)[v] = a;
        }
    } else {
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < d; i += (int64_t)gridDim.x * blockDim.x) {
            float a = 0.f;
            for (int m = 0; m < M; ++m)
                if (level[m] >= 0) a += val[(int64_t)m * ldv + i];
            out[i] = a * inv_M;
        }
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
template <typename T, int LMAX>
void launch_rtn_stats_t(Workspace& ws, const T* g, int64_t d, int M, int64_t ld, const RtnSchedule& sc, const DrawPlan& plan,
                        cudaStream_t s) {
    constexpr size_t smem = (size_t)4 * kRtnThreads * kRtnHeld * sizeof(T);
    static const int resident = resident_blocks(rtn_stats_kernel<T, LMAX>, kRtnThreads, smem);
    // whole waves (a partial last one costs a full one), four of them: how much a block skips differs (one: 910 us, two: 897,
    // four: 866 for 8 x 124M entries)
    const int nb = std::min(rtn_blocks(ws, d, ElemTraits<T>::kVec, M, 4 * resident), ws.rtn_ctas);
    launch_kernel(ws, K_RTN_STATS, rtn_stats_kernel<T, LMAX>, dim3(nb, M), kRtnThreads, smem, s, g, d, ld, ws.gmax_bits, sc,
                  ws.rtn_partial, ws.rtn_ctas, ws.done, plan, ws.status, ws.worker_err);
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

void launch_rtn_emit(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                     const mlmc_rtn_msgs& out, cudaStream_t s) {
    const RtnSchedule sc = make_rtn_schedule(r, L);
    const int nb = rtn_blocks(ws, d, dtype == MLMC_BF16 ? 8 : 4, M, 16);
    auto go = [&](auto kernel, auto* row) {
        launch_kernel(ws, K_RTN_EMIT, kernel, dim3(nb, M), kRtnThreads, 0, s, row, d, ld, ws.gmax_bits, sc, ws.bit_level,
                      ws.p_all, out.val, out.ldv);
    };
    if (dtype == MLMC_BF16) go(rtn_emit_kernel<bf16_t>, static_cast<const bf16_t*>(g));
    else go(rtn_emit_kernel<float>, static_cast<const float*>(g));
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
