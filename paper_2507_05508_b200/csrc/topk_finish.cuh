// Queries of a Top-k selection, and its end: message headers, probabilities and the draw.
#pragma once

#include "common.cuh"

namespace mlmc {

// Memory that a selection accumulates into.
struct ZeroList {
    static constexpr int kMost = 8;
    uint32_t* ptr[kMost];
    uint32_t words[kMost];
    int n;
};
// For nq queries per worker (topk_select.cu).
ZeroList selection_state(Workspace& ws, int dtype, int64_t d, int M, int nq, bool sums);

namespace {

__device__ __forceinline__ void clear_all(const ZeroList& z) {
    for (int a = 0; a < z.n; ++a) {
        uint32_t* p = z.ptr[a];
        const uint32_t n4 = z.words[a] / 4;
        for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x)
            reinterpret_cast<uint4*>(p)[i] = make_uint4(0u, 0u, 0u, 0u);
        for (uint32_t i = n4 * 4 + blockIdx.x * blockDim.x + threadIdx.x; i < z.words[a]; i += gridDim.x * blockDim.x) p[i] = 0u;
    }
}

__device__ __forceinline__ Query make_query(uint32_t k, int64_t d) {
    Query q = {};
    q.k = k;
    q.slot = kNoSlot;
    q.trivial = (k == 0u) ? 1u : ((int64_t)k >= d ? 2u : 0u);
    if (q.trivial == 1u) {
        q.T = kKeyNone;
    } else if (q.trivial == 2u) {
        q.T = 0u;
        q.r = 0xFFFFFFFFu;
    }
    return q;
}

// CAP workers fit the parameter list (24 KB of parameters at 1024 workers).
template <int CAP>
struct DrawnList {
    DrawnBand band[CAP];
};

// Header and emit parameters of one worker whose band (k_lo, k_hi] lies between the thresholds of two queries
// (null: no threshold on that side).  One thread.
__device__ void fill_emit(const FinishPlan& pl, int m, int level, double p_sel, const Query* q_lo, const Query* q_hi,
                          uint32_t k_lo, uint32_t k_hi, EmitParams* out, int* status, int* worker_err) {
    EmitParams e = {};
    e.level = level;
    e.Ta = q_lo ? q_lo->T : kKeyNone;
    e.ra = q_lo ? q_lo->r : 0u;
    e.Tb = q_hi ? q_hi->T : 0u;
    e.rb = q_hi ? q_hi->r : 0xFFFFFFFFu;
    e.inv_p = (p_sel > 0.0) ? 1.0 / p_sel : 0.0;
    e.expect = k_hi - k_lo;
    e.enabled = 1;
    if ((int64_t)e.expect > pl.capacity) {
        e.enabled = 0;
        worker_err[m] = MLMC_ERR_CAPACITY;
        set_status(status, MLMC_ERR_CAPACITY);
    }
    *out = e;
    pl.out_count[m] = e.enabled ? (int64_t)e.expect : 0;
    pl.out_level[m] = e.enabled ? level : -1;
    pl.out_p_sel[m] = p_sel;
}

__device__ void fail_worker(const FinishPlan& pl, int m, EmitParams* out) {
    if (!pl.want_emit) return;
    EmitParams e = {};
    e.level = -1;
    *out = e;
    pl.out_count[m] = 0;
    pl.out_level[m] = -1;
    pl.out_p_sel[m] = 0.0;
}

// The end of a selection, by one block per worker.  q: the worker's queries (in shared memory, complete).
// Adaptive: E[l] = energy of the entries strictly between two thresholds (shared memory); the energy of the threshold
// keys is added from their counts: of the keys equal to T_{l-1} the n - r past rank k_{l-1}, of those equal to T_l the first
// r; Delta_l = sqrt(E_l); p_l = Delta_l / sum Delta (Lemma 3.4); the level draw.  Then the header of the drawn band;
// `level` and `p_sel` are the level drawn on the host and its probability where p is given.  A level per lane of warp 0.
__device__ void finish_selection(const FinishPlan& pl, int m, int is_bf16, const Query* q, const double* E, double* p_all,
                                 double* delta_all, int level, double p_sel, EmitParams* out, int* status, int* worker_err) {
    if (threadIdx.x >= 32) return;
    const int L = pl.L, l = threadIdx.x;
    if (pl.adaptive) {
        double delta = 0.0;
        if (l < L) {
            const Query* up = (l > 0 && q[l - 1].trivial == 0u) ? &q[l - 1] : nullptr;
            const Query* dn = (l < L - 1 && q[l].trivial == 0u) ? &q[l] : nullptr;
            auto square = [&](uint32_t T) -> double {
                const double x = (double)__uint_as_float(is_bf16 ? (T << 16) : T);
                return x * x;
            };
            double e = E[l];
            if (up && dn && up->T == dn->T) {
                e = fma((double)(pl.k[l] - pl.k[l - 1]), square(dn->T), e);  // the whole band is ties
            } else {
                if (up) e = fma((double)(up->n - up->r), square(up->T), e);
                if (dn) e = fma((double)dn->r, square(dn->T), e);
            }
            delta = sqrt(e);
        }
        double p;
        level = warp_draw(delta, L, counter_uniform(pl.seed, pl.step, (uint64_t)m), &p);
        if (l < L) {
            p_all[m * kMaxLevels + l] = p;
            delta_all[m * kMaxLevels + l] = delta;
        }
        if (!pl.want_emit) return;
        p_sel = __shfl_sync(0xFFFFFFFFu, p, level);
        if (l == 0)
            fill_emit(pl, m, level, p_sel, level ? &q[level - 1] : nullptr, level < L - 1 ? &q[level] : nullptr,
                      level ? pl.k[level - 1] : 0u, pl.k[level], out, status, worker_err);
    } else if (l == 0 && pl.want_emit) {
        fill_emit(pl, m, level, p_sel, &q[0], &q[1], q[0].k, q[1].k, out, status, worker_err);
    }
}

}  // namespace
}  // namespace mlmc
