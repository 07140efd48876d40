// Queries of a Top-k selection, and its end: message headers, probabilities and the draw.
#pragma once

#include "common.cuh"

namespace mlmc {
namespace {

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
// keys K is added from their counts, |ranks of K  intersect  (k_{l-1}, k_l]| * val(K)^2; Delta_l = sqrt(E_l);
// p_l = Delta_l / sum Delta (Lemma 3.4); the level draw.  Then the header of the drawn band; `level` and `p_sel` are the
// level drawn on the host and its probability where p is given.
__device__ void finish_selection(const FinishPlan& pl, int m, int is_bf16, const Query* q, double* E, double* p_all,
                                 double* delta_all, int level, double p_sel, EmitParams* out, int* status, int* worker_err) {
    __shared__ double sh_p[kMaxLevels];
    __shared__ double sh_sum;
    const int L = pl.L;
    if (pl.adaptive) {
        const int l = threadIdx.x;
        if (l < L) {
            double x2 = E[l];
            const int64_t lo = l ? (int64_t)pl.k[l - 1] : 0, hi = (int64_t)pl.k[l];
            uint32_t prev_T = kKeyNone;
            for (int j = 0; j < L - 1; ++j) {
                if (q[j].trivial) continue;
                const uint32_t T = q[j].T;
                if (T == prev_T) continue;  // thresholds descend: the same key as the query before is counted once
                prev_T = T;
                const int64_t c0 = q[j].c, c1 = c0 + (int64_t)q[j].n;
                const int64_t ov = min(c1, hi) - max(c0, lo);
                if (ov > 0) {
                    const double x = (double)__uint_as_float(is_bf16 ? (T << 16) : T);
                    x2 = fma((double)ov, x * x, x2);
                }
            }
            E[l] = sqrt(x2);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int i = 0; i < L; ++i) s += E[i];
            sh_sum = s;
        }
        __syncthreads();
        if (l < L) {
            const double s = sh_sum;
            const double p = (s > 0.0) ? E[l] / s : (l == 0 ? 1.0 : 0.0);
            sh_p[l] = p;
            p_all[m * kMaxLevels + l] = p;
            delta_all[m * kMaxLevels + l] = E[l];
        }
        __syncthreads();
    }
    if (threadIdx.x != 0 || !pl.want_emit) return;
    if (pl.adaptive) {
        level = draw_from_probs(sh_p, L, counter_uniform(pl.seed, pl.step, (uint64_t)m));
        fill_emit(pl, m, level, sh_p[level], level ? &q[level - 1] : nullptr, level < L - 1 ? &q[level] : nullptr,
                  level ? pl.k[level - 1] : 0u, pl.k[level], out, status, worker_err);
    } else {
        fill_emit(pl, m, level, p_sel, &q[0], &q[1], q[0].k, q[1].k, out, status, worker_err);
    }
}

}  // namespace
}  // namespace mlmc
