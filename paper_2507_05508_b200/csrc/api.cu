// C ABI of the MLMC compression library: context, argument checks and the launch sequences.
#include <mutex>
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "stopk_sort.cuh"

using namespace mlmc;

struct mlmc_ctx {
    Workspace ws;
    void* slab;
    size_t slab_bytes;
};

namespace {

struct SlabPlanner {
    size_t off = 0;
    size_t take(size_t bytes) {
        const size_t at = off;
        off += (bytes + 255) & ~size_t(255);
        return at;
    }
};

struct DeviceGuard {
    int prev = -1;
    bool ok = true;
    explicit DeviceGuard(int dev) {
        ok = cudaGetDevice(&prev) == cudaSuccess && (prev == dev || cudaSetDevice(dev) == cudaSuccess);
        if (prev == dev) prev = -1;  // nothing to put back
    }
    ~DeviceGuard() {
        if (prev >= 0) cudaSetDevice(prev);
    }
};

int check_common(const mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, int L) {
    if (!ctx || !g) return MLMC_ERR_ARG;
    if (dtype != MLMC_F32 && dtype != MLMC_BF16) return MLMC_ERR_ARG;
    if (d < 1 || d > ctx->ws.d_max || d >= (int64_t(1) << 32)) return MLMC_ERR_ARG;
    if (M < 1 || M > ctx->ws.M_max) return MLMC_ERR_ARG;
    if (L < 1 || L > ctx->ws.L_max) return MLMC_ERR_ARG;
    if (ld < d) return MLMC_ERR_ARG;
    const int64_t esize = (dtype == MLMC_BF16) ? 2 : 4;
    if (reinterpret_cast<uintptr_t>(g) % 16 != 0) return MLMC_ERR_ARG;
    if (M > 1 && (ld * esize) % 16 != 0) return MLMC_ERR_ARG;
    return MLMC_OK;
}

int check_topk_schedule(const int64_t* k, int L, int64_t d) {
    if (!k) return MLMC_ERR_ARG;
    int64_t prev = 0;
    for (int l = 0; l < L; ++l) {
        if (k[l] < prev || k[l] > d) return MLMC_ERR_SCHEDULE;
        prev = k[l];
    }
    return k[L - 1] == d ? MLMC_OK : MLMC_ERR_SCHEDULE;  // Def. 3.1: the top level is the identity
}

template <typename I>
int check_bit_schedule(const I* b, int L, int32_t* b32) {
    if (!b) return MLMC_ERR_ARG;
    int64_t prev = 0;
    for (int l = 0; l < L; ++l) {
        if (b[l] <= prev || b[l] > 23) return MLMC_ERR_SCHEDULE;
        prev = b[l];
        b32[l] = (int32_t)b[l];
    }
    return MLMC_OK;
}

// RTN widths r_0 < ... < r_{L-2} <= 16 (App. G); level L-1 is the identity and has no width.
template <typename I>
int check_rtn_schedule(const I* r, int L, int32_t* r32) {
    if (L < 1 || L > 17) return MLMC_ERR_ARG;
    if (L > 1 && !r) return MLMC_ERR_ARG;
    int64_t prev = 0;
    for (int l = 0; l + 1 < L; ++l) {
        if (r[l] <= prev || r[l] > 16) return MLMC_ERR_SCHEDULE;
        prev = r[l];
        r32[l] = (int32_t)r[l];
    }
    return MLMC_OK;
}

// Mantissa digits mb_0 < ... < mb_{L-1} = F kept by the floating-point levels (App. B); the top level is the identity.
int check_mantissa_schedule(const int32_t* mb, int L, int F) {
    if (!mb) return MLMC_ERR_ARG;
    int prev = 0;
    for (int l = 0; l < L; ++l) {
        if (mb[l] <= prev || mb[l] > F) return MLMC_ERR_SCHEDULE;
        prev = mb[l];
    }
    return mb[L - 1] == F ? MLMC_OK : MLMC_ERR_SCHEDULE;
}

// Lemma 3.2 asks for non-zero probabilities; they are renormalised in fp64.
int normalise_probs(const double* p, int L, double* out) {
    double s = 0.0;
    for (int l = 0; l < L; ++l) {
        if (!(p[l] > 0.0) || !std::isfinite(p[l])) return MLMC_ERR_PROB;
        s += p[l];
    }
    if (std::fabs(s - 1.0) > 1e-9) return MLMC_ERR_PROB;
    for (int l = 0; l < L; ++l) out[l] = p[l] / s;
    return MLMC_OK;
}

int finish(cudaError_t e) { return e == cudaSuccess ? MLMC_OK : MLMC_ERR_CUDA; }

// The selection of a call: thresholds of every query, for adaptive p the probabilities and the draw, the headers.
// brackets (given p, fp32): the first sweep also collects the keys of the bins around last call's boundary bins;
// where both boundary bins of a worker's band fall inside, the candidate sweep has nothing left to do.
void run_selection(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const FinishPlan& plan, bool brackets,
                   cudaStream_t s) {
    launch_hist1(ws, g, dtype, d, M, ld, brackets, nullptr, s);
    launch_resolve1(ws, dtype, M, plan, brackets, false, nullptr, s);
    if (dtype == MLMC_F32) {
        launch_sums_candidates(ws, g, d, M, ld, plan, brackets, nullptr, s);
        launch_digit_passes(ws, g, d, M, ld, plan, false, s);
    }
}

// The same with brackets from a sample of the rows: one sweep.  The three launches in the middle are for workers whose
// brackets missed, and return at once for the others.
void run_sampled_selection(Workspace& ws, const void* g, int64_t d, int M, int64_t ld, const int64_t* k, const FinishPlan& plan,
                           cudaStream_t s) {
    launch_bracket_sweep(ws, static_cast<const float*>(g), d, M, ld, k, plan, s);
    launch_resolve1(ws, MLMC_F32, M, plan, false, true, ws.miss, s);
    launch_hist1(ws, g, MLMC_F32, d, M, ld, false, ws.miss, s);
    launch_resolve1(ws, MLMC_F32, M, plan, false, false, ws.miss, s);
    launch_sums_candidates(ws, g, d, M, ld, plan, false, ws.miss, s);
    launch_digit_passes(ws, g, d, M, ld, plan, true, s);
}

FinishPlan finish_plan(int64_t d, int L, int nq, bool adaptive, uint64_t seed, uint64_t step, const mlmc_topk_msgs* out) {
    FinishPlan pl = {};
    pl.L = L;
    pl.nq = nq;
    pl.adaptive = adaptive ? 1 : 0;
    pl.want_emit = out ? 1 : 0;
    pl.d = d;
    pl.seed = seed;
    pl.step = step;
    if (out) {
        pl.out_count = out->count;
        pl.out_level = out->level;
        pl.out_p_sel = out->p_sel;
        pl.capacity = out->capacity;
    }
    return pl;
}

// Adaptive p: every level boundary is a query.  Rows that a cluster's shared memory holds (at most 2.9 MB) take one launch.
void select_adaptive(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, const int64_t* k, int L,
                     uint64_t seed, uint64_t step, const mlmc_topk_msgs* out, cudaStream_t s) {
    FinishPlan pl = finish_plan(d, L, L - 1, true, seed, step, out);
    for (int l = 0; l < L; ++l) pl.k[l] = (uint32_t)k[l];
    if (cluster_blocks(ws, dtype, d, M, false) > 0) {
        launch_cluster_topk(ws, g, dtype, d, M, ld, pl, nullptr, out, s);
        return;
    }
    if (use_brackets(ws, dtype, d, M, k, L)) {
        run_sampled_selection(ws, g, d, M, ld, k, pl, s);
    } else {
        launch_begin_adaptive(ws, dtype, d, M, k, L, s);
        run_selection(ws, g, dtype, d, M, ld, pl, false, s);
    }
    if (out) launch_emit(ws, g, dtype, d, M, ld, *out, s);
}

// Longer fp32 rows use last call's boundary bins as brackets instead, where the call keeps them.
constexpr int64_t kClusterDrawnBytes = 1 << 20;

// Given p: the level of every worker is drawn here (it depends on seed, step and worker only), and the two ranks that
// bound its band are the only queries.
template <typename Draw>
void select_drawn(Workspace& ws, const void* g, int dtype, int64_t d, int M, int64_t ld, int L, bool brackets, uint64_t seed,
                  uint64_t step, const mlmc_topk_msgs* out, Draw&& draw, cudaStream_t s) {
    brackets = brackets && dtype == MLMC_F32 && L > 1;
    DrawnBand bands[kEmitMaxWorkers];
    for (int m = 0; m < M; ++m) bands[m] = draw(counter_uniform(seed, step, (uint64_t)m));
    const FinishPlan pl = finish_plan(d, L, 2, false, seed, step, out);
    if ((!brackets || d * (int64_t)sizeof(float) <= kClusterDrawnBytes) && cluster_blocks(ws, dtype, d, M, true) > 0) {
        launch_cluster_topk(ws, g, dtype, d, M, ld, pl, bands, out, s);
        return;
    }
    launch_begin_drawn(ws, dtype, d, M, bands, L, brackets, s);
    run_selection(ws, g, dtype, d, M, ld, pl, brackets, s);
    launch_emit(ws, g, dtype, d, M, ld, *out, s);
}

// The kernels' shared-memory limits and cluster attributes belong to the current CUDA context (a device reset starts a new one),
// so every create sets them.  What the device can place is asked for once per device: the queries take a millisecond.
bool configure_kernels(int device, KernelLimits* out) {
    if (configure_select_kernels() != MLMC_OK || configure_bracket_kernels() != MLMC_OK || configure_emit_kernels() != MLMC_OK || configure_float_kernels() != MLMC_OK ||
        configure_segment_kernels() != MLMC_OK || configure_sort_kernels() != MLMC_OK || configure_rtn_kernels() != MLMC_OK ||
        configure_cluster_kernels() != MLMC_OK || configure_bit_kernels() != MLMC_OK)
        return false;
    constexpr int kMostDevices = 64;
    static std::mutex lock;
    static bool known[kMostDevices];
    static KernelLimits limits[kMostDevices];
    std::lock_guard<std::mutex> hold(lock);
    const bool keep = device < kMostDevices;
    if (keep && known[device]) {
        *out = limits[device];
        return true;
    }
    KernelLimits l = {};
    emit_limits(&l);
    bracket_limits(&l);
    float_limits(&l);
    sort_limits(&l);
    rtn_limits(&l);
    cluster_limits(&l);
    bit_limits(&l);
    if (keep) {
        limits[device] = l;
        known[device] = true;
    }
    *out = l;
    return true;
}

}  // namespace

extern "C" {

int mlmc_create(mlmc_ctx** out, int device, int64_t d_max, int M_max, int L_max) {
    if (!out || d_max < 1 || d_max >= (int64_t(1) << 32) || M_max < 1 || M_max > kEmitMaxWorkers || L_max < 1 ||
        L_max > kMaxLevels)
        return MLMC_ERR_ARG;
    DeviceGuard guard(device);
    if (!guard.ok) return MLMC_ERR_CUDA;
    int sms = 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return MLMC_ERR_CUDA;
    KernelLimits limits;
    if (!configure_kernels(device, &limits)) return MLMC_ERR_CUDA;

    mlmc_ctx* ctx = new (std::nothrow) mlmc_ctx();
    if (!ctx) return MLMC_ERR_NOMEM;
    Workspace& ws = ctx->ws;
    ws.limits = limits;
    ws.device = device;
    ws.d_max = d_max;
    ws.M_max = M_max;
    ws.L_max = L_max;
    ws.sm_count = sms;
    ws.launches = 0;
    ws.timing = false;
    ws.last_emit_tiles = 0;
    ws.timing_used = 0;
    ws.ev_start = ws.ev_stop = nullptr;
    ws.ev_id = nullptr;
    for (int i = 0; i < K_COUNT; ++i) ws.launches_by_id[i] = 0;
    ws.sum_ctas = ws.sm_count * 4;
    ws.cur_sum_ctas = 0;
    // candidate keys: a quarter of the row (boundary bins normally hold a few percent of it); small rows fit whole
    ws.cand_cap = d_max / 4 > (int64_t(1) << 20) ? d_max / 4 : (d_max < (int64_t(1) << 20) ? d_max : (int64_t(1) << 20));
    ws.cand_cap = (ws.cand_cap + 3) & ~int64_t(3);  // 16-byte rows
    ws.stat_ctas = ws.sm_count * 4;
    const int64_t emit_tiles = (d_max + kEmitTile - 1) / kEmitTile;
    const int64_t agg_tiles = (d_max + kAggTile - 1) / kAggTile;
    ws.max_tiles = emit_tiles * M_max;

    SlabPlanner pl;
    const size_t o_status = pl.take(sizeof(int));
    const size_t o_werr = pl.take(sizeof(int) * M_max);
    const size_t o_hist1 = pl.take(sizeof(uint32_t) * kBins1 * M_max);
    const size_t o_table1 = pl.take((size_t)kBins1 * M_max);
    const size_t o_hist23 = pl.take(sizeof(uint32_t) * kMaxQueries * kBins23 * 2 * M_max);
    const size_t o_map2 = pl.take((size_t)kMaxQueries * kBins23 * M_max);
    const size_t o_done = pl.take(sizeof(uint32_t) * M_max);
    const size_t o_acc = pl.take(sizeof(uint32_t) * 2 * M_max);
    const size_t o_queries = pl.take(sizeof(Query) * kMaxQueries * M_max);
    const size_t o_sum = pl.take(sizeof(double) * kMaxLevels * ws.sum_ctas * M_max);
    const size_t o_cpart = pl.take(sizeof(unsigned long long) * kEnergyCells * 2 * M_max);
    const size_t o_ckeys = pl.take(sizeof(uint32_t) * ws.cand_cap * M_max);
    const size_t o_ccount = pl.take(sizeof(uint32_t) * M_max);
    const size_t o_cover = pl.take(sizeof(int) * M_max);
    const size_t o_pall = pl.take(sizeof(double) * kMaxLevels * M_max);
    const size_t o_dall = pl.take(sizeof(double) * kMaxLevels * M_max);
    const size_t o_u = pl.take(sizeof(double) * M_max);
    const size_t o_emit = pl.take(sizeof(EmitParams) * M_max);
    const size_t o_tdesc = pl.take(sizeof(uint4) * ws.max_tiles);
    const size_t o_ldesc = pl.take(sizeof(uint4) * emit_counts((int)emit_tiles).total() * M_max);
    const size_t o_tlist = pl.take(sizeof(uint2) * ws.max_tiles);
    const size_t o_listn = pl.take(sizeof(uint32_t));
    const size_t o_tmax = pl.take(sizeof(uint32_t) * ws.max_tiles * kEmitGroups);
    const size_t o_groupn = pl.take(sizeof(uint32_t) * M_max);
    const size_t o_cfloor = pl.take(sizeof(uint32_t) * M_max);
    const size_t o_aggoff = pl.take(sizeof(uint32_t) * (agg_tiles + 1) * M_max);
    const size_t o_gmax = pl.take(sizeof(uint32_t) * 2 * M_max);
    const size_t o_S = pl.take(sizeof(unsigned long long) * kMaxLevels * ws.stat_ctas * M_max);
    const size_t o_blevel = pl.take(sizeof(int32_t) * M_max);
    ws.big_cap = d_max < (int64_t(1) << 20) ? d_max : (int64_t(1) << 20);
    ws.rtn_ctas = ws.sm_count * 8;
    const size_t o_rtn = pl.take(sizeof(double) * kMaxLevels * ws.rtn_ctas * M_max);
    const size_t o_pbin = pl.take(sizeof(uint32_t) * kMaxLevels * M_max);
    const size_t o_brk = pl.take(sizeof(uint4) * M_max);
    const size_t o_bhit = pl.take(sizeof(int) * M_max);
    const size_t o_bstat = pl.take(sizeof(unsigned long long) * 8);
    const size_t o_runs = pl.take(sizeof(BracketRuns) * M_max);
    const size_t o_miss = pl.take(sizeof(int) * M_max);
    // one block of up to 32 warps per SM, or one per worker where there are more workers than SMs
    const size_t o_partn = pl.take(sizeof(uint32_t) * 32 * std::max(ws.sm_count, M_max));
    ws.seg_scratch = nullptr;
    ws.seg_bytes = 0;
    ws.sig_d = ws.sig_ld = -1;
    ws.sig_M = ws.sig_L = ws.sig_dtype = -1;

    ctx->slab_bytes = pl.off;
    if (cudaMalloc(&ctx->slab, ctx->slab_bytes) != cudaSuccess) {
        cudaGetLastError();
        delete ctx;
        return MLMC_ERR_NOMEM;
    }
    if (cudaMemset(ctx->slab, 0, ctx->slab_bytes) != cudaSuccess) {
        cudaFree(ctx->slab);
        delete ctx;
        return MLMC_ERR_CUDA;
    }
    char* base = static_cast<char*>(ctx->slab);
    ws.status = reinterpret_cast<int*>(base + o_status);
    ws.worker_err = reinterpret_cast<int*>(base + o_werr);
    ws.hist1 = reinterpret_cast<uint32_t*>(base + o_hist1);
    ws.table1 = reinterpret_cast<uint8_t*>(base + o_table1);
    ws.hist2 = ws.hist3 = reinterpret_cast<uint32_t*>(base + o_hist23);
    ws.map2 = reinterpret_cast<uint8_t*>(base + o_map2);
    ws.done = reinterpret_cast<uint32_t*>(base + o_done);
    ws.acc_word = reinterpret_cast<uint32_t*>(base + o_acc);
    ws.queries = reinterpret_cast<Query*>(base + o_queries);
    ws.sum_partial = reinterpret_cast<double*>(base + o_sum);
    ws.cand_S = reinterpret_cast<unsigned long long*>(base + o_cpart);
    ws.cand_keys = reinterpret_cast<uint32_t*>(base + o_ckeys);
    ws.cand_count = reinterpret_cast<uint32_t*>(base + o_ccount);
    ws.cand_overflow = reinterpret_cast<int*>(base + o_cover);
    ws.p_all = reinterpret_cast<double*>(base + o_pall);
    ws.delta_all = reinterpret_cast<double*>(base + o_dall);
    ws.u_dev = reinterpret_cast<double*>(base + o_u);
    ws.emit = reinterpret_cast<EmitParams*>(base + o_emit);
    ws.tile_desc = reinterpret_cast<uint4*>(base + o_tdesc);
    ws.level_desc = reinterpret_cast<uint4*>(base + o_ldesc);
    ws.tile_list = reinterpret_cast<uint2*>(base + o_tlist);
    ws.list_n = reinterpret_cast<uint32_t*>(base + o_listn);
    ws.tile_max = reinterpret_cast<uint32_t*>(base + o_tmax);
    ws.group_n = reinterpret_cast<uint32_t*>(base + o_groupn);
    ws.cand_floor = reinterpret_cast<uint32_t*>(base + o_cfloor);
    ws.agg_offsets = reinterpret_cast<uint32_t*>(base + o_aggoff);
    ws.gmax_bits = reinterpret_cast<uint32_t*>(base + o_gmax);
    ws.S_partial = reinterpret_cast<unsigned long long*>(base + o_S);
    ws.bit_level = reinterpret_cast<int32_t*>(base + o_blevel);
    ws.rtn_partial = reinterpret_cast<double*>(base + o_rtn);
    ws.runs = reinterpret_cast<BracketRuns*>(base + o_runs);
    ws.miss = reinterpret_cast<int*>(base + o_miss);
    ws.part_n = reinterpret_cast<uint32_t*>(base + o_partn);
    ws.prev_bin = reinterpret_cast<uint32_t*>(base + o_pbin);
    ws.bracket = reinterpret_cast<uint4*>(base + o_brk);
    ws.bracket_hit = reinterpret_cast<int*>(base + o_bhit);
    ws.bracket_stats = reinterpret_cast<unsigned long long*>(base + o_bstat);
    cudaMemset(ws.prev_bin, 0xFF, sizeof(uint32_t) * kMaxLevels * M_max);
    if (cudaDeviceSynchronize() != cudaSuccess) {
        cudaFree(ctx->slab);
        delete ctx;
        return MLMC_ERR_CUDA;
    }
    *out = ctx;
    return MLMC_OK;
}

int mlmc_destroy(mlmc_ctx* ctx) {
    if (!ctx) return MLMC_ERR_ARG;
    DeviceGuard guard(ctx->ws.device);
    cudaDeviceSynchronize();
    if (ctx->ws.ev_start) {
        for (int i = 0; i < kTimingPool; ++i) {
            cudaEventDestroy(ctx->ws.ev_start[i]);
            cudaEventDestroy(ctx->ws.ev_stop[i]);
        }
        delete[] ctx->ws.ev_start;
        delete[] ctx->ws.ev_stop;
        delete[] ctx->ws.ev_id;
    }
    if (ctx->ws.seg_scratch) cudaFree(ctx->ws.seg_scratch);
    const cudaError_t e = cudaFree(ctx->slab);
    delete ctx;
    return finish(e);
}

int mlmc_get_status(mlmc_ctx* ctx, void* stream) {
    if (!ctx) return MLMC_ERR_ARG;
    DeviceGuard guard(ctx->ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int st = 0;
    if (cudaMemcpyAsync(&st, ctx->ws.status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return MLMC_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return MLMC_ERR_CUDA;
    if (st != 0) {
        if (cudaMemsetAsync(ctx->ws.status, 0, sizeof(int), s) != cudaSuccess) return MLMC_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return MLMC_ERR_CUDA;
    }
    return st;
}

int64_t mlmc_launch_count(const mlmc_ctx* ctx) { return ctx ? ctx->ws.launches : 0; }

static const char* const kKernelNames[] = {
    "begin", "uniforms", "hist1", "resolve1", "sums_candidates", "cand_pass2", "cand_pass3", "band_header", "copy_probs", "emit",
    "agg_offsets", "aggregate_topk", "absmax", "bit_stats", "bit_pack", "aggregate_bitwise", "tile_list", "band_count",
    "float_pack", "aggregate_floatbits", "rtn_stats", "rtn_emit", "aggregate_dense", "segment_resolve",
    "segment_sweep", "segment_buckets", "segment_norms", "segment_draw", "cluster_topk", "cluster_bitwise", "cluster_rtn", "sort_rows",
    "sample", "bracket_sweep", "candidate_hist", "missed_hist1", "missed_sums"};
static_assert(sizeof(kKernelNames) / sizeof(kKernelNames[0]) == K_COUNT, "a name for every kernel id");

int mlmc_kernel_count(void) { return K_COUNT; }

const char* mlmc_kernel_name(int id) { return (id >= 0 && id < K_COUNT) ? kKernelNames[id] : ""; }

int mlmc_timing_enable(mlmc_ctx* ctx, int on) {
    if (!ctx) return MLMC_ERR_ARG;
    Workspace& ws = ctx->ws;
    DeviceGuard guard(ws.device);
    if (on && !ws.ev_start) {
        ws.ev_start = new (std::nothrow) cudaEvent_t[kTimingPool];
        ws.ev_stop = new (std::nothrow) cudaEvent_t[kTimingPool];
        ws.ev_id = new (std::nothrow) int[kTimingPool];
        if (!ws.ev_start || !ws.ev_stop || !ws.ev_id) return MLMC_ERR_NOMEM;
        for (int i = 0; i < kTimingPool; ++i)
            if (cudaEventCreate(&ws.ev_start[i]) != cudaSuccess || cudaEventCreate(&ws.ev_stop[i]) != cudaSuccess)
                return MLMC_ERR_CUDA;
    }
    ws.timing = on != 0;
    ws.timing_used = 0;
    return MLMC_OK;
}

int mlmc_timing_read(mlmc_ctx* ctx, double* total_ms, int64_t* launches, void* stream) {
    if (!ctx || !total_ms || !launches) return MLMC_ERR_ARG;
    Workspace& ws = ctx->ws;
    DeviceGuard guard(ws.device);
    if (cudaStreamSynchronize(static_cast<cudaStream_t>(stream)) != cudaSuccess) return MLMC_ERR_CUDA;
    for (int i = 0; i < K_COUNT; ++i) {
        total_ms[i] = 0.0;
        launches[i] = 0;
    }
    for (int i = 0; i < ws.timing_used; ++i) {
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, ws.ev_start[i], ws.ev_stop[i]) != cudaSuccess) return MLMC_ERR_CUDA;
        total_ms[ws.ev_id[i]] += ms;
        launches[ws.ev_id[i]]++;
    }
    ws.timing_used = 0;
    return MLMC_OK;
}

int mlmc_read_u(mlmc_ctx* ctx, uint64_t seed, uint64_t step, int M, double* u_host, void* stream) {
    if (!ctx || !u_host || M < 1 || M > ctx->ws.M_max) return MLMC_ERR_ARG;
    DeviceGuard guard(ctx->ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    launch_uniforms(ctx->ws, M, seed, step, s);
    if (cudaMemcpyAsync(u_host, ctx->ws.u_dev, sizeof(double) * M, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return MLMC_ERR_CUDA;
    return finish(cudaStreamSynchronize(s));
}

int mlmc_read_bracket_stats(mlmc_ctx* ctx, uint64_t* stats_host, void* stream) {
    if (!ctx || !stats_host) return MLMC_ERR_ARG;
    DeviceGuard guard(ctx->ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(stats_host, ctx->ws.bracket_stats, sizeof(uint64_t) * 3, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return MLMC_ERR_CUDA;
    return finish(cudaStreamSynchronize(s));
}

int mlmc_read_sample_stats(mlmc_ctx* ctx, uint64_t* stats_host, void* stream) {
    if (!ctx || !stats_host) return MLMC_ERR_ARG;
    DeviceGuard guard(ctx->ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (cudaMemcpyAsync(stats_host, ctx->ws.bracket_stats + 4, sizeof(uint64_t) * 3, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return MLMC_ERR_CUDA;
    return finish(cudaStreamSynchronize(s));
}

int mlmc_read_listed_tiles(mlmc_ctx* ctx, int M, uint32_t* listed_host, int64_t* tiles_host, void* stream) {
    if (!ctx || !listed_host || !tiles_host || M < 1 || M > ctx->ws.M_max) return MLMC_ERR_ARG;
    DeviceGuard guard(ctx->ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    *tiles_host = ctx->ws.last_emit_tiles * kEmitGroups;
    if (cudaMemcpyAsync(listed_host, ctx->ws.group_n, sizeof(uint32_t) * M, cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return MLMC_ERR_CUDA;
    return finish(cudaStreamSynchronize(s));
}

int mlmc_level_probs(mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, int kind,
                     const int64_t* sched, int L, const double* p_host, double* p_out, double* delta_out,
                     void* stream) {
    if (int rc = check_common(ctx, g, dtype, d, M, ld, L)) return rc;
    if (!p_out || (kind != MLMC_TOPK && kind != MLMC_BITWISE && kind != MLMC_RTN)) return MLMC_ERR_ARG;
    Workspace& ws = ctx->ws;
    double pn[kMaxLevels];
    int32_t b32[kMaxLevels];
    if (kind == MLMC_TOPK) {
        if (int rc = check_topk_schedule(sched, L, d)) return rc;
    } else if (kind == MLMC_BITWISE) {
        if (int rc = check_bit_schedule(sched, L, b32)) return rc;
    } else {
        if (int rc = check_rtn_schedule(sched, L, b32)) return rc;
    }
    if (p_host)
        if (int rc = normalise_probs(p_host, L, pn)) return rc;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
    const bool need_data = (p_host == nullptr) || (delta_out != nullptr);
    if (need_data) {
        if (kind == MLMC_TOPK) {
            select_adaptive(ws, g, dtype, d, M, ld, sched, L, 0, 0, nullptr, s);
        } else if (kind == MLMC_BITWISE) {
            const DrawPlan plan = bit_draw_plan(ws, b32, L, 0, 0, nullptr);
            launch_absmax(ws, g, dtype, d, M, ld, plan, nullptr, nullptr, s);
            launch_bit_stats(ws, g, dtype, d, M, ld, b32, L, plan, s);
        } else {
            const DrawPlan plan = rtn_draw_plan(ws, L, 0, 0, nullptr);
            launch_absmax(ws, g, dtype, d, M, ld, plan, nullptr, nullptr, s);
            launch_rtn_stats(ws, g, dtype, d, M, ld, b32, L, plan, s);
        }
    }
    launch_copy_probs(ws, M, L, p_host ? pn : nullptr, p_out, delta_out, s);
    return finish(cudaGetLastError());
}

int mlmc_compress_topk(mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, const int64_t* k,
                       int L, const double* p, uint64_t seed, uint64_t step, const mlmc_topk_msgs* out,
                       void* stream) {
    if (int rc = check_common(ctx, g, dtype, d, M, ld, L)) return rc;
    if (!out || !out->idx || !out->val || !out->count || !out->level || !out->p_sel || out->capacity < 0)
        return MLMC_ERR_ARG;
    if (int rc = check_topk_schedule(k, L, d)) return rc;
    double pn[kMaxLevels];
    if (p)
        if (int rc = normalise_probs(p, L, pn)) return rc;
    Workspace& ws = ctx->ws;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
    if (!p) {
        select_adaptive(ws, g, dtype, d, M, ld, k, L, seed, step, out, s);
    } else {
        // the bins stored by earlier calls belong to one problem: another shape or schedule starts afresh
        bool same = ws.sig_d == d && ws.sig_ld == ld && ws.sig_M == M && ws.sig_L == L && ws.sig_dtype == dtype;
        for (int l = 0; same && l < L; ++l) same = ws.sig_k[l] == k[l];
        if (!same) {
            cudaMemsetAsync(ws.prev_bin, 0xFF, sizeof(uint32_t) * kMaxLevels * ws.M_max, s);
            ws.sig_d = d; ws.sig_ld = ld; ws.sig_M = M; ws.sig_L = L; ws.sig_dtype = dtype;
            for (int l = 0; l < L; ++l) ws.sig_k[l] = k[l];
        }
        select_drawn(ws, g, dtype, d, M, ld, L, true, seed, step, out, [&](double u) {
            const int l = draw_from_probs(pn, L, u);
            return DrawnBand{pn[l], l, l ? (uint32_t)k[l - 1] : 0u, (uint32_t)k[l]};
        }, s);
    }
    return finish(cudaGetLastError());
}

int mlmc_compress_bitwise(mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* b,
                          int L, const double* p, uint64_t seed, uint64_t step, const mlmc_bit_msgs* out,
                          void* stream) {
    if (int rc = check_common(ctx, g, dtype, d, M, ld, L)) return rc;
    if (!out || !out->planes || !out->gmax || !out->level || !out->p_sel || out->w_max < 1) return MLMC_ERR_ARG;
    int32_t b32[kMaxLevels];
    if (int rc = check_bit_schedule(b, L, b32)) return rc;
    double pn[kMaxLevels];
    if (p)
        if (int rc = normalise_probs(p, L, pn)) return rc;
    Workspace& ws = ctx->ws;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
    const DrawPlan plan = bit_draw_plan(ws, b32, L, seed, step, out);
    if (launch_bit_cluster(ws, g, dtype, d, M, ld, b32, L, plan, p ? pn : nullptr, *out, s)) return finish(cudaGetLastError());
    launch_absmax(ws, g, dtype, d, M, ld, plan, p ? pn : nullptr, zero_batches(ws) ? out : nullptr, s);
    if (!p) launch_bit_stats(ws, g, dtype, d, M, ld, b32, L, plan, s);
    launch_bit_pack(ws, g, dtype, d, M, ld, b32, L, *out, s);
    return finish(cudaGetLastError());
}

int mlmc_aggregate(mlmc_ctx* ctx, int kind, const void* msgs, const int32_t* b, int L, int M, int64_t d, float* out,
                   void* stream) {
    if (!ctx || !msgs || !out) return MLMC_ERR_ARG;
    Workspace& ws = ctx->ws;
    if (d < 1 || d > ws.d_max || M < 1 || M > ws.M_max) return MLMC_ERR_ARG;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, 4);
    if (kind == MLMC_TOPK) {
        const mlmc_topk_msgs* t = static_cast<const mlmc_topk_msgs*>(msgs);
        if (!t->idx || !t->val || !t->count || !t->level) return MLMC_ERR_ARG;
        launch_aggregate_topk(ws, *t, M, d, out, s);
    } else if (kind == MLMC_BITWISE) {
        const mlmc_bit_msgs* t = static_cast<const mlmc_bit_msgs*>(msgs);
        if (!t->planes || !t->gmax || !t->level || !t->p_sel || L < 1 || L > kMaxLevels) return MLMC_ERR_ARG;
        int32_t b32[kMaxLevels];
        if (int rc = check_bit_schedule(b, L, b32)) return rc;
        launch_aggregate_bitwise(ws, *t, b32, L, M, d, out, s);
    } else {
        return MLMC_ERR_ARG;
    }
    return finish(cudaGetLastError());
}

int mlmc_compress_stopk(mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, int64_t s_len,
                        const double* p, uint64_t seed, uint64_t step, const mlmc_topk_msgs* out, void* stream) {
    if (!ctx || s_len < 1 || d < 1) return MLMC_ERR_ARG;
    const int64_t L = (d + s_len - 1) / s_len;
    if (L <= kMaxLevels) {  // few segments: the general Top-k path with the uniform schedule k_l = min(d, s (l + 1))
        int64_t k[kMaxLevels];
        for (int64_t l = 0; l < L; ++l) k[l] = (s_len * (l + 1) < d) ? s_len * (l + 1) : d;
        return mlmc_compress_topk(ctx, g, dtype, d, M, ld, k, (int)L, p, seed, step, out, stream);
    }
    if (int rc = check_common(ctx, g, dtype, d, M, ld, 1)) return rc;
    if (!out || !out->idx || !out->val || !out->count || !out->level || !out->p_sel || out->capacity < 0)
        return MLMC_ERR_ARG;
    Workspace& ws = ctx->ws;
    if (L > ws.big_cap) return MLMC_ERR_ARG;
    if (!p) {
        // Adaptive p with many segments: Lemma 3.4 needs the norm of every segment
        DeviceGuard guard(ws.device);
        cudaStream_t s = static_cast<cudaStream_t>(stream);
        if (int rc = reserve_segments(ws)) return rc;
        set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
        launch_begin_adaptive(ws, dtype, d, M, nullptr, 1, s);
        launch_hist1(ws, g, dtype, d, M, ld, false, nullptr, s);
        launch_segments(ws, g, dtype, d, M, ld, s_len, L, seed, step, s);
        launch_band_header(ws, M, finish_plan(d, 3, 2, false, seed, step, out), s);
        launch_emit(ws, g, dtype, d, M, ld, *out, s);
        return finish(cudaGetLastError());
    }
    double sum = 0.0;
    for (int64_t l = 0; l < L; ++l) {
        if (!(p[l] > 0.0) || !std::isfinite(p[l])) return MLMC_ERR_PROB;
        sum += p[l];
    }
    if (std::fabs(sum - 1.0) > 1e-9) return MLMC_ERR_PROB;
    // running sums of the normalised p in ascending l: the draw is min{ l : u < cdf_l }, the last cdf is 1
    std::vector<double> cdf((size_t)L);
    double c = 0.0;
    for (int64_t l = 0; l < L; ++l) cdf[(size_t)l] = (c += p[l] / sum);
    cdf[(size_t)L - 1] = 1.0;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
    select_drawn(ws, g, dtype, d, M, ld, 3, false, seed, step, out, [&](double u) {
        const int64_t l = std::upper_bound(cdf.begin(), cdf.end(), u) - cdf.begin();
        const int64_t hi = s_len * (l + 1);
        return DrawnBand{p[l] / sum, (int32_t)l, (uint32_t)(s_len * l), (uint32_t)(hi < d ? hi : d)};
    }, s);
    return finish(cudaGetLastError());
}

int mlmc_compress_floatbits(mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* mb,
                            int L, const double* p, uint64_t seed, uint64_t step, const mlmc_float_msgs* out,
                            void* stream) {
    if (int rc = check_common(ctx, g, dtype, d, M, ld, L)) return rc;
    if (!out || !out->expo || !out->planes || !out->level || !out->p_sel || out->w_max < 1) return MLMC_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(out->expo) % 16 != 0 || reinterpret_cast<uintptr_t>(out->planes) % 16 != 0)
        return MLMC_ERR_ARG;
    if (int rc = check_mantissa_schedule(mb, L, dtype == MLMC_BF16 ? 7 : 23)) return rc;
    double pn[kMaxLevels];
    if (p) {
        if (int rc = normalise_probs(p, L, pn)) return rc;
    } else {
        // App. B's lemma: p^l proportional to 2^-l for the unit schedule; for a general schedule its worst-case
        // argument gives p^l proportional to the largest residual of the level, 2^-mb_{l-1} - 2^-mb_l
        double sum = 0.0;
        for (int l = 0; l < L; ++l) {
            pn[l] = std::ldexp(1.0, -(l ? mb[l - 1] : 0)) - std::ldexp(1.0, -mb[l]);
            sum += pn[l];
        }
        for (int l = 0; l < L; ++l) pn[l] /= sum;
    }
    Workspace& ws = ctx->ws;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
    launch_compress_floatbits(ws, g, dtype, d, M, ld, mb, L, pn, seed, step, *out, s);
    return finish(cudaGetLastError());
}

int mlmc_aggregate_floatbits(mlmc_ctx* ctx, const mlmc_float_msgs* msgs, const int32_t* mb, int L, int M, int64_t d,
                             float* out, void* stream) {
    if (!ctx || !msgs || !out || !msgs->expo || !msgs->planes || !msgs->level || !msgs->p_sel) return MLMC_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(msgs->expo) % 16 != 0) return MLMC_ERR_ARG;  // read 16 bytes at a time
    Workspace& ws = ctx->ws;
    if (d < 1 || d > ws.d_max || M < 1 || M > ws.M_max || L < 1 || L > kMaxLevels) return MLMC_ERR_ARG;
    if (!mb) return MLMC_ERR_ARG;
    int prev = 0;
    for (int l = 0; l < L; ++l) {
        if (mb[l] <= prev || mb[l] > 23) return MLMC_ERR_SCHEDULE;
        prev = mb[l];
    }
    DeviceGuard guard(ws.device);
    set_call_size(ws, d, M, 4);
    launch_aggregate_floatbits(ws, *msgs, mb, L, M, d, out, static_cast<cudaStream_t>(stream));
    return finish(cudaGetLastError());
}

int mlmc_compress_rtn(mlmc_ctx* ctx, const void* g, int dtype, int64_t d, int M, int64_t ld, const int32_t* r, int L,
                      const double* p, uint64_t seed, uint64_t step, const mlmc_rtn_msgs* out, void* stream) {
    if (int rc = check_common(ctx, g, dtype, d, M, ld, L)) return rc;
    if (!out || !out->val || !out->c || !out->level || !out->p_sel || out->ldv < d) return MLMC_ERR_ARG;
    if (reinterpret_cast<uintptr_t>(out->val) % 16 != 0) return MLMC_ERR_ARG;
    int32_t r32[kMaxLevels] = {};
    if (int rc = check_rtn_schedule(r, L, r32)) return rc;
    double pn[kMaxLevels];
    if (p)
        if (int rc = normalise_probs(p, L, pn)) return rc;
    Workspace& ws = ctx->ws;
    DeviceGuard guard(ws.device);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    set_call_size(ws, d, M, dtype == MLMC_BF16 ? 2 : 4);
    const DrawPlan plan = rtn_draw_plan(ws, L, seed, step, out);
    if (launch_rtn_cluster(ws, g, dtype, d, M, ld, r32, L, plan, p ? pn : nullptr, *out, s)) return finish(cudaGetLastError());
    launch_absmax(ws, g, dtype, d, M, ld, plan, p ? pn : nullptr, nullptr, s);  // c = max |g|, and the NaN / Inf check
    if (!p) launch_rtn_stats(ws, g, dtype, d, M, ld, r32, L, plan, s);
    launch_rtn_emit(ws, g, dtype, d, M, ld, r32, L, *out, s);
    return finish(cudaGetLastError());
}

int mlmc_aggregate_rtn(mlmc_ctx* ctx, const mlmc_rtn_msgs* msgs, int M, int64_t d, float* out, void* stream) {
    if (!ctx || !msgs || !out || !msgs->val || !msgs->level || msgs->ldv < d) return MLMC_ERR_ARG;
    Workspace& ws = ctx->ws;
    if (d < 1 || d > ws.d_max || M < 1 || M > ws.M_max) return MLMC_ERR_ARG;
    DeviceGuard guard(ws.device);
    set_call_size(ws, d, M, 4);
    launch_aggregate_dense(ws, msgs->val, msgs->level, M, d, msgs->ldv, out, static_cast<cudaStream_t>(stream));
    return finish(cudaGetLastError());
}

}  // extern "C"
