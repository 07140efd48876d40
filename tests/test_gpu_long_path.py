"""The kernels of long rows on the inputs where a selection can go wrong.

Short rows of up to 32 workers (Top-k) or as many as the GPU has SMs (bit-wise, RTN) take one-launch kernels, so the edge cases of
the parity tests, which are short, run there.  Here the same cases have one worker more than those kernels take, and run
through the histogram sweep, the second sweep, the digit passes and the tile list, or through the separate statistics and
message kernels.
"""
import numpy as np
import pytest
import torch

from paper_2507_05508_b200 import workloads as wl
from test_gpu_ext import check_rtn, check_stopk
from test_gpu_parity import check_bitwise, check_topk, padded, to_dev

pytestmark = pytest.mark.gpu

TOPK_M = 33          # one more than the Top-k cluster kernel takes
DENSE_M = 260        # more one-block clusters than there are SMs


@pytest.fixture(scope="module")
def B():
    from paper_2507_05508_b200 import binding
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.mlmc_create(0, 170_000, DENSE_M, 32)
    yield c
    B.mlmc_destroy(c)


def rows(g_np, M=TOPK_M):
    """M rows from a few, each at another offset."""
    return np.stack([np.roll(g_np[i % len(g_np)], 17 * i) for i in range(M)])


def launched(B, ctx, call):
    """The kernels of one call."""
    B.mlmc_timing_enable(ctx, True)
    call()
    names = set(B.mlmc_timing_read(ctx))
    B.mlmc_timing_enable(ctx, False)
    return names


def test_these_workers_take_the_long_path(B, ctx):
    g = to_dev(np.random.default_rng(1).standard_normal((DENSE_M, 3000)).astype(np.float32))
    out = B.TopkBuffers(TOPK_M, 3000)
    for p in (None, [0.5, 0.5]):
        names = launched(B, ctx, lambda: B.mlmc_compress_topk(ctx, g[:TOPK_M], [100, 3000], p, 0, 0, out))
        assert {"hist1", "sums_candidates", "cand_pass3", "tile_list", "emit"} <= names and "cluster_topk" not in names
        names = launched(B, ctx, lambda: B.mlmc_compress_topk(ctx, g[:TOPK_M - 1], [100, 3000], p, 0, 0, out))
        assert names == {"cluster_topk"}
    bits, rtn = B.BitBuffers(DENSE_M, 3000, 4), B.RtnBuffers(DENSE_M, 3000)
    assert launched(B, ctx, lambda: B.mlmc_compress_bitwise(ctx, g, [1, 2, 4, 8], None, 0, 0, bits)) == {"absmax", "bit_stats", "bit_pack"}
    assert launched(B, ctx, lambda: B.mlmc_compress_rtn(ctx, g, [2, 4], None, 0, 0, rtn)) == {"absmax", "rtn_stats", "rtn_emit"}
    assert launched(B, ctx, lambda: B.mlmc_compress_bitwise(ctx, g[:8], [1, 2, 4, 8], None, 0, 0, bits)) == {"cluster_bitwise"}
    assert launched(B, ctx, lambda: B.mlmc_compress_rtn(ctx, g[:8], [2, 4], None, 0, 0, rtn)) == {"cluster_rtn"}


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("case", ["all_equal", "all_zero", "ties", "outlier", "signed_zero_denormal", "tiny_d"])
def test_topk_degenerate_inputs(B, ora, ctx, case, dtype):
    rng = np.random.default_rng(22)
    d = 10_003
    k = [1, 10, 100, 100, 5000, d]
    if case == "all_equal":
        g_np = np.full((1, d), -0.75, dtype=np.float32)
    elif case == "all_zero":
        g_np = np.zeros((1, d), dtype=np.float32)
    elif case == "ties":
        g_np = rng.integers(-4, 5, (3, d)).astype(np.float32)
    elif case == "outlier":
        g_np = rng.standard_normal((2, d)).astype(np.float32) * 1e-6
        g_np[0, 777] = 3e30
        g_np[1, d - 1] = -3e30
    elif case == "signed_zero_denormal":
        g_np = rng.choice(np.array([0.0, -0.0, 1e-45, -1e-45, 1e-39, 1.0], dtype=np.float32), (3, d))
    else:
        g_np, k = rng.standard_normal((4, 5)).astype(np.float32), [1, 3, 5]
    g = to_dev(rows(g_np))
    if dtype == "bf16":
        g = padded(g.to(torch.bfloat16), 8)
    for step in range(2):
        check_topk(B, ora, ctx, g, k, None, 9, step, expect_excluded=2)
        check_topk(B, ora, ctx, g, k, list(wl.geometric_probs(len(k))), 9, step)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_topk_every_level_is_reachable(B, ora, ctx, dtype):
    rng = np.random.default_rng(21)
    d = 20_001
    g_np = (rng.standard_normal((2, d)) * 10.0 ** rng.uniform(-3, 0, (2, d))).astype(np.float32)
    g_np[:, ::5] = np.round(g_np[:, ::5], 2)             # ties
    g = to_dev(rows(g_np))
    if dtype == "bf16":
        g = padded(g.to(torch.bfloat16), 8)
    k = [1, 2, 50, 50, 1000, 1001, 12_000, 20_000, d]
    for l in range(len(k)):
        p = np.full(len(k), 1e-6)
        p[l] = 1.0 - 1e-6 * (len(k) - 1)
        check_topk(B, ora, ctx, g, k, list(p), 1, l)
    check_topk(B, ora, ctx, g, k, None, 1, 0, expect_excluded=2)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_level_probs(B, ora, ctx, dtype):
    w = wl.shrink(wl.C5A, 30_011, TOPK_M)
    k = wl.topk_schedule(w)
    g = padded(wl.gradients(w, 2, "cuda"), 8)
    if dtype == "bf16":
        g = padded(g.to(torch.bfloat16), 8)
    gh = wl.as_numpy_bits(g)
    p_out = torch.zeros((TOPK_M, len(k)), dtype=torch.float64, device="cuda")
    d_out = torch.zeros_like(p_out)
    for p in (None, list(wl.geometric_probs(len(k)))):
        B.mlmc_level_probs(ctx, g, B.MLMC_TOPK, k, p, p_out, d_out)
        assert B.mlmc_get_status(ctx) == B.MLMC_OK
        for m in range(TOPK_M):
            o = ora.topk(gh[m], k, None)
            assert np.allclose(p_out[m].cpu().numpy(), o.p if p is None else p, rtol=1e-11, atol=1e-15)
            assert np.allclose(d_out[m].cpu().numpy(), o.delta, rtol=1e-12, atol=0)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_topk_device_errors(B, ctx, dtype):
    """A message that does not fit, and a NaN: the other workers' messages are what they are without them."""
    g = to_dev(np.random.default_rng(24).standard_normal((TOPK_M, 5000)).astype(np.float32))
    if dtype == "bf16":
        g = padded(g.to(torch.bfloat16), 8)
    k, p = [10, 100, 5000], [0.2, 0.3, 0.5]
    for probs in (p, None):
        full, small = B.TopkBuffers(TOPK_M, 4900), B.TopkBuffers(TOPK_M, 50)
        B.mlmc_compress_topk(ctx, g, k, probs, 3, 0, full)
        assert B.mlmc_get_status(ctx) == B.MLMC_OK
        B.mlmc_compress_topk(ctx, g, k, probs, 3, 0, small)
        assert B.mlmc_get_status(ctx) == B.MLMC_ERR_CAPACITY
        assert B.mlmc_get_status(ctx) == B.MLMC_OK
        bad = g.clone()
        bad[5, 4321], bad[32, 0] = float("nan"), float("-inf")
        void = B.TopkBuffers(TOPK_M, 4900)
        B.mlmc_compress_topk(ctx, padded(bad, 8), k, probs, 3, 0, void)
        assert B.mlmc_get_status(ctx) == B.MLMC_ERR_NONFINITE
        for m in range(TOPK_M):
            n = int(full.count[m])
            assert [int(small.level[m]), int(small.count[m])] == ([int(full.level[m]), n] if n <= 50 else [-1, 0])
            if n <= 50:
                assert torch.equal(small.idx[m, :n], full.idx[m, :n]) and torch.equal(small.val[m, :n], full.val[m, :n])
            if m in (5, 32):
                assert int(void.level[m]) == -1 and int(void.count[m]) == 0
            else:
                assert int(void.level[m]) == int(full.level[m]) and torch.equal(void.idx[m, :n], full.idx[m, :n])


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_emission_reads_only_batches_that_can_hold_band_entries(B, ctx, dtype):
    per_word = 2 if dtype == "bf16" else 1
    batch = 512 * per_word
    tile = 8 * batch
    d = (20 if dtype == "f32" else 15) * tile + 123
    rng = np.random.default_rng(5)
    g_np = (rng.standard_normal((TOPK_M, d)) * 1e-3).astype(np.float32)
    g_np[:, 7 * tile:9 * tile] *= 1e3                       # one loud layer: tiles 7 and 8
    g = to_dev(g_np)
    if dtype == "bf16":
        g = padded(g.to(torch.bfloat16), 8)
    k = [64, 1024, d]
    out = B.TopkBuffers(TOPK_M, d)
    for step, p in ((0, [0.98, 0.01, 0.01]), (1, [0.01, 0.98, 0.01]), (2, [0.005, 0.005, 0.99])):
        B.mlmc_compress_topk(ctx, g, k, p, 11, step, out)
        assert B.mlmc_get_status(ctx) == B.MLMC_OK
        listed, batches = B.mlmc_read_listed_tiles(ctx, TOPK_M)
        assert batches == (d + tile - 1) // tile * 8
        for m in range(TOPK_M):
            n, lv = int(out.count[m]), int(out.level[m])
            touched = torch.unique((out.idx[m, :n].to(torch.int64) & 0xFFFFFFFF) // batch).numel()
            assert touched <= listed[m] <= batches
            assert listed[m] == batches if lv == 2 else listed[m] <= 16


def test_stopk_few_segments_and_given_p(B, ora, ctx):
    rng = np.random.default_rng(31)
    d = 10_007
    g_np = (rng.standard_normal((2, d)) * 10.0 ** rng.uniform(-3, 0, (2, d))).astype(np.float32)
    g_np[1, ::3] = 0.0
    g = to_dev(rows(g_np))
    check_stopk(B, ora, ctx, g, 1000, None, 4, 0, expect_excluded=2)
    for s in (1000, 100):
        L = -(-d // s)
        check_stopk(B, ora, ctx, g, s, [1.0 / L] * L, 4, s)


# bit-wise and RTN: degenerate rows, and rows with a NaN or an Inf among others
def test_dense_degenerate_and_void_rows(B, ora, ctx):
    rng = np.random.default_rng(41)
    d = 1_100
    some = (rng.standard_t(3, (5, d)) * 1e-2).astype(np.float32)
    some[0] = 0.0
    some[1] = 0.0
    some[1, 17] = -1e-40                                     # denormal maximum
    some[2, 999] = 3e30                                      # (a message value 3e38 / p is beyond fp32)
    some[3, ::2] = np.abs(some[3, 1]) * rng.choice([-1.0, 1.0], d // 2)
    g_np = rows(some, DENSE_M)
    g = to_dev(g_np)
    for p in (None, list(wl.geometric_probs(4))):
        check_bitwise(B, ora, ctx, g, [1, 2, 4, 8], p, 5, 0)
        check_rtn(B, ora, ctx, to_dev(rows(some[[0, 3, 4]], DENSE_M)), [2, 4, 8], p, 5, 0)
    bad = g_np.copy()
    bad[7, 1000], bad[259, 0] = np.nan, -np.inf
    for p in (None, list(wl.geometric_probs(4))):
        clean, void = B.BitBuffers(DENSE_M, d, 4), B.BitBuffers(DENSE_M, d, 4)
        B.mlmc_compress_bitwise(ctx, g, [1, 2, 4, 8], p, 5, 1, clean)
        assert B.mlmc_get_status(ctx) == B.MLMC_OK
        B.mlmc_compress_bitwise(ctx, to_dev(bad), [1, 2, 4, 8], p, 5, 1, void)
        assert B.mlmc_get_status(ctx) == B.MLMC_ERR_NONFINITE
        dense = torch.full((d,), float("nan"), dtype=torch.float32, device="cuda")
        B.mlmc_aggregate(ctx, B.MLMC_BITWISE, void, [1, 2, 4, 8], DENSE_M, d, dense)
        assert torch.isfinite(dense).all()                   # void messages add nothing
        r_clean, r_void = B.RtnBuffers(DENSE_M, d), B.RtnBuffers(DENSE_M, d)
        B.mlmc_compress_rtn(ctx, g, [2, 4, 8], p, 5, 1, r_clean)
        assert B.mlmc_get_status(ctx) == B.MLMC_OK
        B.mlmc_compress_rtn(ctx, to_dev(bad), [2, 4, 8], p, 5, 1, r_void)
        assert B.mlmc_get_status(ctx) == B.MLMC_ERR_NONFINITE
        good = [m for m in range(DENSE_M) if m not in (7, 259)]
        for x, y in ((clean, void), (r_clean, r_void)):
            assert y.level[[7, 259]].tolist() == [-1, -1]
            assert torch.equal(x.level[good], y.level[good]) and torch.equal(x.p_sel[good], y.p_sel[good])
        widths = [1, 1, 2, 4]
        for m in good:
            n = 1 + widths[int(clean.level[m])]
            assert torch.equal(clean.planes[m, :n], void.planes[m, :n])
        assert torch.equal(r_clean.val[good], r_void.val[good])


def test_codes_are_those_of_the_division(B):
    """The 23-bit code of every entry against the IEEE division, for 10^7 pairs with divisors over the whole fp32 range: the
    library forms the quotient from the divisor's reciprocal by two corrections."""
    M, d = 20, 500_000
    c = B.mlmc_create(0, d, M, 32)
    rng = np.random.default_rng(7)
    try:
        out = B.BitBuffers(M, d, 23)
        # entries: a uniform share of the divisor, or the divisor over a power of two, with the last bits changed
        top = np.ldexp(rng.uniform(1.0, 2.0, M), np.linspace(-140, 126, M).astype(int)).astype(np.float32)
        share = rng.random((M, d))
        share[:, ::2] = np.exp2(-rng.integers(0, 24, (M, d // 2)).astype(np.float64))
        bits = (share * top[:, None].astype(np.float64)).astype(np.float32).view(np.int32) + rng.integers(-2, 3, (M, d), dtype=np.int32)
        g = np.minimum(np.maximum(bits, 0).view(np.float32), top[:, None])
        g[:, 0] = top
        B.mlmc_compress_bitwise(c, to_dev(g), [23], [1.0], 0, 0, out)
        assert B.mlmc_get_status(c) == B.MLMC_OK
        assert np.array_equal(out.gmax.cpu().numpy(), top)
        planes = out.planes.cpu().numpy().view(np.uint8)
        for m in range(M):
            e = g[m] / top[m]                                # fp32 by IEEE rules
            q = np.minimum(np.floor(np.ldexp(e.astype(np.float64), 23)), 2.0 ** 23 - 1).astype(np.uint32)
            code = np.zeros(out.words * 32, dtype=np.uint32)
            for j in range(1, 24):
                code = (code << np.uint32(1)) | np.unpackbits(planes[m, j], bitorder="little")
            assert np.array_equal(code[:d], q), f"divisor {top[m]}"
    finally:
        B.mlmc_destroy(c)
