"""The lengths at which the library changes its kernels, and the edges of their tiles, against the CPU oracle.

Every case runs compress and aggregate through the C ABI and compares messages and averages (the checks of the parity tests).
"""
import numpy as np
import pytest
import torch

from paper_2507_05508_b200 import workloads as wl
from test_gpu_ext import check_floatbits, check_rtn
from test_gpu_parity import check_bitwise, check_topk, padded, to_dev

pytestmark = pytest.mark.gpu

BITS = [1, 2, 4, 8, 16, 23]


@pytest.fixture(scope="module")
def B():
    from paper_2507_05508_b200 import binding
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.mlmc_create(0, 2_500_000, 20, 32)
    yield c
    B.mlmc_destroy(c)


def layered(d, M, dtype="f32", seed=5):
    """Heavy-tailed rows with a few layers of different scale."""
    rng = np.random.default_rng(seed)
    scale = np.repeat(10.0 ** rng.uniform(-4, -1, 7), -(-d // 7))[:d]
    g = torch.from_numpy((rng.standard_t(3, (M, d)) * scale).astype(np.float32)).cuda()
    return padded(g.to(torch.bfloat16) if dtype == "bf16" else g, 8)


def geometric(L):
    return list(wl.geometric_probs(L))


def doubling(d, first):
    k = []
    while first < d:
        k.append(first)
        first *= 2
    return k + [d]


# one block or two; the longest row of a cluster with given p and with adaptive p, fp32 and bf16; one entry more
@pytest.mark.parametrize("dtype,d,M,adaptive", [
    ("f32", 511, 2, True), ("f32", 16_384, 3, True), ("f32", 16_385, 3, True), ("f32", 262_144, 2, False), ("f32", 262_145, 2, False),
    ("f32", 704_512, 1, True), ("f32", 704_513, 1, True), ("bf16", 32_769, 2, True), ("bf16", 524_289, 1, False),
    ("bf16", 1_032_192, 1, True), ("bf16", 1_032_193, 1, True)])
def test_topk_row_lengths(B, ora, ctx, dtype, d, M, adaptive):
    k = doubling(d, max(1, d // 500))
    check_topk(B, ora, ctx, layered(d, M, dtype), k, None if adaptive else geometric(len(k)), 3, 1, expect_excluded=1)


# the average in one launch (up to four tiles per SM) and in two
@pytest.mark.parametrize("d,M", [(4_096, 20), (4_097, 1), (2_424_832, 2), (2_424_833, 2)])
def test_topk_average_lengths(B, ora, ctx, d, M):
    k = [d // 3, d]
    check_topk(B, ora, ctx, layered(d, M), k, [0.5, 0.5], 1, 2)


# bands from a few entries per batch of 512 words to whole batches, on both sides of the staged emission, with and without ties
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("share", [0.02, 0.12, 0.125, 0.5, 1.0])
def test_dense_and_sparse_bands(B, ora, ctx, dtype, share):
    d = 530_001
    lo = int(d * (1 - share) / 2)
    k = [lo, lo + max(1, int(d * share)), d] if share < 1.0 else [0, d]
    p = [1e-9] * len(k)
    p[1] = 1.0 - 1e-9 * (len(k) - 1)
    g = layered(d, 2, dtype)
    check_topk(B, ora, ctx, g, k, p, 4, 0)
    rng = np.random.default_rng(8)
    ties = torch.from_numpy(rng.choice(np.array([0.5, -0.5, 0.25, 3.0, 0.1], dtype=np.float32), (2, d))).cuda()
    check_topk(B, ora, ctx, padded(ties.to(g.dtype), 8), k, p, 4, 1)


# thresholds that share a leading-digit bin, trivial ranks, and so many levels that the second sweep takes smaller blocks
@pytest.mark.parametrize("case", ["shared_bins", "trivial_ranks", "many_levels"])
def test_second_sweep_intervals(B, ora, ctx, case):
    d = 720_003
    if case == "shared_bins":
        g = to_dev((1.0 + 0.02 * np.random.default_rng(1).random((1, d))).astype(np.float32))
        k = [int(d * f) for f in (0.1, 0.2, 0.21, 0.5, 0.9, 0.99)] + [d]
    elif case == "trivial_ranks":
        g, k = layered(d, 1), [0, 0, 7, 7, d // 2, d, d]
    else:
        g, k = layered(d, 1), sorted({int(d * (i + 1) / 32) for i in range(31)}) + [d]
    check_topk(B, ora, ctx, g, k, None, 2, 3, expect_excluded=1)


# a group of 1024 entries, a group per warp, the longest row of a cluster, and one entry more
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d,M", [(1, 1), (1_023, 3), (1_025, 20), (16_384, 2), (16_385, 2), (458_752, 1), (458_753, 1)])
def test_dense_row_lengths(B, ora, ctx, dtype, d, M):
    g = layered(d, M, dtype)
    for p in (None, geometric(6)):
        check_bitwise(B, ora, ctx, g, BITS, p, 7, 1)
    for p in (None, geometric(5)):
        check_rtn(B, ora, ctx, g, [2, 4, 8, 16], p, 7, 1)


# schedules outside the one-launch kernels: a field above 8 bits, more levels
@pytest.mark.parametrize("b", [[9, 23], [2, 9, 12, 20], list(range(1, 11)), [3, 11, 19]])
def test_bitwise_schedules_of_a_short_row(B, ora, ctx, b):
    g = layered(5_003, 3)
    check_bitwise(B, ora, ctx, g, b, None, 9, 0)
    check_bitwise(B, ora, ctx, g, b, geometric(len(b)), 9, 0)


# the divisor of the bit-wise quotient at both ends of fp32 and around the limits between which it is used as it is
@pytest.mark.parametrize("top", [2.0 ** -100, 0.999 * 2.0 ** -60, 2.0 ** -60, 1.0, 2.0 ** 100, 1.001 * 2.0 ** 100, 3.4e38])
@pytest.mark.parametrize("d", [4_001, 460_001])
def test_bitwise_scales(B, ora, ctx, top, d):
    rng = np.random.default_rng(2)
    g = rng.uniform(-1, 1, (1, d)) * np.exp(-rng.uniform(0, 12, (1, d)))
    g[0, 0] = 1.0
    g = to_dev((g * top).astype(np.float32))
    check_bitwise(B, ora, ctx, g, BITS, None, 1, 0)
    check_bitwise(B, ora, ctx, g, [23], [1.0], 1, 0)


# planes one by one and by bit transposes, ragged words, groups of zeros
@pytest.mark.parametrize("mb", [[1, 2, 4, 8, 16, 23], [5, 11, 23], [23]])
@pytest.mark.parametrize("d", [31, 33, 1_024, 70_001])
def test_floatbits_lengths(B, ora, ctx, mb, d):
    g = layered(d, 2)
    g[:, d // 3:d // 2] = 0.0
    check_floatbits(B, ora, ctx, g, mb, geometric(len(mb)), 6, 0)


# statistics of long rows: trips of the ring and what is left of them, few and many levels
@pytest.mark.parametrize("r", [[2, 4, 8, 16], list(range(1, 17))])
@pytest.mark.parametrize("d", [460_800, 460_801, 1_000_003])
def test_rtn_long_rows(B, ora, ctx, r, d):
    check_rtn(B, ora, ctx, layered(d, 1), r, None, 3, 0)


# buffers that start at any element: the averages take vectors only where the addresses allow it
@pytest.mark.parametrize("d", [8_192, 2_424_836])
def test_averages_into_unaligned_buffers(B, ctx, d):
    M, k = 2, [d // 50, d]
    g = layered(d, M)
    plain = torch.empty(d, dtype=torch.float32, device="cuda")
    shifted = torch.full((d + 8,), float("nan"), dtype=torch.float32, device="cuda")
    for off in (1, 2, 3):
        msgs = B.TopkBuffers(M, d)
        B.mlmc_compress_topk(ctx, g, k, [0.5, 0.5], 3, off, msgs)
        for average in (lambda out: B.mlmc_aggregate(ctx, B.MLMC_TOPK, msgs, None, M, d, out),
                        lambda out: B.mlmc_aggregate_topk_noalloc(msgs, M, d, out)):
            average(plain)
            average(shifted[off:off + d])
            assert torch.equal(plain, shifted[off:off + d])
        rtn, moved = B.RtnBuffers(M, d), B.RtnBuffers(M, d)
        B.mlmc_compress_rtn(ctx, g, [2, 4], [0.3, 0.3, 0.4], 3, off, rtn)
        room = torch.zeros(M * rtn.ldv + 8, dtype=torch.float32, device="cuda")
        val = room[off:off + M * rtn.ldv]
        val.copy_(rtn.val.flatten())
        moved.level.copy_(rtn.level)
        moved.struct.val = val.data_ptr()
        B.mlmc_aggregate_rtn(ctx, rtn, M, d, plain)
        for msg in (rtn, moved):
            for out in (torch.empty(d, dtype=torch.float32, device="cuda"), shifted[off:off + d]):
                B.mlmc_aggregate_rtn(ctx, msg, M, d, out)
                assert torch.equal(plain, out)
    assert B.mlmc_get_status(ctx) == B.MLMC_OK
    floats = B.FloatBuffers(M, d, 23)
    floats.struct.expo += 4
    with pytest.raises(B.MlmcError) as e:
        B.mlmc_aggregate_floatbits(ctx, floats, [23], M, d, plain)
    assert e.value.code == B.MLMC_ERR_ARG


# p_l = Delta_l / sum Delta and the running sums of the draw go over the levels in ascending order, on every path: the results
# follow bit for bit from the norms
@pytest.mark.parametrize("kind,d,M", [("topk", 9_001, 16), ("topk", 9_001, 40), ("topk", 1_100_001, 12), ("bitwise", 9_001, 16),
                                      ("bitwise", 500_001, 12), ("rtn", 9_001, 16), ("rtn", 500_001, 12)])
def test_probabilities_and_draw_follow_from_the_norms(B, kind, d, M):
    g = layered(d, M)
    sched = {"topk": doubling(d, 1 + d // 3000)[:30], "bitwise": BITS, "rtn": [2, 4, 8, 16]}[kind]
    if kind == "topk":
        sched[-1] = d
    L = len(sched) + (kind == "rtn")
    # the norms of both calls are exact integer sums but for RTN, where a short row's message and its norms by themselves come
    # from different kernels: d additions in fp64, in another order
    tol = d * 2.0 ** -53 if kind == "rtn" else 0.0
    c = B.mlmc_create(0, d, M, 32)
    try:
        p_out = torch.zeros((M, L), dtype=torch.float64, device="cuda")
        delta = torch.zeros((M, L), dtype=torch.float64, device="cuda")
        code = {"topk": B.MLMC_TOPK, "bitwise": B.MLMC_BITWISE, "rtn": B.MLMC_RTN}[kind]
        B.mlmc_level_probs(c, g, code, sched, None, p_out, delta)
        p_out, delta = p_out.cpu().numpy(), delta.cpu().numpy()
        for m in range(M):
            total = 0.0
            for x in delta[m].tolist():
                total += x
            assert (p_out[m] == delta[m] / total).all()
        for step in range(6):
            u = B.mlmc_read_u(c, 5, step, M)
            if kind == "topk":
                out = B.TopkBuffers(M, wl.max_band(sched))
                B.mlmc_compress_topk(c, g, sched, None, 5, step, out)
            elif kind == "bitwise":
                out = B.BitBuffers(M, d, 8)
                B.mlmc_compress_bitwise(c, g, sched, None, 5, step, out)
            else:
                out = B.RtnBuffers(M, d)
                B.mlmc_compress_rtn(c, g, sched, None, 5, step, out)
            assert B.mlmc_get_status(c) == B.MLMC_OK
            levels, p_sel = out.level.tolist(), out.p_sel.tolist()
            for m in range(M):
                cdf, last = 0.0, max(l for l in range(L) if p_out[m, l] > 0)
                for l in range(L):
                    cdf += p_out[m, l]
                    if u[m] < cdf or l == last:
                        break
                assert levels[m] == l and abs(p_sel[m] - p_out[m, l]) <= tol * p_out[m, l]
    finally:
        B.mlmc_destroy(c)


RESET = """
import ctypes, sys
import numpy as np
sys.path.insert(0, sys.argv[1])
from paper_2507_05508_b200 import binding as B
import oracle
rt = ctypes.CDLL("libcudart.so.12")
vp, sz = ctypes.c_void_p, ctypes.c_size_t
rt.cudaMalloc.argtypes, rt.cudaMemcpy.argtypes = [vp, sz], [vp, vp, sz, ctypes.c_int]
M, d, k = 2, 40_000, [100, 5000, 40_000]
g = np.random.default_rng(1).standard_normal((M, d)).astype(np.float32)

def device(n):
    p = vp()
    assert rt.cudaMalloc(ctypes.byref(p), n) == 0
    return p.value

for step in range(2):                      # the second round runs in a new CUDA context of the same process
    ctx = B.mlmc_create(0, d, M, 32)
    at = device(g.nbytes)
    assert rt.cudaMemcpy(at, g.ctypes.data, g.nbytes, 1) == 0
    fields = [device(M * d * 4), device(M * d * 4), device(M * 8), device(M * 4), device(M * 8)]
    msgs = B.mlmc_topk_msgs(*fields, d)
    sched = (ctypes.c_int64 * 3)(*k)
    assert B.lib().mlmc_compress_topk(ctx, at, B.MLMC_F32, d, M, d, sched, 3, None, 1, step, ctypes.byref(msgs), None) == 0
    assert B.lib().mlmc_get_status(ctx, None) == 0
    level = np.zeros(M, np.int32)
    idx = np.zeros((M, d), np.uint32)
    assert rt.cudaMemcpy(level.ctypes.data, fields[3], level.nbytes, 2) == 0
    assert rt.cudaMemcpy(idx.ctypes.data, fields[0], idx.nbytes, 2) == 0
    for m in range(M):
        o = oracle.topk(g[m], k, p=None, seed=1, step=step, worker=m)
        assert level[m] == o.level and np.array_equal(idx[m, :o.idx.size], o.idx)
    B.mlmc_destroy(ctx)
    assert rt.cudaDeviceReset() == 0
print("both contexts agree with the oracle")
"""


def test_create_after_a_device_reset(ora):
    """Kernel attributes belong to the CUDA context: a context created after cudaDeviceReset (which ends the process's own
    context only) works as the first one did."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET, root], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "both contexts agree" in r.stdout, r.stdout + r.stderr


# what a cluster holds and one entry more; as many workers as fit the GPU at a time in one, two and three waves
@pytest.mark.parametrize("dtype,d,M,adaptive", [
    ("f32", 745_472, 1, True), ("f32", 745_473, 1, True), ("bf16", 524_288, 1, True), ("bf16", 524_289, 1, True), ("bf16", 65_536, 20, True),
    ("f32", 131_072, 14, True), ("f32", 131_072, 20, True), ("f32", 262_144, 7, True), ("f32", 262_144, 13, False), ("f32", 262_144, 20, False)])
def test_topk_cluster_waves(B, ora, ctx, dtype, d, M, adaptive):
    k = doubling(d, max(1, d // 500))
    check_topk(B, ora, ctx, layered(d, M, dtype), k, None if adaptive else geometric(len(k)), 3, 1, expect_excluded=1)
