"""Adaptive Top-k of long fp32 rows: brackets from a sample of the row, and messages that skip batches which round to 0."""
import numpy as np
import pytest
import torch

from test_gpu_ext import check_rtn
from test_gpu_parity import check_bitwise, padded, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_05508_b200 import binding
    binding.lib()
    return binding


def sampled_entries(d):
    """Mask of the entries that a sample by clusters of 1, 2, .. 16 blocks reads: sectors of eight, one per stratum."""
    mask = np.zeros(d, dtype=bool)
    sectors = d // 8
    for blocks in (1, 2, 4, 8, 16):
        strata = 8192 * blocks
        i = np.arange(strata, dtype=np.uint64)
        first, end = i * np.uint64(sectors) // np.uint64(strata), (i + np.uint64(1)) * np.uint64(sectors) // np.uint64(strata)
        h = (i * np.uint64(0x9E3779B1)) & np.uint64(0xFFFFFFFF)
        at = first + (h * (end - first) >> np.uint64(32))
        mask[(at[:, None] * np.uint64(8) + np.arange(8, dtype=np.uint64)).astype(np.int64).ravel()] = True
    return mask


def rows(case, M, d, seed=71):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g = padded(torch.randn((M, d), generator=gen, device="cuda"), 4)
    if case == "layers":
        g *= torch.repeat_interleave(10.0 ** (torch.rand(40, generator=gen, device="cuda") * 4 - 5), -(-d // 40))[:d]
    elif case == "ties":
        g.mul_(2.0).round_()
    elif case == "zeros":
        g *= torch.rand(d, generator=gen, device="cuda") < 0.03
    elif case == "unseen":            # the sample sees nothing but zeros: more than there is room for
        g[:, torch.from_numpy(sampled_entries(d)).cuda()] = 0.0
    elif case == "misled":            # the sample sees entries of another scale: every row has a bracket that misses
        g[:, torch.from_numpy(sampled_entries(d)).cuda()] *= 1000.0
    elif case == "constant":
        g.fill_(0.25)
    return g


def check_adaptive(B, ctx, g, k):
    """Norms, probabilities, levels and bands of some workers against a stable sort of their rows on the device."""
    M = g.shape[0]
    out = B.TopkBuffers(M, max(b - a for a, b in zip([0] + k[:-1], k)))
    p = torch.zeros((M, len(k)), dtype=torch.float64, device="cuda")
    delta = torch.zeros_like(p)
    B.mlmc_level_probs(ctx, g, B.MLMC_TOPK, k, None, p, delta)
    B.mlmc_compress_topk(ctx, g, k, None, 5, 1, out)
    assert B.mlmc_get_status(ctx) == B.MLMC_OK
    u = B.mlmc_read_u(ctx, 5, 1, M)
    for m in sorted({0, 1, M // 2, M - 1}):
        order = torch.sort(g[m].abs(), descending=True, stable=True).indices
        sq = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), g[m].double()[order].square()])
        norms = torch.stack([sq[a + 1:b + 1].sum() for a, b in zip([0] + k[:-1], k)]).sqrt()
        assert torch.allclose(delta[m], norms, rtol=1e-9, atol=0.0)
        want = norms / norms.sum() if norms.sum() > 0 else torch.eye(len(k), dtype=torch.float64, device="cuda")[0]
        assert torch.allclose(p[m], want, rtol=1e-9, atol=1e-15)
        level = int(out.level[m])
        cdf = torch.cumsum(p[m], 0).tolist()
        assert p[m, level] > 0 and (level == 0 or u[m] >= cdf[level - 1] - 1e-9) and u[m] < cdf[level] + 1e-9
        band = torch.sort(order[(k[level - 1] if level else 0):k[level]]).values
        n = int(out.count[m])
        assert n == band.numel() and torch.equal(out.idx[m, :n].long() & 0xFFFFFFFF, band)
        value = g[m][band].double() / float(out.p_sel[m])
        # a product below the normal range is rounded to a multiple of 2^-149: by half of that at most
        assert torch.allclose(out.val[m, :n].double(), value, rtol=1e-6, atol=2.0 ** -150)


HELD, MISSED, LEFT_OUT = range(3)


def check_sampled(B, ctx, g, k, want):
    """check_adaptive, and what became of the workers' brackets: `want` of HELD, MISSED, LEFT_OUT per worker; empty: two sweeps."""
    before = B.mlmc_read_sample_stats(ctx)
    check_adaptive(B, ctx, g, k)      # two selections
    seen = [b - a for a, b in zip(before, B.mlmc_read_sample_stats(ctx))]
    assert seen == [2 * sum(w == i for w in want) for i in range(3)], (seen, k)


@pytest.mark.parametrize("case", ["layers", "normal", "ties", "zeros", "unseen", "misled", "constant"])
@pytest.mark.parametrize("d,M", [((1 << 21) + 1, 128), ((1 << 25) + 515, 8), ((1 << 27) + 3, 2)])
def test_adaptive_topk_from_a_sample(B, case, d, M):
    """Probabilities, levels and bands against a sort of every row on the device.  Its fp64 sums over a whole row round by at
    most d 2^-53 of the sum, 1.5e-8 for the longest row here; running sums of random order stay far below."""
    g = rows(case, M, d)
    want = {"layers": HELD, "normal": HELD, "misled": MISSED}.get(case, LEFT_OUT)
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        for k in ([d // 10_000 << l for l in range(13)] + [d], [d * (i + 1) // 10 for i in range(9)] + [d],
                  [0, 1, 2, d // 3, d // 3 + 1, d, d]):
            if len(k) == 10 and M == 128:
                check_sampled(B, ctx, g, k, [])         # ten brackets of so small samples are too wide
            elif case == "ties" and M == 128:
                check_adaptive(B, ctx, g, k)            # the list has about the room for the equal magnitudes
            else:
                check_sampled(B, ctx, g, k, [want] * M)
    finally:
        B.mlmc_destroy(ctx)


def test_held_and_missed_rows_of_one_call(B):
    """The workers with a missed bracket take the two sweeps of whole rows, the others do not; a schedule without a threshold."""
    M, d = 8, (1 << 25) + 515
    g = rows("normal", M, d)
    g[5] = rows("misled", 1, d)
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        check_sampled(B, ctx, g, doubling(d), [HELD] * 5 + [MISSED] + [HELD] * 2)
        g[0] = rows("misled", 1, d)
        check_sampled(B, ctx, g, equal(d, 5), [MISSED] + [HELD] * 4 + [MISSED] + [HELD] * 2)
        check_sampled(B, ctx, g, [d], [HELD] * M)
        g[7] = 0.0
        check_sampled(B, ctx, g, doubling(d), [LEFT_OUT] * M)
    finally:
        B.mlmc_destroy(ctx)


@pytest.mark.parametrize("kept", [32, 31, 1])
def test_candidates_are_kept_in_place(B, kept):
    """Of every 32 entries of the batches that hold candidates, `kept` share a bin with the threshold and the others lie in the bin
    above: the pass that keeps the former moves every key by 0 places, by few or by many."""
    M, d = 8, (1 << 25) + 515
    gen = torch.Generator(device="cuda").manual_seed(73)
    g = padded(torch.randn((M, d), generator=gen, device="cuda"), 4)
    g.mul_(1e-3)
    for m in range(M):
        at = torch.arange(d // 50, device="cuda") + m * 12_345
        key = torch.randint(0, 1 << 16, (len(at),), generator=gen, device="cuda", dtype=torch.int32) + 0x3F000000
        key += ((at * 7 % 32) >= kept).int() << 16
        g[m, at] = key.view(torch.float32) * torch.where(at % 3 == 0, -1.0, 1.0)
    above = d // 50 * (32 - kept) // 32
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        check_sampled(B, ctx, g, [above + (d // 50 - above) // 3, d], [HELD] * M)
        check_sampled(B, ctx, g, [above // 2, above + (d // 50 - above) // 3, d], [HELD] * M)
    finally:
        B.mlmc_destroy(ctx)


def test_sampled_rows_report_non_finite_entries(B):
    d = (1 << 27) + 5
    g = rows("normal", 2, d)
    g[1, d - 1] = float("nan")
    k = [d // 100, d // 10, d]
    out = B.TopkBuffers(2, d)
    ctx = B.mlmc_create(0, d, 2, 32)
    try:
        B.mlmc_compress_topk(ctx, g, k, None, 0, 0, out)
        assert B.mlmc_get_status(ctx) == B.MLMC_ERR_NONFINITE
        assert out.level[1] == -1 and out.count[1] == 0 and out.level[0] >= 0
    finally:
        B.mlmc_destroy(ctx)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [1_700_000, 1_700_353, 1_700_864 + 1])
def test_batches_that_round_to_zero_are_not_read(B, ora, dtype, d):
    """Calls above 100 MB; few entries far above the others, so that most batches round to 0 at the coarse levels and none at the
    fine ones; random signs, so that a missed sign plane shows."""
    M = 32 if dtype == "bf16" else 16
    rng = np.random.default_rng(72)
    g_np = (rng.standard_normal((M, d)) * 1e-3).astype(np.float32)
    for m in range(M):
        g_np[m, rng.integers(0, d, 50)] *= 200.0
    g_np[0, d // 2], g_np[1, -1], g_np[2, 0] = 1.0, -1.0, 1.0
    g_np[3] *= 1e-30
    g = to_dev(g_np)
    if dtype == "bf16":
        g = padded(g.to(torch.bfloat16), 8)
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        for step in range(2):         # levels drawn worker by worker
            check_bitwise(B, ora, ctx, g, [1, 2, 4, 8, 16, 23], [1 / 6] * 6, 1, step)
            check_rtn(B, ora, ctx, g, [2, 4, 8, 16], [0.2] * 5, 1, step)
        check_bitwise(B, ora, ctx, g, [1, 2, 4, 8, 16, 23], None, 1, 0)
        check_rtn(B, ora, ctx, g, [2, 4, 8, 16], None, 1, 0, expect_excluded=2)
    finally:
        B.mlmc_destroy(ctx)


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("d", [12 * 144 * 1024, 12 * 144 * 1024 + 1])
def test_groups_per_warp(B, ora, dtype, d):
    """The last row of 32 workers whose message has three blocks per SM (148 SMs: twelve groups for each of 144 warps), and the first with
    four: layers, so that some groups are read and some are not."""
    M = 32
    gen = torch.Generator(device="cuda").manual_seed(d)
    scale = torch.repeat_interleave(10.0 ** (torch.rand(40, generator=gen, device="cuda") * 4 - 5), -(-d // 40))[:d]
    g = padded((torch.randn((M, d), generator=gen, device="cuda") * scale).to(torch.bfloat16 if dtype == "bf16" else torch.float32), 8)
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        check_bitwise(B, ora, ctx, g, [1, 2, 4, 8, 16, 23], [1 / 6] * 6, 1, 0)
    finally:
        B.mlmc_destroy(ctx)


def kernel_ms(B, ctx, call):
    """Milliseconds of every kernel in one call."""
    import ctypes as C
    call(), call()
    L, n = B.lib(), B.lib().mlmc_kernel_count()
    ms, launches = (C.c_double * n)(), (C.c_int64 * n)()
    L.mlmc_timing_enable(ctx, 1)
    L.mlmc_timing_read(ctx, ms, launches, B._stream())
    call()
    assert L.mlmc_timing_read(ctx, ms, launches, B._stream()) == B.MLMC_OK
    L.mlmc_timing_enable(ctx, 0)
    return {L.mlmc_kernel_name(i).decode(): ms[i] for i in range(n) if launches[i]}


@pytest.mark.parametrize("case,some", [("ties", 8), ("zeros", 8), ("constant", 8), ("zeros", 1)])
def test_rows_whose_candidates_have_no_room_are_not_swept(B, case, some):
    """A threshold among equal magnitudes that are more than the candidate list holds, in some workers' rows: the sample shows it, and
    the sweep between the brackets, which takes longer than the histogram sweep that follows, is left out (5 us against 170)."""
    M, d = 8, 1 << 25
    g = rows("normal", M, d)
    g[M - some:] = rows(case, some, d)
    k = [d // 10_000 << l for l in range(14)] + [d]
    p = torch.zeros((M, len(k)), dtype=torch.float64, device="cuda")
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        ms = kernel_ms(B, ctx, lambda: B.mlmc_level_probs(ctx, g, B.MLMC_TOPK, k, None, p, None))
        assert ms["bracket_sweep"] < 0.5 * ms["missed_hist1"], ms
        check_sampled(B, ctx, g, k, [LEFT_OUT] * M)
    finally:
        B.mlmc_destroy(ctx)


def equal(d, n):
    return [d * (i + 1) // n for i in range(n - 1)] + [d]


def doubling(d):
    return [d // 10_000 << l for l in range(14)] + [d]


@pytest.mark.parametrize("d,M,one,two", [
    (1 << 25, 8, [equal(1 << 25, 10), doubling(1 << 25)], [equal(1 << 25, 15), equal(1 << 25, 16)]),
    (2_100_001, 128, [equal(2_100_001, 5)], [equal(2_100_001, 10), equal(2_100_001, 15), doubling(2_100_001)]),
    (3_400_000, 80, [], [equal(3_400_000, 5), doubling(3_400_000)]),
    ((1 << 25) - 1, 8, [], [[1, (1 << 25) - 1]]),
])
def test_calls_that_one_sweep_serves(B, d, M, one, two):
    """Few workers and levels take one sweep; wide brackets (many workers, and so few samples of each), many levels and sweeps that
    leave SMs without a block cost more than the second sweep."""
    g = rows("layers", M, d)
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        for k in one + two:
            p = torch.zeros((M, len(k)), dtype=torch.float64, device="cuda")
            names = kernel_ms(B, ctx, lambda: B.mlmc_level_probs(ctx, g, B.MLMC_TOPK, k, None, p, None))
            assert ("bracket_sweep" in names) == (k in one) and ("sums_candidates" in names) == (k in two), (k, names)
            check_sampled(B, ctx, g, k, [HELD] * M if k in one else [])
    finally:
        B.mlmc_destroy(ctx)


@pytest.mark.parametrize("p", [None, [0.2] * 5])
def test_rows_of_one_scale_do_not_pay_for_the_look_at_the_batches(B, p):
    """RTN messages of calls above 100 MB look at every batch's largest entry.  Where no batch rounds to 0 (entries of one scale) they
    take as long as the messages that read everything, 1.62 times the dense average beside them; with the looks it was 1.89."""
    M, d = 8, 3_300_000
    gen = torch.Generator(device="cuda").manual_seed(74)
    g = padded(torch.randn((M, d), generator=gen, device="cuda"), 4)
    out, dense = B.RtnBuffers(M, d), torch.empty(d, device="cuda")
    ctx = B.mlmc_create(0, d, M, 32)

    def call():
        B.mlmc_compress_rtn(ctx, g, [2, 4, 8, 16], p, 1, 0, out)
        B.mlmc_aggregate_rtn(ctx, out, M, d, dense)

    try:
        ms = [kernel_ms(B, ctx, call) for _ in range(30)]
        emit, average = (min(x[name] for x in ms) for name in ("rtn_emit", "aggregate_dense"))
        assert emit < 1.76 * average, (emit, average)
    finally:
        B.mlmc_destroy(ctx)
