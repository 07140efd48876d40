"""Short Top-k rows: the cluster kernel at every cluster size, and the average in one launch."""
import numpy as np
import pytest
import torch

from test_gpu_dispatch import doubling, geometric, layered
from test_gpu_ext import check_stopk
from test_gpu_parity import check_topk, padded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_05508_b200 import binding
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.mlmc_create(0, 2_500_000, 32, 32)
    yield c
    B.mlmc_destroy(c)


def rows(kind, d, M, dtype):
    rng = np.random.default_rng(d)
    if kind == "layers":
        return layered(d, M, dtype)
    if kind == "one_bin":      # every key is a boundary key: the lists of the warps are too short
        x = 1.0 + 0.02 * rng.random((M, d))
    elif kind == "ties":
        x = rng.choice(np.array([0.5, -0.5, 0.25, 3.0, 0.1]), (M, d))
    else:                      # zeros, and entries over the whole exponent range
        x = rng.standard_normal((M, d)) * 10.0 ** rng.uniform(-30, 10, (M, d)) * (rng.random((M, d)) < 0.3)
    return padded(torch.from_numpy(x.astype(np.float32)).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32), 8)


# rows of a block, of clusters of two to sixteen, and one entry more; few queries (every block resolves them all) and 31
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["layers", "one_bin", "ties", "zeros"])
@pytest.mark.parametrize("d", [7, 513, 8_192, 8_193, 16_385, 30_001, 65_537, 300_001])
def test_cluster_sizes(B, ora, ctx, dtype, kind, d):
    g = rows(kind, d, 2, dtype)
    few, many = [max(1, d // 9), d], sorted({d * (i + 1) // 32 for i in range(31)} - {0}) + [d]
    for k in (few, [0] + few, many, [0, 0] + many[2:-1] + [d]):
        check_topk(B, ora, ctx, g, k, None, 5, 1, expect_excluded=1)
        check_topk(B, ora, ctx, g, k, geometric(len(k)), 5, 2, expect_excluded=1)


# the longest bf16 rows of a cluster with given p, in one wave and in two
@pytest.mark.parametrize("d,M", [(1_032_192, 2), (1_032_193, 2), (524_288, 12), (524_289, 12)])
def test_bf16_rows_given_p(B, ora, ctx, d, M):
    k = doubling(d, d // 500)
    check_topk(B, ora, ctx, layered(d, M, "bf16"), k, geometric(len(k)), 3, 1, expect_excluded=1)


# more segments than levels, given p: the longest fp32 rows of a cluster, which keep no brackets
@pytest.mark.parametrize("d", [262_145, 745_472, 745_473])
def test_segments_given_p(B, ora, ctx, d):
    s = d // 100
    L = -(-d // s)
    check_stopk(B, ora, ctx, layered(d, 3), s, geometric(L), 3, 1)
    check_stopk(B, ora, ctx, rows("ties", d, 2, "f32"), s, [1.0 / L] * L, 3, 2)


# fp32, given p: the longest rows on 8 blocks where clusters of 16 run at a time and where they take turns, and one entry more
@pytest.mark.parametrize("d,M", [(262_144, 2), (262_145, 2), (262_144, 20), (372_736, 9), (372_737, 9), (372_736, 24)])
def test_rows_on_eight_blocks(B, ora, ctx, d, M):
    s = d // 40
    L = -(-d // s)
    check_stopk(B, ora, ctx, layered(d, M), s, geometric(L), 3, 1)
    if d <= 262_144:
        k = doubling(d, d // 500)
        check_topk(B, ora, ctx, layered(d, M), k, geometric(len(k)), 3, 1, expect_excluded=1)


# edges of the tiles; empty, void and dense messages; lanes per search edge from 32 to 4
@pytest.mark.parametrize("d", [1, 1_023, 1_025, 4_097, 200_001, 1_212_417])
@pytest.mark.parametrize("M", [1, 3, 9, 32])
def test_average_in_one_launch(B, ctx, d, M):
    rng = np.random.default_rng(M)
    out = B.TopkBuffers(M, d)
    ref = np.zeros(d, dtype=np.float32)
    for m in range(M):
        share = [0.0, 1.0, 0.001, 0.3][m % 4] if M > 1 else 0.3
        idx = np.flatnonzero(rng.random(d) < share).astype(np.int32)
        val = rng.standard_normal(idx.size).astype(np.float32)
        void = m % 7 == 6
        out.idx[m, :idx.size] = torch.from_numpy(idx).cuda()
        out.val[m, :idx.size] = torch.from_numpy(val).cuda()
        out.count[m], out.level[m] = idx.size, -1 if void else 0
        if not void:
            ref[idx] += val
    dense = torch.full((d,), float("nan"), device="cuda")
    B.mlmc_aggregate(ctx, B.MLMC_TOPK, out, None, M, d, dense)
    # the additions are those of the loop above, in the same order; the product with 1 / M rounds once
    assert np.array_equal(dense.cpu().numpy(), ref * np.float32(1.0 / M))


# in one launch, in two, and in two without a context; some lanes per search and one
@pytest.mark.parametrize("d", [5_000, 2_424_833, 70_000_001])
def test_counts_below_zero_are_empty_messages(B, d):
    M = 9
    rng = np.random.default_rng(d)
    out = B.TopkBuffers(M, 1000)
    ref = np.zeros(d, dtype=np.float32)
    for m in range(M):
        idx = np.sort(rng.choice(d, 1000, replace=False)).astype(np.int32)
        val = rng.standard_normal(1000).astype(np.float32)
        out.idx[m], out.val[m] = torch.from_numpy(idx).cuda(), torch.from_numpy(val).cuda()
        out.count[m], out.level[m] = (-1, -(1 << 40), 1000)[m % 3], 0
        if m % 3 == 2:
            ref[idx] += val
    ref *= np.float32(1.0 / M)
    c = B.mlmc_create(0, d, M, 32)
    try:
        for average in (lambda to: B.mlmc_aggregate(c, B.MLMC_TOPK, out, None, M, d, to),
                        lambda to: B.mlmc_aggregate_topk_noalloc(out, M, d, to)):
            dense = torch.full((d,), float("nan"), device="cuda")
            average(dense)
            assert np.array_equal(dense.cpu().numpy(), ref)  # the same additions in the same order
    finally:
        B.mlmc_destroy(c)
