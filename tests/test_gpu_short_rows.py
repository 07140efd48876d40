"""The average of short Top-k messages in one launch."""
import numpy as np
import pytest
import torch

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
