"""Level statistics on pairs of entries: zeros, numbers below the normal range and the largest magnitude in either place."""
import numpy as np
import pytest
import torch

from test_gpu_ext import check_rtn
from test_gpu_parity import check_bitwise, padded

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_05508_b200 import binding
    binding.lib()
    return binding


@pytest.fixture(scope="module")
def ctx(B):
    c = B.mlmc_create(0, 700_000, 3, 32)
    yield c
    B.mlmc_destroy(c)


def rows(kind, d, dtype):
    rng = np.random.default_rng(d)
    x = rng.standard_normal((2, d))
    if kind == "tiny":           # most entries below the normal range or zero, the others small beside the largest
        x *= 10.0 ** rng.uniform(-44, -36, (2, d)) * (rng.random((2, d)) < 0.7)
        x[:, ::97] = 1e-33 * rng.standard_normal(x[:, ::97].shape)
    elif kind == "largest":      # half of the entries have the largest magnitude
        x = np.where(rng.random((2, d)) < 0.5, np.sign(x) * 0.75, x * 0.1)
    elif kind == "large":
        x *= 1e35
    return padded(torch.from_numpy(x.astype(np.float32)).cuda().to(torch.bfloat16 if dtype == "bf16" else torch.float32), 8)


# short rows in one launch and long ones in three
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("kind", ["tiny", "largest", "large"])
@pytest.mark.parametrize("d", [20_003, 600_001])
def test_statistics(B, ora, ctx, dtype, kind, d):
    g = rows(kind, d, dtype)
    check_rtn(B, ora, ctx, g, [2, 4, 8, 16], None, 3, 1)
    check_bitwise(B, ora, ctx, g, [1, 2, 4, 8, 16, 23], None, 3, 1)
    check_bitwise(B, ora, ctx, g, [2, 14, 23], None, 3, 2)


# Largest magnitudes for which a grid step or its reciprocal leaves the fp32 range: an entry and its negative then differ in the clipping.
@pytest.mark.parametrize("widths", [[2, 4, 8, 16], [1, 2, 9], [16], [1]])
@pytest.mark.parametrize("largest", [1e-41, 1e-44, 1e-36, 2e38, 3.3e38])
@pytest.mark.parametrize("d", [5_003, 20_003, 600_001])
def test_grids_out_of_range(B, ora, ctx, d, largest, widths):
    rng = np.random.default_rng(d)
    x = np.clip(rng.standard_normal((2, d)), -3, 3) / 3 * largest * (rng.random((2, d)) < 0.9)
    x[0, 5], x[1, 6] = largest, -largest
    g = padded(torch.from_numpy(x.astype(np.float32)).cuda(), 8)
    L = len(widths) + 1
    p = torch.zeros((2, L), dtype=torch.float64, device="cuda")
    delta = torch.zeros((2, L), dtype=torch.float64, device="cuda")
    B.mlmc_level_probs(ctx, g, B.MLMC_RTN, widths, None, p, delta)
    assert B.mlmc_get_status(ctx) == 0
    for m in range(2):
        o = ora.rtn(x[m].astype(np.float32), widths, None)
        # either side adds d squares in fp64, in an order of its own: d roundings of 2^-53 each at most, halved by the root
        assert np.allclose(delta[m].cpu().numpy(), o.delta, rtol=d * 2.0 ** -53 + 1e-14, atol=0)
        assert np.allclose(p[m].cpu().numpy(), o.p, rtol=2 * (d * 2.0 ** -53 + 1e-14), atol=1e-300)
    if largest < 1.0:  # otherwise the messages' values, divided by their probability, leave the range
        check_rtn(B, ora, ctx, g, widths, None, 3, 1)
        check_rtn(B, ora, ctx, g, widths, [1.0 / L] * L, 3, 2)


# A call of more than 100 MB, whose message looks at the batches: no entry rounds to 0 where delta overflows.
def test_grid_out_of_range_in_a_long_message(B, ora):
    d = 26_300_003
    x = np.random.default_rng(0).uniform(-1.0, 1.0, (1, d)).astype(np.float32)
    x[0, :d // 2] *= 1e-3
    x *= np.float32(3e38)
    out = B.RtnBuffers(1, d)
    c = B.mlmc_create(0, d, 1, 32)
    try:
        B.mlmc_compress_rtn(c, padded(torch.from_numpy(x).cuda(), 8), [1, 2], [0.999, 0.0005, 0.0005], 3, 1, out)
        assert B.mlmc_get_status(c) == 0
        o = ora.rtn(x[0], [1, 2], [0.999, 0.0005, 0.0005], seed=3, step=1, worker=0)
        assert o.level == 0 and int(out.level[0]) == 0
        assert np.array_equal(out.val[0, :d].cpu().numpy(), o.val)  # +-c, divided by p in fp64 and rounded once
    finally:
        B.mlmc_destroy(c)
