"""Long bf16 rows: the histogram with several counts per bin, and what lies outside its window."""
import pytest
import torch

from test_gpu_parity import padded
from test_gpu_sampled import check_adaptive

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    from paper_2507_05508_b200 import binding
    binding.lib()
    return binding


WARPS, TILE, BATCH = 32, 8192, 1024  # warps of a block; entries of a tile and of a batch
FROM = 8                             # batches per warp from which on a row is sampled


def blocks(d, M):
    """Blocks per row: those of launch_hist1."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    waves = 2 if sms // M * M * 20 < sms * 19 else 1
    return max(1, min(-(-d // (8 * 4096)), sms * waves // M))


def batches_per_warp(d, M):
    return -(-(-(-d // TILE) * TILE // BATCH) // (blocks(d, M) * WARPS))


def sampled(d, M):
    """Mask of the keys that the blocks of a row sample: a vector of eight per thread, from its share of the row."""
    share = (d // 8) // 1024
    t = torch.arange(1024)
    mask = torch.zeros(d, dtype=torch.bool)
    for block in range(blocks(d, M)):
        at = t * share + (block * 37 + t * 11) % share
        mask[(at[:, None] * 8 + torch.arange(8)).flatten()] = True
    return mask.cuda()


# one block per row: the longest row that is too short to be sampled, one entry more, a ragged end; two blocks per row
@pytest.mark.parametrize("case", ["layers", "zeros", "few_zeros", "wide", "tiny", "sample_above", "sample_below", "constant", "uniform", "signs"])
@pytest.mark.parametrize("d,per_sm,n,columns", [(28 * TILE, 1.0, 1, False), (28 * TILE + 1, 1.0, 1, True), (262_147, 1.0, 1, True),
                                                (700_001, 0.68, 2, True)])
def test_thresholds_and_norms(B, case, d, per_sm, n, columns):
    M = int(torch.cuda.get_device_properties(0).multi_processor_count * per_sm)
    assert blocks(d, M) == n and (batches_per_warp(d, M) >= FROM) == columns
    gen = torch.Generator(device="cuda").manual_seed(d)
    g = torch.randn((M, d), generator=gen, device="cuda")
    if case == "layers":
        g *= torch.repeat_interleave(10.0 ** (torch.rand(40, generator=gen, device="cuda") * 4 - 5), -(-d // 40))[:d]
    elif case in ("zeros", "few_zeros"):
        g *= torch.rand((M, d), generator=gen, device="cuda") < (0.05 if case == "zeros" else 0.995)
    elif case == "wide":              # over 60 octaves
        g *= 2.0 ** (torch.rand((M, d), generator=gen, device="cuda") * 60 - 40)
    elif case == "tiny":              # the window starts at the smallest numbers
        g *= 2.0 ** -120
    elif case == "sample_above":      # the window lies above everything else, by 16, 26 and 50 octaves
        g[:, sampled(d, M)] = 8.0
        for i, octaves in enumerate((16, 26, 50)):
            g[i::3, ~sampled(d, M)] *= 2.0 ** -octaves
    elif case == "sample_below":      # and below, by 4, 10 and 50
        g[:, sampled(d, M)] = 1.0
        for i, octaves in enumerate((4, 10, 50)):
            g[i::3, ~sampled(d, M)] *= 2.0 ** octaves
    elif case == "uniform":           # half of the keys lie in the octave of the largest
        g.uniform_(-1.0, 1.0, generator=gen)
    elif case == "signs":
        g.sign_()
    else:
        g.fill_(0.25)
    g = padded(g.to(torch.bfloat16), 8)
    ctx = B.mlmc_create(0, d, M, 32)
    try:
        check_adaptive(B, ctx, g, [d // 500 << l for l in range(8)] + [d])
        check_adaptive(B, ctx, g, [0, 1, d // 3, d // 3 + 1, d - 1, d])
    finally:
        B.mlmc_destroy(ctx)
