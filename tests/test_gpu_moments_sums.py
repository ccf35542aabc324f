"""fm_band_moments adds its strands with at least the 53 bits of an FP64 sum:
values whose sum needs all of them, spread over the strands of a thread or
over the lanes of a warp, give the exact mean."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])  # 16-byte aligned: four strands a thread; else one
@pytest.mark.parametrize("where", [(0, 1, 2, 3), (0, 3, 17, 40), (255, 128, 64, 1)])  # four strands (256 pixels apart)
def test_sums_keep_fp64_bits(where, shift):
    from paper_1204_4293_gb300 import fastmap as fm
    n = 64
    vals = [2.0 ** 20, 2.0 ** -5 + 2.0 ** -28, 2.0 ** -32, -2.0 ** 20]  # 53 bits from the first to the last
    x = torch.zeros(n * n + shift, device="cuda")[shift:]
    for p, v in zip(where, vals):
        x[p] = v
    got = fm.fm_band_moments(x.view(1, 1, n, n)).cpu()[0, 0, 0].item()
    assert got * n * n == vals[1] + vals[2]
