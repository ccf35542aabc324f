"""fm_band_moments of maps above 4096^2: a strand still holds at most 16 pixels,
so the fp32 sum of equal pixels is off by at most 15 roundings."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,rest", [(4100, 2.0 ** -21), (12000, 2.0 ** -18)])
def test_strands_of_large_maps_stay_short(n, rest):
    from paper_1204_4293_gb300 import fastmap as fm
    # from a partial sum of rest 2^24 on every addition rounds up
    x = 1.0 + rest + 2.0 ** -22
    got = fm.fm_band_moments(torch.full((1, 1, n, n), x, device="cuda")).cpu()[0, 0, 0].item()
    assert abs(got - x) <= 15 * 2.0 ** -24 * x
