"""The fp32 transform's mean gain: rounded constants make every amplitude too
small by the same share, which the last scaling takes up to the nearest
multiple of 2^-23; what is left is at most half of that, 2^-24, and 1e-8 for
the reciprocals of the KS multiply."""
import pytest
import torch

pytestmark = pytest.mark.gpu
BOUND = 2.0 ** -24 + 1e-8


def _gain(got, ref):
    return float((got.double() * ref).sum() / (ref * ref).sum()) - 1.0


@pytest.mark.parametrize("n", [32, 64, 128, 256, 512, 1024, 2048])
def test_fp32_amplitudes_are_not_biased(n):
    from paper_1204_4293_gb300 import fastmap as fm
    g = torch.Generator(device="cuda").manual_seed(n)
    batch = max(1, 1024 // n) ** 2 if n < 1024 else 1
    g1, g2 = (0.1 * torch.randn(batch, n, n, device="cuda", generator=g) for _ in range(2))
    kE, kB = fm.fm_ks_invert(g1.double(), g2.double(), with_b=True)
    # one call of every map, and map by map (up to 256^2: the one-kernel form)
    calls = [(g1, g2, kE, kB)] + [(g1[b:b + 1], g2[b:b + 1], kE[b:b + 1], kB[b:b + 1]) for b in range(min(batch, 4))]
    for a, b, rE, rB in calls:
        e, m = fm.fm_ks_invert(a.contiguous(), b.contiguous(), with_b=True)
        if a.numel() >= 4096 * 4:  # enough pixels for a mean
            assert abs(_gain(e, rE)) <= BOUND and abs(_gain(m, rB)) <= BOUND
            assert abs(_gain(fm.fm_ks_invert(a.contiguous(), b.contiguous())[0], rE)) <= BOUND
    f1, f2 = fm.fm_ks_forward(kE.float())
    r1, r2 = fm.fm_ks_forward(kE)
    assert abs(_gain(f1, r1)) <= BOUND and abs(_gain(f2, r2)) <= BOUND
