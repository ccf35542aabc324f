"""The starlet of values near the top of the type's range (the plain fp32
form, fp64): finite and, scaled by a power of two, bit-identical to that of
small values; infinities and NaN reach the outputs that their taps reach."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fm():
    from paper_1204_4293_gb300 import fastmap
    return fastmap


def _map(n, dtype):
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand(2, n, n, device="cuda", dtype=dtype, generator=g) + 0.5
    return torch.where(torch.rand(2, n, n, device="cuda", generator=g) < 0.3, -x, x)


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n,J,dtype,kw", [(100, 5, torch.float32, {"fuse_depth": -1, "large_path": 1}),
                                          (128, 6, torch.float32, {"fuse_depth": -1, "large_path": 3}),
                                          (37, 4, torch.float32, {"fuse_depth": -1}),
                                          (256, 7, torch.float64, {}), (74, 5, torch.float64, {}),
                                          (1024, 4, torch.float64, {}), (37, 4, torch.float64, {})])
def test_values_near_the_top_of_the_range(n, J, dtype, kw, boundary):
    fm = _fm()
    top = 125 if dtype == torch.float32 else 1021  # |x| < 2^top 1.5, sums of two below the largest value
    x = _map(n, dtype)
    ref = fm.fm_starlet_forward(x, J, boundary=boundary, **kw)
    got = fm.fm_starlet_forward(torch.ldexp(x, torch.tensor(top)), J, boundary=boundary, **kw)
    assert torch.isfinite(got).all()
    assert torch.equal(got, torch.ldexp(ref, torch.tensor(top)))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_fp64_bad_pixel_stays_within_the_taps(bad):
    fm = _fm()
    n, J, py, px = 128, 3, 60, 71
    x = _map(n, torch.float64)
    clean = fm.fm_starlet_forward(x, J)
    x[1, py, px] = bad
    got = fm.fm_starlet_forward(x, J)
    for j, reach in ((0, 2), (1, 6), (2, 6)):  # half widths of one and two scales' taps
        m = torch.zeros(n, n, dtype=torch.bool, device="cuda")
        m[py - reach:py + reach + 1, px - reach:px + reach + 1] = True
        assert torch.equal(got[1, j][~m], clean[1, j][~m])
        assert not torch.isfinite(got[1, j, py, px])
    assert torch.equal(got[0], clean[0])
