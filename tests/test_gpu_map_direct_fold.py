"""The folded direct M_ap (rows y + dy and y - dy together, one row a warp) at
the edges of its blocks, groups of taps and parts, against the FP64 oracle,
and the reach of a single bad pixel."""
import numpy as np
import pytest
import torch

import oracle
from helpers import rel_err
from paper_1204_4293_gb300 import synth

pytestmark = pytest.mark.gpu

# side x cut radius: around the 256- (fp64 128-) column tiles, around whole
# blocks of 8 (4) columns, aperture larger than the field, several parts
CASES = [(1, 3.0), (7, 1.0), (31, 2.5), (64, 6.9), (128, 8.0), (129, 9.0), (255, 3.0), (256, 7.0), (257, 15.0), (40, 70.0),
         (200, 33.3)]


def _fm():
    from paper_1204_4293_gb300 import fastmap
    return fastmap


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("n,cut", CASES)
def test_direct_and_masked_at_block_edges(n, cut, dtype):
    fm = _fm()
    filt = fm.FM_FILTER_S98
    tol = 1e-5 if dtype == np.float32 else 1e-12
    g1, g2 = (a.astype(dtype) for a in synth.white((2, n, n), seed=n, scale=0.1))
    w = (np.abs(synth.white((n, n), seed=n + 1)) * (synth.white((n, n), seed=n + 2) > -0.8)).astype(dtype)
    d = [a.astype(np.float64) for a in (g1, g2, w)]
    t = [torch.from_numpy(a).cuda() for a in (g1, g2, w)]
    m = fm.fm_map_direct(t[0], t[1], filt, cut).cpu().numpy()
    ref = oracle.map_direct(d[0], d[1], filt, cut)
    assert np.abs(ref).max() == 0 or rel_err(m, ref) <= tol
    if n == 1 or cut == 1.0:  # S98 vanishes at its radius, up to the rounding of 1 - 1
        assert np.abs(m).max() <= 1e-6
    m, cov = fm.fm_map_direct_masked(*t, filt, cut, coverage=True)
    mr, cr = oracle.map_direct_masked(*d, filt, cut)
    m, cov = m.cpu().numpy().astype(np.float64), cov.cpu().numpy().astype(np.float64)
    # sums of positive weights only: relative error, pixel by pixel
    assert np.all(np.abs(cov - cr) <= (1e-5 if dtype == np.float32 else 1e-13) * cr)
    s = mr * cr
    assert np.abs(s).max() == 0 or rel_err(m * cov, s) <= tol


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_bad_pixel_stays_within_the_radius(bad):
    fm = _fm()
    n, theta, py, px = 96, 9.0, 41, 50
    g1, g2 = (torch.from_numpy(a.astype(np.float32)).cuda() for a in synth.white((2, n, n), seed=3, scale=0.1))
    clean = fm.fm_map_direct(g1, g2, fm.FM_FILTER_JBJ04, theta, cut_over_theta=1.0)
    g1[py, px] = bad
    m = fm.fm_map_direct(g1, g2, fm.FM_FILTER_JBJ04, theta, cut_over_theta=1.0)
    y, x = torch.meshgrid(torch.arange(n), torch.arange(n), indexing="ij")
    inside = ((y - py) ** 2 + (x - px) ** 2 <= theta ** 2).cuda()
    assert torch.equal(m[~inside], clean[~inside])
    assert not torch.isfinite(m[inside]).any()
