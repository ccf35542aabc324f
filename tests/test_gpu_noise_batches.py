"""Noise maps over full and short last batches (a batch: 32 realisations):
the S/N's bands lie behind the last batch's pyramids or in the first pyramid,
and the sums of a call may be 16-byte aligned or not.

Tolerance of the S/N: one fp32 rounding of w / sqrt(var), 6e-8, and that of
the comparison's own fp32 bands (the same kernels): 2.5e-7 of |w| / sqrt(var)."""
import numpy as np
import pytest
import torch

from helpers import shear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 512, 1024])
@pytest.mark.parametrize("R,accum", [(2, 0), (31, 0), (32, 0), (33, 0), (64, 0), (65, 1), (96, 0)])
def test_snr_is_the_band_over_its_deviation(n, R, accum):
    from paper_1204_4293_gb300 import fastmap as fm
    J = 4
    g1, g2 = (torch.from_numpy(v).cuda() for v in shear(n, seed=3, dtype=np.float32))
    fm.fm_tune(fm.FM_TUNE_KS_REAL, 1)  # small maps too by the kernels of the noise maps, so that the bands are equal
    try:
        for _ in range(2):  # recorded, then replayed
            var, snr = fm.fm_map_noise(g1, g2, J, R, seed=9, accum=accum)
            ref = fm.fm_map_starlet(g1, g2, J)[:J - 1].double() / var.sqrt()
            # a pixel whose two realisations agree has variance 0 and an infinite S/N on both sides
            assert (((snr.double() - ref).abs() <= 2.5e-7 * ref.abs()) | (snr.double() == ref)).all()
    finally:
        fm.fm_tune(fm.FM_TUNE_KS_REAL, -1)
        fm.fm_trim()


@pytest.mark.parametrize("R", [5, 37])
def test_sums_aligned_to_eight_bytes(R):
    from paper_1204_4293_gb300 import fastmap as fm
    n, J = 64, 4
    g1, g2 = (torch.from_numpy(v).cuda() for v in shear(n, seed=3, dtype=np.float32))
    size = 2 * (J - 1) * n * n
    odd = torch.zeros(size + 1, dtype=torch.float64, device="cuda")[1:].view(2, J - 1, n, n)
    assert odd.data_ptr() % 16 == 8
    a = fm.fm_map_noise_accumulate(g1, g2, J, 0, R, seed=9, sums=odd)
    b = fm.fm_map_noise_accumulate(g1, g2, J, 0, R, seed=9)
    assert torch.equal(a, b)
    fm.fm_trim()
