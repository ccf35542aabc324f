"""The rotated shear of the noise maps, one realisation at a time: its bands
(fp32) against the fp64 pipeline on the oracle's rotated shear.

Tolerance: the rotation adds at most 4.7e-8 of |gamma| a pixel, and each of
the two fp32 transforms' log2(n^2) <= 24 levels at most 6e-8 of its input's
rms: sqrt(2 * 24) * 6e-8 = 4.2e-7 rms of the convergence, times 6 for the
largest of up to 2^24 pixels = 2.5e-6, doubled for the smoothing's own
roundings."""
import numpy as np
import pytest
import torch

import oracle
from helpers import shear

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,r", [(16, 3, 0), (32, 3, 4), (64, 4, 1), (256, 6, 7), (512, 5, 2), (1024, 7, 99), (2048, 4, 3),
                                   (4096, 3, 1)])
def test_one_realisation_matches_fp64(n, J, r):
    from paper_1204_4293_gb300 import fastmap as fm
    seed = 2**63 + 12345
    g1, g2 = shear(n, seed=5, dtype=np.float32)
    sums = fm.fm_map_noise_accumulate(torch.from_numpy(g1).cuda(), torch.from_numpy(g2).cuda(), J, r, 1, seed=seed)
    a, c = oracle.rotate_shear(g1.astype(np.float64), g2.astype(np.float64), r, seed)
    ta, tc = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (a, c))
    ref = fm.fm_map_starlet(ta, tc, J)
    rms = fm.fm_ks_invert(ta, tc)[0].pow(2).mean().sqrt().item()
    assert (sums[0] - ref[:J - 1]).abs().max().item() / rms <= 5e-6
    fm.fm_trim()
