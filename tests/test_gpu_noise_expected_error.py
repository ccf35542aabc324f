"""Rounding error of the fp32 expected variance against the fp64 call's, over
all bands: 0.425 x 2^-24 a rounding (rms, values spread evenly over their
binade), about 18 roundings a one-dimensional transform and six transforms."""
import numpy as np
import pytest
import torch

from helpers import shear

pytestmark = pytest.mark.gpu
BOUND = 0.425 * 2.0 ** -24 * (6 * 18) ** 0.5  # 2.6e-7


def _errors(n, J):
    from paper_1204_4293_gb300 import fastmap as fm
    g1, g2 = (torch.from_numpy(a.astype(np.float32)).cuda() for a in shear(n, seed=n))
    ref = fm.fm_map_noise_expected(g1.double(), g2.double(), J)
    return fm.fm_map_noise_expected(g1, g2, J).double() - ref, ref


@pytest.mark.parametrize("n,J", [(32, 3), (64, 4), (128, 5), (256, 6), (512, 7), (1024, 7)])
def test_error_over_all_bands(n, J):
    d, ref = _errors(n, J)
    assert (d.pow(2).mean() / ref.pow(2).mean()).sqrt().item() <= BOUND


@pytest.mark.parametrize("n,J", [(64, 4), (256, 6), (512, 7), (1024, 7), (1024, 4), (256, 3)])
def test_error_of_each_band(n, J):
    d, ref = _errors(n, J)
    rel = d.pow(2).mean(dim=(-1, -2)).sqrt() / ref.mean(dim=(-1, -2))
    assert rel.max().item() <= BOUND, rel.tolist()
