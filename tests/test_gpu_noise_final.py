"""fm_noise_finalize: the fp32 S/N formed without FP64 square root and
division stays correctly rounded up to 2^-16 of an ulp, over the whole range
of variances and at its ends (zero, infinite, tiny and huge values)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1])  # 1: arrays aligned to their element only
def test_snr_rounding_over_the_variance_range(shift):
    from paper_1204_4293_gb300 import fastmap as fm
    n, J = 64, 3
    rng = np.random.default_rng(3)
    ne = (J - 1) * n * n
    v = np.exp(rng.uniform(np.log(1e-60), np.log(1e60), ne))
    v[: ne // 2] = np.exp(rng.uniform(np.log(1e-12), np.log(1e3), ne // 2))
    w = (rng.standard_normal(ne) * np.exp(rng.uniform(-60, 60, ne) / 2)).astype(np.float32)
    v[:6] = [0.0, 0.0, np.inf, 1e-300, 1e300, 4.0]
    w[:6] = [1.0, 0.0, 2.0, 1e-30, 1e30, 0.0]

    def put(a, dtype):
        t = torch.empty(a.size + shift, dtype=dtype, device="cuda")[shift:]
        return t.copy_(torch.from_numpy(a))

    sums = put(np.concatenate([np.zeros(ne), v]), torch.float64).view(2, J - 1, n, n)  # R = 2: variance = S2
    pyr = put(np.concatenate([w, np.zeros(n * n, np.float32)]), torch.float32).view(J, n, n)
    var, snr = fm.fm_noise_finalize(sums, 2, pyramid=pyr)
    assert np.array_equal(var.cpu().numpy().ravel(), v)
    got = snr.cpu().numpy().ravel()
    with np.errstate(all="ignore"):
        ref = w.astype(np.float64) / np.sqrt(v)
        ref32 = ref.astype(np.float32)
    special = ~np.isfinite(ref) | (np.abs(ref) < 1e-37) | (np.abs(ref) > 1e38)
    assert np.array_equal(got[special], ref32[special], equal_nan=True)
    ulp = np.spacing(np.abs(ref32[~special])).astype(np.float64)
    assert np.all(np.abs(got[~special] - ref[~special]) <= ulp * (0.5 + 2.0 ** -16))
