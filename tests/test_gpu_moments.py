"""fm_band_moments at the edges of its strands, vectors and array groups,
against numpy in FP64, and on values whose sums leave the fp32 range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fm():
    from paper_1204_4293_gb300 import fastmap
    return fastmap


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,J,batch,shift", [(1, 2, 3, 0), (5, 1, 1, 0), (63, 3, 2, 0), (64, 2, 1, 1), (66, 2, 2, 0),
                                             (257, 3, 1, 0), (1024, 4, 4, 0), (1030, 2, 1, 3)])
def test_moments_match_numpy(n, J, batch, shift, dtype):
    fm = _fm()
    g = torch.Generator().manual_seed(n * J + batch)
    x = torch.randn(batch * J * n * n + shift, generator=g, dtype=torch.float64)
    x = (0.3 + x + 0.1 * x * x).to(dtype).cuda()[shift:].view(batch, J, n, n)  # shift: not 16-byte aligned
    got = fm.fm_band_moments(x).cpu().numpy()
    d = x.double().cpu().numpy().reshape(batch, J, -1)
    mean = d.mean(-1)
    d = d - mean[..., None]
    m2, a3, m3, m4 = (d ** 2).mean(-1), (np.abs(d) ** 3).mean(-1), (d ** 3).mean(-1), (d ** 4).mean(-1)
    # fp32 strands of at most 16 terms, each term of at most four roundings
    # (the pixel itself may be rounded to fp32, the mean is)
    u = 24 * 2.0 ** -24
    assert np.all(np.abs(got[..., 0] - mean) <= u * (np.abs(mean) + np.sqrt(m2)))
    assert np.all(np.abs(got[..., 1] - m2) <= u * (m2 + mean ** 2 * u))
    if n > 1:
        assert np.all(np.abs(got[..., 2] - m3 / m2 ** 1.5) <= 3 * u * a3 / m2 ** 1.5 + u)
        assert np.all(np.abs(got[..., 3] - (m4 / m2 ** 2 - 3)) <= 4 * u * m4 / m2 ** 2)


def test_moments_of_sums_beyond_fp32():
    # |x| = 2^30: x^4 = 2^120, so strands stay finite and their fp32 sum would not
    fm = _fm()
    x = torch.ones((1, 1, 512, 512), device="cuda")
    x[..., ::2] = -1.0
    got = fm.fm_band_moments(x * 2.0 ** 30).cpu().numpy()[0, 0]
    assert got[0] == 0.0 and got[1] == 2.0 ** 60 and got[2] == 0.0 and abs(got[3] + 2.0) <= 1e-12
    x[0, 0, 7, 9] = float("inf")
    got = fm.fm_band_moments(x).cpu().numpy()[0, 0]
    assert got[0] == float("inf") and np.isnan(got[1])
