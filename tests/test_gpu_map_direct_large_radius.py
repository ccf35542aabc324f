"""The direct and the masked sum at radii up to the largest one (2048 px), where
a CTA holds four, two or one warps, and on buffers aligned to their element
only, against an FP64 convolution."""
import numpy as np
import pytest
import torch

signal = pytest.importorskip("scipy.signal")
from helpers import rel_err  # noqa: E402
from paper_1204_4293_gb300 import synth  # noqa: E402

pytestmark = pytest.mark.gpu


def _reference(g1, g2, w, R):
    """JBJ04 with theta = R cut at R, over every offset inside the field."""
    n = g1.shape[0]
    d = np.arange(-(n - 1), n, dtype=np.float64)
    dx, dy = d[None, :], d[:, None]
    r2 = dx * dx + dy * dy
    disc = (r2 > 0) & (r2 <= R * R)
    r2s = np.where(r2 > 0, r2, 1.0)
    x = 0.5 * r2 / R ** 2
    q = np.where(disc, x * np.exp(-x) / R ** 2, 0.0)
    a, b = -q * (dx * dx - dy * dy) / r2s, -q * 2 * dx * dy / r2s

    def corr(t, m):
        return signal.fftconvolve(m, t[::-1, ::-1], mode="full")[n - 1:2 * n - 1, n - 1:2 * n - 1]

    m = corr(a, g1 * w) + corr(b, g2 * w)
    if np.isscalar(w):
        return m
    k = np.arange(-int(R), int(R) + 1, dtype=np.float64)
    n_r = int((k[None, :] ** 2 + k[:, None] ** 2 <= R * R).sum()) - 1
    data = corr(disc.astype(np.float64), w)
    return n_r * m / data, data / n_r


def _unaligned(a):
    return torch.empty(a.size + 1, device="cuda", dtype=torch.from_numpy(a).dtype)[1:].view(a.shape).copy_(torch.from_numpy(a))


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("R", [150.3, 292.0, 345.0, 590.5, 815.0, 1345.0, 1745.2, 2047.9, 2048.0])
def test_large_radii(R, dtype):
    from paper_1204_4293_gb300 import fastmap as fm
    n = 130 if R < 1000 else 67
    tol = 1e-5 if dtype == np.float32 else 1e-12
    g1, g2 = (x.astype(dtype) for x in synth.white((2, n, n), seed=int(R), scale=0.1))
    w = (np.abs(synth.white((n, n), seed=7)) + 0.1).astype(dtype)
    d = [x.astype(np.float64) for x in (g1, g2, w)]
    t = [_unaligned(x) for x in (g1, g2, w)]
    m = fm.fm_map_direct(t[0], t[1], fm.FM_FILTER_JBJ04, R, cut_over_theta=1.0)
    assert rel_err(m.cpu().numpy(), _reference(d[0], d[1], 1.0, R)) <= tol
    m, cov = fm.fm_map_direct_masked(*t, fm.FM_FILTER_JBJ04, R, cut_over_theta=1.0, coverage=True)
    mr, cr = _reference(*d, R)
    assert rel_err(m.cpu().numpy(), mr) <= tol and rel_err(cov.cpu().numpy(), cr) <= tol
