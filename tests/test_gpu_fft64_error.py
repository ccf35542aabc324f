"""Rounding error of the fp64 Kaiser-Squires inversion against extended
precision.  The bounds are what the complex transform with every angle rounded
in FP64 measured on these fields (64^2, 256^2): the real-output form and its
tables may not be further off."""
import numpy as np
import pytest
import torch

sf = pytest.importorskip("scipy.fft")
pytestmark = pytest.mark.gpu
if np.finfo(np.longdouble).eps > 1e-18:
    pytest.skip("no extended precision", allow_module_level=True)


def _ks_extended(g1, g2):
    L = np.longdouble
    n = g1.shape[0]
    k = np.fft.fftfreq(n, 1.0 / n).astype(L)
    k1, k2 = k[None, :], k[:, None]
    den = k1 * k1 + k2 * k2
    den[0, 0] = 1
    d = ((k1 * k1 - k2 * k2) / den - 1j * (2 * k1 * k2 / den)).astype(np.clongdouble)
    z = sf.ifft2(sf.fft2((g1.astype(L) + 1j * g2.astype(L)).astype(np.clongdouble)) * d)
    return z.real, z.imag


@pytest.mark.parametrize("n,bound", [(64, 3.78e-16), (256, 4.67e-16)])
def test_fp64_ks_error_against_extended_precision(n, bound):
    from paper_1204_4293_gb300 import fastmap as fm

    def rms(a):
        return float(np.sqrt(np.mean((a * a).astype(np.float64))))

    errs = []
    for seed in range(4):
        rng = np.random.default_rng(seed)
        g1, g2 = (rng.standard_normal((n, n)) * 0.1 for _ in range(2))
        kE, kB = _ks_extended(g1, g2)
        t = [torch.from_numpy(a).cuda()[None] for a in (g1, g2)]
        e0 = fm.fm_ks_invert(*t)[0][0].cpu().numpy()  # kappa_E alone: the real-output form
        e1, b1 = (a[0].cpu().numpy() for a in fm.fm_ks_invert(*t, with_b=True))
        errs.append([rms(e0 - kE) / rms(kE), rms(e1 - kE) / rms(kE), rms(b1 - kB) / rms(kB)])
    assert np.all(np.mean(errs, axis=0) <= bound), np.mean(errs, axis=0)
