"""The fp64 register-resident Kaiser-Squires transforms at every size they
serve: the complex form, the real-output form (kappa_E alone), the forward
transform, unaligned outputs and the corner, Nyquist and axis modes, against
the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import rel_err, shear

pytestmark = pytest.mark.gpu


def _fm():
    from paper_1204_4293_gb300 import fastmap
    return fastmap


@pytest.mark.parametrize("n,batch", [(32, 2), (64, 3), (128, 1), (256, 2), (512, 1), (1024, 2), (2048, 1), (4096, 1)])
def test_fp64_inverse_forms_match_oracle(n, batch):
    fm = _fm()
    maps = [shear(n, seed=30 + b, dtype=np.float64) for b in range(batch)]
    g1, g2 = (torch.from_numpy(np.stack([m[k] for m in maps])).cuda() for k in (0, 1))
    kE, kB = fm.fm_ks_invert(g1, g2, with_b=True)
    kR, _ = fm.fm_ks_invert(g1, g2)
    un = torch.empty(batch * n * n + 1, dtype=torch.float64, device="cuda")[1:].view(batch, n, n)  # 8-byte aligned
    c = fm._cfg(fm.FM_F64)
    import ctypes
    assert fm.lib.fm_ks_invert(fm._ptr(g1), fm._ptr(g2), fm._ptr(un), None, n, batch, ctypes.byref(c), fm._stream()) == 0
    for b in range(batch):
        rE, rB = oracle.ks_invert(*maps[b])
        assert rel_err(kE[b].cpu().numpy(), rE) <= 1e-12 and rel_err(kB[b].cpu().numpy(), rB) <= 1e-12
        assert rel_err(kR[b].cpu().numpy(), rE) <= 1e-12
        assert rel_err(un[b].cpu().numpy(), rE) <= 1e-12


@pytest.mark.parametrize("n", [64, 512, 2048])
def test_fp64_single_modes(n):
    fm = _fm()
    y, x = np.mgrid[0:n, 0:n].astype(np.float64)
    for kx, ky in ((n // 2, 3), (5, n // 2), (n // 2, n // 2), (n // 2, 0), (0, n // 2), (0, 7), (9, 0), (17, 40)):
        ph = 2 * np.pi * (kx * x + ky * y) / n
        m = (np.cos(ph + 0.3), np.sin(2 * ph + 1.1) + 0.5 * np.cos(ph - 0.7))
        t = [torch.from_numpy(a).cuda() for a in m]
        kE, _ = fm.fm_ks_invert(*t)
        rE, _ = oracle.ks_invert(*m)
        assert np.abs(kE.cpu().numpy() - rE).max() <= 1e-12 * max(np.sqrt(np.mean(rE ** 2)), 1e-3), (kx, ky)
        f1, f2 = fm.fm_ks_forward(t[0])
        r1, r2 = oracle.ks_forward(m[0])
        assert max(np.abs(f1.cpu().numpy() - r1).max(), np.abs(f2.cpu().numpy() - r2).max()) <= 1e-12
