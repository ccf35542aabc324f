"""Outputs laid over the shear of a batch of small maps: in place, and a
pyramid or kappa over other maps' inputs, which must all be read first."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,batch", [(64, 5, 40), (128, 6, 9), (256, 6, 4), (256, 6, 1)])
def test_outputs_over_the_inputs(n, J, batch):
    from paper_1204_4293_gb300 import fastmap as fm
    g = torch.Generator(device="cuda").manual_seed(n)
    g1, g2 = (0.1 * torch.randn(batch, n, n, device="cuda", generator=g) for _ in range(2))
    ref = fm.fm_map_starlet(g1, g2, J)
    kE, kB = fm.fm_ks_invert(g1, g2, with_b=True)
    px = n * n
    for first in (0, px, px // 2):  # the shear at the pyramid's start, a map on, and half a map on
        buf = torch.zeros(batch * J * px + 2 * px, device="cuda")
        a = buf[first:first + batch * px].view(batch, n, n).copy_(g1)
        out = buf[:batch * J * px].view(batch, J, n, n)
        assert torch.equal(fm.fm_map_starlet(a, g2, J, out=out), ref)
    fm_lib, stream = fm.lib, torch.cuda.current_stream().cuda_stream
    for first in (0, px):  # kappa_E in place, then a map ahead of the shear; kappa_B in gamma2's place
        buf = torch.zeros((batch + 1) * px, device="cuda")
        a, b = buf[first:first + batch * px].view(batch, n, n).copy_(g1), g2.clone()
        assert fm_lib.fm_ks_invert(a.data_ptr(), b.data_ptr(), buf.data_ptr(), b.data_ptr(), n, batch, None, stream) == 0
        assert torch.equal(buf[:batch * px].view(batch, n, n), kE) and torch.equal(b, kB)
