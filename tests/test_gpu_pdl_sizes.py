"""Programmatic dependent launch on and off, on both sides of the grid sizes
between which a kernel lets the next one in early: bit-identical maps."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,batch,dtype", [(512, 6, 1, torch.float32), (512, 6, 9, torch.float32),
                                             (1024, 7, 1, torch.float32), (2048, 8, 1, torch.float32),
                                             (4096, 9, 1, torch.float32), (2048, 7, 1, torch.float64)])
def test_maps_do_not_depend_on_early_launches(n, J, batch, dtype):
    from paper_1204_4293_gb300 import fastmap as fm
    g = torch.Generator(device="cuda").manual_seed(n)
    g1, g2 = (0.1 * torch.randn(batch, n, n, device="cuda", dtype=dtype, generator=g) for _ in range(2))
    fm.fm_tune(fm.FM_TUNE_PDL, 0)
    try:
        ref = fm.fm_map_starlet(g1, g2, J)
    finally:
        fm.fm_tune(fm.FM_TUNE_PDL, -1)
    for _ in range(4):  # back to back
        out = fm.fm_map_starlet(g1, g2, J)
    assert torch.equal(out, ref)
