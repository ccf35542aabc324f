"""One pass per large scale (large_path 4) on sides that are no multiple of its
512- or 256-column blocks: ragged last blocks narrower than the halo, rows
that a residue lacks, both boundaries, spacings beyond 128 px (which take the
row and column passes after it), against those passes (bit-identical) and the
FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from helpers import band_errs
from paper_1204_4293_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n,J,batch", [(32, 5, 3), (68, 6, 2), (132, 7, 2), (256, 8, 1), (260, 8, 2), (516, 8, 1), (640, 9, 2),
                                       (1000, 9, 1), (1028, 10, 1), (1500, 7, 2), (2052, 9, 1)])
def test_ragged_large_scales(n, J, batch, boundary):
    from paper_1204_4293_gb300 import fastmap as fm
    kap = np.stack([synth.grf_kappa(n, seed=n + b) + synth.white((n, n), seed=b, scale=0.05) for b in range(batch)])
    t = torch.from_numpy(kap.astype(np.float32)).cuda()
    a = fm.fm_starlet_forward(t, J, boundary=boundary, fuse_depth=2, large_path=4)
    b = fm.fm_starlet_forward(t, J, boundary=boundary, fuse_depth=2, large_path=1)
    torch.cuda.synchronize()
    assert fm.fm_device_error() == 0
    assert torch.equal(a, b)
    ref = oracle.starlet(t[-1].double().cpu().numpy(), J, boundary)
    assert max(band_errs(a[-1].cpu().numpy(), ref)) <= 1e-5


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n,J,batch", [(4, 2, 2), (8, 3, 3), (16, 4, 2), (34, 5, 2), (62, 5, 1), (66, 6, 1), (130, 7, 2), (500, 8, 1),
                                       (1024, 9, 1)])
def test_fp64_scales_in_one_pass(n, J, batch, boundary):
    # every scale from spacing 1 on, alone and after an explicit fused depth,
    # against the tile and the row and column passes (bit-identical)
    from paper_1204_4293_gb300 import fastmap as fm
    kap = np.stack([synth.grf_kappa(n, seed=n + b) + synth.white((n, n), seed=b, scale=0.05) for b in range(batch)])
    t = torch.from_numpy(kap).cuda()
    ref = fm.fm_starlet_forward(t, J, boundary=boundary, large_path=1)
    for fuse in (0, 1, 2):
        got = fm.fm_starlet_forward(t, J, boundary=boundary, fuse_depth=fuse)
        assert torch.equal(got, ref), fuse
    o = oracle.starlet(kap[-1], J, boundary)
    assert max(band_errs(ref[-1].cpu().numpy(), o)) <= 1e-12
    tiny = fm.fm_starlet_forward(t * 1e-306, J, boundary=boundary)  # the exponent shift near denormals
    want = fm.fm_starlet_forward(t * 1e-306, J, boundary=boundary, large_path=1)
    assert torch.allclose(tiny, want, rtol=0, atol=1e-320)
