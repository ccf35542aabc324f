"""Small maps in one kernel (a cluster of CTAs a map): bit-identical to the
separate kernels that larger batches take, for every size, depth and
boundary, and correct against the FP64 oracle; unaligned outputs and explicit
plans keep the other kernels."""
import numpy as np
import pytest
import torch

import oracle
from helpers import band_errs, rel_err

pytestmark = pytest.mark.gpu


def _fm():
    from paper_1204_4293_gb300 import fastmap
    return fastmap


def _shear(n, batch, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [0.1 * torch.randn(batch, n, n, device="cuda", generator=g) for _ in range(2)]


@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("n,J", [(64, 2), (64, 6), (128, 3), (128, 7), (256, 5), (256, 8)])
def test_small_maps_equal_the_batched_kernels(n, J, boundary):
    fm = _fm()
    most = {64: 256, 128: 48, 256: 6}[n]  # maps of one call that take the one-kernel form
    g1, g2 = _shear(n, most, n + J)
    fm.fm_tune(fm.FM_TUNE_TILE, 1)  # names a kernel: the separate ones
    try:
        ref = fm.fm_map_starlet(g1, g2, J, boundary=boundary)
        kE, kB = fm.fm_ks_invert(g1, g2, with_b=True)
        st = fm.fm_starlet_forward(kE, J, boundary=boundary)
    finally:
        fm.fm_tune(fm.FM_TUNE_TILE, -1)
    launches = fm.fm_launch_count()
    for b in (1, 3, most):
        a, c = g1[:b].contiguous(), g2[:b].contiguous()
        assert torch.equal(fm.fm_map_starlet(a, c, J, boundary=boundary), ref[:b])
        e, m = fm.fm_ks_invert(a, c, with_b=True)
        assert torch.equal(e, kE[:b]) and torch.equal(m, kB[:b])
        assert torch.equal(fm.fm_ks_invert(a, c)[0], kE[:b])
        assert torch.equal(fm.fm_starlet_forward(kE[:b].contiguous(), J, boundary=boundary), st[:b])
    assert fm.fm_launch_count() - launches == 12  # one kernel a call
    d = [x[0].double().cpu().numpy() for x in (g1, g2)]
    rE, rB = oracle.ks_invert(*d)
    assert rel_err(kE[0].cpu().numpy(), rE) <= 1e-5 and rel_err(kB[0].cpu().numpy(), rB) <= 1e-5
    assert max(band_errs(ref[0].cpu().numpy(), oracle.starlet(rE, J, boundary))) <= 1e-5


def test_small_maps_unaligned_and_captured():
    fm = _fm()
    n, J = 128, 5
    g1, g2 = _shear(n, 2, 9)
    ref = fm.fm_map_starlet(g1, g2, J)
    un = [torch.empty(2 * n * n + 1, device="cuda")[1:].view(2, n, n).copy_(x) for x in (g1, g2)]
    out = torch.empty(2 * J * n * n + 1, device="cuda")[1:].view(2, J, n, n)
    assert torch.equal(fm.fm_map_starlet(*un, J), ref)  # inputs need no alignment
    fm.fm_map_starlet(*un, J, out=out)
    assert torch.equal(out, ref)
    assert torch.equal(fm.fm_map_starlet(g1, g2, J, fuse_depth=2), ref)
    cap = torch.empty_like(ref)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        fm.fm_map_starlet(g1, g2, J, out=cap)
    g1.mul_(2.0)
    g2.mul_(2.0)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(cap, 2.0 * ref)  # a power of two scales exactly
