"""One recorded noise graph serves every buffer and seed of a shape: calls
with other inputs, seeds and streams, issued back to back, give what eager
launches give, and so do batched maps whose buffers change or come back."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _fm():
    from paper_1204_4293_gb300 import fastmap
    return fastmap


def _shear(n, seed, lead=()):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return [0.1 * torch.randn(lead + (n, n), device="cuda", generator=g) for _ in range(2)]


@pytest.mark.parametrize("n,J,R,dtype", [(64, 4, 40, torch.float32), (512, 5, 70, torch.float32), (16, 3, 5, torch.float64)])
def test_noise_graph_serves_other_buffers_seeds_and_streams(n, J, R, dtype):
    fm = _fm()
    ins = [[a.to(dtype) for a in _shear(n, s)] for s in range(3)]
    ins.append([torch.empty(n * n + 1, device="cuda", dtype=dtype)[1:].view(n, n).copy_(a) for a in ins[0]])  # unaligned
    fm.fm_tune(fm.FM_TUNE_GRAPHS, 0)
    try:
        ref = [fm.fm_map_noise(*g, J, R, seed=100 + k) for k, g in enumerate(ins)]
    finally:
        fm.fm_tune(fm.FM_TUNE_GRAPHS, -1)
    streams = [torch.cuda.Stream() for _ in range(2)]
    torch.cuda.synchronize()
    got = []
    for k, g in enumerate(ins):  # no synchronisation between calls on alternating streams
        with torch.cuda.stream(streams[k % 2]):
            got.append(fm.fm_map_noise(*g, J, R, seed=100 + k))
    torch.cuda.synchronize()
    for (v, s), (rv, rs) in zip(got, ref):
        assert torch.equal(v, rv) and torch.equal(s, rs)
    fm.fm_trim()


def test_batched_maps_with_new_and_returning_buffers():
    fm = _fm()
    g1, g2 = _shear(256, 5, (6,))
    fm.fm_tune(fm.FM_TUNE_CHUNK_BYTES, 2 << 20)  # several chunks
    try:
        out = torch.empty((6, 5, 256, 256), device="cuda")
        ref = fm.fm_map_starlet(g1, g2, 5)
        for k in range(8):
            assert torch.equal(fm.fm_map_starlet(g1, g2, 5, out=out.zero_()), ref)  # launched, recorded, replayed
            assert torch.equal(fm.fm_map_starlet(g1.clone(), g2.clone(), 5), ref)
    finally:
        fm.fm_tune(fm.FM_TUNE_CHUNK_BYTES, -1)
    fm.fm_trim()
