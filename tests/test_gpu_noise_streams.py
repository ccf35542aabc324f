"""Noise calls of one small shape that keep overlapping on two streams run on a
graph and scratch each; results are those of calls one after the other, and
larger shapes share one."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,J,R,graphs", [(64, 4, 400, 2), (256, 6, 100, 2), (512, 5, 60, 1)])
def test_overlapping_noise_calls(n, J, R, graphs):
    from paper_1204_4293_gb300 import fastmap as fm
    g = torch.Generator(device="cuda").manual_seed(n)
    ins = [[0.1 * torch.randn(n, n, device="cuda", generator=g) for _ in range(2)] for _ in range(2)]
    fm.fm_trim()
    ref = [fm.fm_map_noise(*ins[k], J, R, seed=k) for k in range(2)]
    fm.fm_trim()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in range(2)]
    fm.fm_alloc_stats(reset=True)
    got = []
    for k in range(12):  # no synchronisation
        with torch.cuda.stream(streams[k % 2]):
            got.append(fm.fm_map_noise(*ins[k % 2], J, R, seed=k % 2))
    torch.cuda.synchronize()
    assert fm.fm_alloc_stats()[0] == graphs
    for k, (v, s) in enumerate(got):
        assert torch.equal(v, ref[k % 2][0]) and torch.equal(s, ref[k % 2][1])
    fm.fm_trim()
