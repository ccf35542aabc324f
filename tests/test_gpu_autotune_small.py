"""An autotuned plan describes the separate kernels: small maps that run in
one kernel keep that form with an entry in the table, whatever batch it was
tuned for, and larger batches of the shape follow the entry."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def fm():
    from paper_1204_4293_gb300 import fastmap
    fastmap.fm_autotune_clear()
    yield fastmap
    fastmap.fm_autotune_clear()


def _launches(fm, *args, **kw):
    before = fm.fm_launch_count()
    out = fm.fm_map_starlet(*args, **kw)
    return out, fm.fm_launch_count() - before


@pytest.mark.parametrize("n,J,most", [(64, 5, 256), (128, 6, 48), (256, 6, 6)])
def test_tuned_small_maps_stay_in_one_kernel(fm, n, J, most):
    g = torch.Generator(device="cuda").manual_seed(n)
    g1, g2 = (0.1 * torch.randn(most + 1, n, n, device="cuda", generator=g) for _ in range(2))
    ref, untuned = _launches(fm, g1, g2, J)
    assert untuned > 1  # above the limit: separate kernels
    for tuned_batch in (1, most + 1):
        plan = fm.fm_autotune(n, J, tuned_batch)
        assert 0 < plan["ms"] <= plan["default_ms"]
        for b in (1, most):
            out, launched = _launches(fm, g1[:b].contiguous(), g2[:b].contiguous(), J)
            assert launched == 1 and torch.equal(out, ref[:b])
            assert _launches(fm, g1[:b].contiguous(), g2[:b].contiguous(), J, fuse_depth=1)[1] > 1
    # an entry of one fused scale and two passes a scale reaches the large batch alone
    fm.fm_autotune_set(n, J, fuse_depth=1, large_path=1, tile=1, chunk_mb=0)
    assert _launches(fm, g1, g2, J)[1] > untuned and _launches(fm, g1[:1], g2[:1], J)[1] == 1
