"""fp64 plans run as they are named: the built-in depth and path stand for the
untuned form (one pass a scale, no tile), any other depth and path for the
tile of that depth and the path after it; results do not depend on the plan."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture
def fm():
    from paper_1204_4293_gb300 import fastmap
    fastmap.fm_autotune_clear()
    yield fastmap
    fastmap.fm_autotune_clear()


def _launches(fm, kappa, J, **kw):
    before = fm.fm_launch_count()
    out = fm.fm_starlet_forward(kappa, J, **kw)
    return out, fm.fm_launch_count() - before


@pytest.mark.parametrize("n,J", [(32, 5), (64, 5), (512, 7)])
def test_fp64_plans_run_as_named(fm, n, J):
    f64 = fm.FM_F64
    builtin_path = 4 if n >= 64 else 3
    kappa = torch.randn(2, n, n, device="cuda", dtype=torch.float64, generator=torch.Generator(device="cuda").manual_seed(n))
    ref, untuned = _launches(fm, kappa, J)
    assert untuned == J - 1  # one pass a scale
    for depth in (1, 2, 3):
        for path in (1, 3, 4):
            fm.fm_autotune_set(n, J, precision=f64, fuse_depth=depth, large_path=path, tile=1, chunk_mb=64)
            out, launched = _launches(fm, kappa, J)
            assert torch.equal(out, ref)
            if (depth, path) == (3, builtin_path):
                assert launched == untuned
            elif path == 4:
                assert launched == 1 + (J - 1 - depth)  # the tile, one pass a scale after it
            else:
                explicit, want = _launches(fm, kappa, J, fuse_depth=depth, large_path=path)
                assert launched == want and torch.equal(explicit, ref)
            assert fm.fm_starlet_fuse_depth(n, J, precision=f64) == depth
    fm.fm_autotune_clear()


@pytest.mark.parametrize("n,J", [(32, 4), (256, 6)])
def test_fp64_tuner_baseline_is_the_untuned_call(fm, n, J):
    kappa = torch.randn(1, n, n, device="cuda", dtype=torch.float64)
    untuned = _launches(fm, kappa, J)[1]
    plan = fm.fm_autotune(n, J, 1, precision=fm.FM_F64)
    launched = _launches(fm, kappa, J)[1]
    if plan["ms"] == plan["default_ms"]:  # the baseline was kept
        assert launched == untuned
    else:
        assert plan["ms"] < plan["default_ms"]
