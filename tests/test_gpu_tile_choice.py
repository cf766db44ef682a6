"""nm_autotune_tile compares tile widths by one measure, whether a width's plan comes from the cache or from tuning."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_a_cached_slow_plan_does_not_win(tmp_path, monkeypatch):
    """The warm launches a cached plan was reported with are shorter than any plan's cold launch: with them the width whose plan
    is cached won, here with the gather kernel on a layer the tuner has a faster one for."""
    from paper_2507_17301_b200 import nm
    path = str(tmp_path / "plans.txt")
    w = torch.randn((512, 1, 1, 512), device="cuda")
    x = torch.randn((1, 7, 7, 512), device="cuda")
    slow = nm.nm_plan_t()
    slow.variant = 1
    nm.nm_plan_cache_store(path, nm.nm_plan_key(512, 1, 1, 512, 2, 4, 128, x.shape, has_bias=False), slow)
    monkeypatch.setenv("NM_PLAN_CACHE", path)
    tile, plan, ms = nm.nm_autotune_tile(w, 2, 4, [64, 128], x)
    assert ms > 0
    assert (tile, plan.variant == 1) == (64, False)
    tile, plan, _ = nm.nm_autotune_tile(w, 2, 4, [128], x)     # the cached plan alone is still taken
    assert (tile, plan.variant) == (128, 1)
