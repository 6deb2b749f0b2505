"""Scratch memory of the wrappers' default form: what ran with a small workspace
runs on, and nothing larger is held than a call uses."""
import numpy as np
import pytest

import synth
from conftest import axis_camera, make_scene, single_region_workload
from test_gpu_uplift import gb  # noqa: F401

pytestmark = pytest.mark.gpu


def test_no_capacity_for_views_that_list_nothing(gb):  # noqa: F811
    """dup_capacity = 0 is enough for a scene behind its cameras, whatever the number of views."""
    rng = np.random.default_rng(5)
    means = np.stack([rng.normal(size=50), rng.normal(size=50), -1.0 - rng.random(50)], axis=1)
    scene = make_scene(means, np.full((50, 3), 0.1), np.tile([1.0, 0.0, 0.0, 0.0], (50, 1)), np.full(50, 0.5))
    for V in (1, 2, 9):
        wl = single_region_workload(scene, [axis_camera(70, 50)] * V, 8, [(0, 1.0)], 1)
        up = gb.Uplift(wl, dup_capacity=0)
        st = up.run()
        assert st["status"] == 0 and st["visible"] == 0 and st["contributions"] == 0
        assert not up.accum.any() and (up.topk_idx == -1).all()


def test_levels_hold_no_view_parts_of_chunks(gb):  # noqa: F811
    """scoup_uplift_levels runs one view at a time: its workspace is that form's."""
    base = synth.tiny_workload(3, n=2000, V=4)
    up = gb.LevelUplift(synth.level_workloads(base, (2, 4, 8)))
    b = up.base
    assert b.workspace.numel() == gb.scoup_uplift_workspace_size(b.n, b.maxw, b.maxh, b.dup_capacity)
    assert up.run()["status"] == 0


@pytest.fixture(scope="module")
def several_views():
    from paper_2605_13600_gb300 import scoup
    wl = synth.uplift_cfg1()
    up = scoup.Uplift(wl)
    assert up._chunk_views
    return wl, up.run(), up.accum.clone()


def gb_size(up):
    from paper_2605_13600_gb300 import scoup
    return scoup.scoup_uplift_workspace_size(up.n, up.maxw, up.maxh, up.dup_capacity)


def _same(up, want):
    _, stats, accum = want
    assert not up._chunk_views
    assert up.workspace.numel() == gb_size(up)
    st = up.run()
    assert st == stats
    # sums of positive FP32 terms in another order
    assert np.allclose(up.accum.cpu().numpy(), accum.cpu().numpy(), rtol=1e-4, atol=1e-6 * float(accum.max()))


def test_small_form_where_memory_is_short(gb, several_views, monkeypatch):  # noqa: F811
    """Little free memory on the device: the form with two view parts, same counters and sums."""
    import torch
    wl = several_views[0]
    free, total = torch.cuda.mem_get_info()
    spare = torch.cuda.memory_reserved() - torch.cuda.memory_allocated()
    need = gb.scoup_uplift_chunked_workspace_size(wl.scene.n, 160, 120, 0)
    monkeypatch.setattr(torch.cuda, "mem_get_info", lambda device=None: (4 * need - spare, total))
    _same(gb.Uplift(wl), several_views)


def test_small_form_where_the_allocation_fails(gb, several_views):  # noqa: F811
    """The chunked workspace does not fit the process's memory limit, the other one does; asked for, it is an error."""
    import torch
    wl, dup = several_views[0], 10_000_000
    small = gb.scoup_uplift_workspace_size(wl.scene.n, 160, 120, dup)
    large = gb.scoup_uplift_chunked_workspace_size(wl.scene.n, 160, 120, dup)
    assert large - small > 1 << 30
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    limit = torch.cuda.memory_reserved() + small + (1 << 29)  # the scene, its maps and accumulator are a few MB
    torch.cuda.set_per_process_memory_fraction(limit / torch.cuda.get_device_properties(0).total_memory)
    try:
        _same(gb.Uplift(wl, dup_capacity=dup), several_views)
        with pytest.raises(torch.cuda.OutOfMemoryError):
            gb.Uplift(wl, dup_capacity=dup, chunked=True)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
