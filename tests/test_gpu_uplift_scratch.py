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
