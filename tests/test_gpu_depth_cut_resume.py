"""The second pass behind the depth cut, counted.  A near layer of at least twice
the optical depth of a cut in every block of 2 x 2 tiles, the blocks at the image's
edges included, lies over the left 12 of a block's 32 columns: the cut falls into
it, the block's right tiles are open there, and all that they hold is found by the
second pass."""
import numpy as np
import pytest

import synth
from conftest import axis_camera, make_scene
from parity import check_accum, check_topk
from test_gpu_uplift import gb  # noqa: F401

pytestmark = pytest.mark.gpu

F, C, K = 100.0, 32, 4
W, H, NEAR, FAR = 376, 344, 240_000, 30_000
CUT_OPTICAL = 42.0  # kCutOptical of the library


@pytest.fixture(scope="module")
def covered():
    rng = np.random.default_rng(73)
    n = NEAR + FAR
    px, py = rng.uniform(0, W, n), rng.uniform(0, H, n)
    px[:NEAR] = 32 * np.floor(px[:NEAR] / 32) + rng.uniform(0, 12, NEAR)
    z = np.concatenate([rng.uniform(1.9, 2.1, NEAR), rng.uniform(3.0, 6.0, FAR)])
    means = np.stack([(px - W / 2) * z / F, (py - H / 2) * z / F, z], axis=1)
    scales = np.exp(rng.normal(np.log(0.048), 0.2, (n, 3)))
    scales[NEAR:] *= 2.0
    quats = rng.normal(size=(n, 4))
    quats /= np.linalg.norm(quats, axis=1, keepdims=True)
    o = rng.uniform(0.9, 0.99, n)
    o[NEAR:] = rng.uniform(0.3, 0.95, FAR)
    # what the near layer puts into each block: 2 pi sigma^2 Li2(o) pixels of optical depth (Li2 about o + 0.645 o^3)
    s = scales[:NEAR]
    area = (s[:, 0] * s[:, 1] + s[:, 1] * s[:, 2] + s[:, 0] * s[:, 2]) / 3.0
    mass = 2 * np.pi * (area * (F / z[:NEAR]) ** 2 + 0.3) * (o[:NEAR] + 0.645 * o[:NEAR] ** 3)
    bw = (W + 31) // 32
    block = (py[:NEAR] // 32).astype(int) * bw + (px[:NEAR] // 32).astype(int)
    depth = np.bincount(block, mass) / 1024.0
    assert depth.min() > CUT_OPTICAL and np.median(depth) > 2 * CUT_OPTICAL, (depth.min(), np.median(depth))
    scene = make_scene(means, scales, quats, o)
    cams = [axis_camera(W, H, F), axis_camera(W, H, F, cx=W / 2 - 2.0), axis_camera(W, H, F, cx=W / 2 + 2.0)]
    maps, offs, rpv, R = synth.scenes._pack_maps(synth.scenes._draw_seeds(rng, cams, [30] * 3), cams, "cpu")
    ci, cv = synth.region_codes(rng, R, C, K)
    return synth.UpliftWorkload("covered", scene, cams, maps, offs, ci, cv, C, K, K, rpv)


def test_second_pass(gb, oracle_lib, covered):  # noqa: F811
    acc, risk, cnt = oracle_lib.uplift(covered)
    tiles = ((W + 15) // 16) * ((H + 15) // 16) * len(covered.cams)
    for kw in (dict(chunked=True), dict(), dict(compensated=True), dict(views=True)):
        one = kw.pop("views", False)
        up = gb.Uplift(covered, **kw)
        if one:
            up._chunk_views = False  # one view at a time: whole lists
            up.workspace = up.workspace[:gb.scoup_uplift_workspace_size(up.n, up.maxw, up.maxh, up.dup_capacity)].clone()
        st = up.run()
        resumed = gb.scoup_selftest_resumed_tiles(up.workspace)
        if one:
            assert resumed == 0
        else:
            assert 0.45 * tiles <= resumed <= tiles, (resumed, tiles)
        assert st["status"] == 0
        info = check_accum(up.accum_value().cpu().numpy(), acc, risk)
        assert info["n_bad"] == 0, (kw, info)
        tk = check_topk(up.topk_idx.cpu().numpy(), up.topk_val.cpu().numpy(), acc, risk, K)
        assert tk["n_problems"] == 0, (kw, tk)
        assert st["visible"] == cnt["visible"] and st["duplicates"] == cnt["duplicates"]
        assert abs(st["contributions"] - cnt["contributions"]) <= 2 * cnt["at_risk"]
