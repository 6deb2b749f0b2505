"""The depth cut of the tile lists (chunks of views of scenes from 2^18
Gaussians on): a near layer dense enough to set every block's cut covers only
the left part of each 32 x 32 pixel block, so the tiles are still open at the
cut and the second pass (the lists behind it) carries a large share of every
result.  Uplift in its forms, both renders and the backward, which take the
whole lists, against the FP64 oracle; and the same on an image small enough
for one list per tile."""
import numpy as np
import pytest

import synth
from parity import check_accum, check_topk
from test_gpu_render import check_render
from test_gpu_render_bwd import _compare

pytestmark = pytest.mark.gpu

F, C, K = 100.0, 32, 4
SIZES = [(376, 344, 220_000, 44_000), (104, 88, 60_000, 24_000)]  # image, near and far Gaussians


@pytest.fixture(scope="module")
def gb():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_13600_gb300 import build
    build.build()
    import paper_2605_13600_gb300 as gb
    return gb


@pytest.fixture(scope="module", params=SIZES, ids=["blocks", "tiles"])
def half_covered(request):
    from conftest import axis_camera, make_scene
    W, H, NEAR, FAR = request.param
    rng = np.random.default_rng(71)
    n = NEAR + FAR
    px, py = rng.uniform(0, W, n), rng.uniform(0, H, n)
    px[:NEAR] = 32 * np.floor(px[:NEAR] / 32) + rng.uniform(0, 12, NEAR)
    z = np.concatenate([rng.uniform(1.9, 2.1, NEAR), rng.uniform(3.0, 6.0, FAR)])
    means = np.stack([(px - W / 2) * z / F, (py - H / 2) * z / F, z], axis=1)
    scales = np.exp(rng.normal(np.log(0.02), 0.3, (n, 3))) * (2.0 if W > 300 else 1.0)
    scales[NEAR:] *= 2.0
    quats = rng.normal(size=(n, 4))
    quats /= np.linalg.norm(quats, axis=1, keepdims=True)
    scene = make_scene(means, scales, quats, rng.uniform(0.3, 0.95, n))
    cams = [axis_camera(W, H, F), axis_camera(W - 7, H - 9, F), axis_camera(W, H, F, cx=W / 2 + 3.0)]
    maps, offs, rpv, R_tot = synth.scenes._pack_maps(synth.scenes._draw_seeds(rng, cams, [30] * 3), cams, "cpu")
    ci, cv = synth.region_codes(rng, R_tot, C, K)
    return synth.UpliftWorkload("half_covered", scene, cams, maps, offs, ci, cv, C, K, K, rpv)


def test_uplift_forms(gb, oracle_lib, half_covered):
    wl = half_covered
    acc, risk, cnt = oracle_lib.uplift(wl)
    counters = []
    for kw in (dict(chunked=True), dict(), dict(compensated=True)):
        up = gb.Uplift(wl, **kw)
        if not kw:
            up._chunk_views = False  # one view at a time, two pipelines
            up.workspace = up.workspace[:gb.scoup_uplift_workspace_size(up.n, up.maxw, up.maxh, up.dup_capacity)].clone()
        st = up.run(stats=True)
        info = check_accum(up.accum_value().cpu().numpy(), acc, risk)
        assert info["n_bad"] == 0, (kw, info)
        tk = check_topk(up.topk_idx.cpu().numpy(), up.topk_val.cpu().numpy(), acc, risk, wl.K)
        assert tk["n_problems"] == 0, (kw, tk)
        assert st["visible"] == cnt["visible"] and st["duplicates"] == cnt["duplicates"], (kw, st, cnt)
        assert abs(st["contributions"] - cnt["contributions"]) <= 2 * cnt["at_risk"], (kw, st, cnt)
        counters.append(st)
    assert counters[0] == counters[1]


@pytest.mark.parametrize("kernel", ["tensor", "simt"])
def test_render_and_backward(gb, oracle_lib, monkeypatch, half_covered, kernel):
    import torch
    if kernel == "simt":
        monkeypatch.setenv("SCOUP_RENDER_SIMT", "1")
    wl = half_covered
    rng = np.random.default_rng(72)
    idx, val = synth.sparse_topk_codes(rng, wl.scene.n, C, K)
    cam = wl.cams[1]
    r = gb.Render(wl.scene, idx, val, C, [cam])
    (What, T, last), st = r.run(0)
    Wo, To, risk, cnt = oracle_lib.render(wl.scene, idx, val.astype(np.float64), C, cam)
    check_render(What.cpu().numpy(), T.cpu().numpy(), Wo, To, risk)
    assert abs(st["contributions"] - cnt["contributions"]) <= 2 * risk.sum()
    if kernel == "simt":
        return
    g = rng.normal(size=(cam.height, cam.width, C)).astype(np.float32)
    g[risk] = 0.0
    d_val = torch.zeros((wl.scene.n, K), device="cuda")
    d_op = torch.zeros(wl.scene.n, device="cuda")
    gb.scoup_render_backward(r.scene, r.topk_idx, r.topk_val, K, C, cam, torch.as_tensor(g, device="cuda"), d_val, d_op,
                             r.workspace)
    dv_o, do_o = oracle_lib.render_backward(wl.scene, idx, val.astype(np.float64), C, cam, g.astype(np.float64))
    _compare(d_val.cpu().numpy(), dv_o, "d_val")
    _compare(d_op.cpu().numpy(), do_o, "d_opacity")
