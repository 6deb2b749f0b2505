"""Windows cut out of a depth bucket that holds more than one window, in lists of
blocks of tiles (key words with tile bits) and of single tiles: many equal depths,
many neighbouring ones inside a bucket, and a far Gaussian that makes the buckets
wide.  Uplift in its forms, renders and backward against the FP64 oracle."""
import numpy as np
import pytest

import synth
from conftest import axis_camera, make_scene
from parity import check_accum, check_topk
from test_gpu_render import check_render
from test_gpu_render_bwd import _compare
from test_gpu_uplift import gb  # noqa: F401

pytestmark = pytest.mark.gpu

C, K = 32, 4


@pytest.fixture(scope="module", params=[(64, 48), (83, 79)], ids=["tiles", "blocks"])
def sheets(request):
    W, H = request.param
    rng = np.random.default_rng(91)
    n = 2400
    z = np.full(n, 3.0, np.float32)
    z[800:1600] = np.float32(3.0) + rng.integers(1, 40, 800).astype(np.float32) * np.float32(2.0 ** -22)
    z[1600:] = rng.uniform(3.0, 3.01, 800)
    z[-1] = 3000.0
    z = z[rng.permutation(n)]
    means = np.stack([rng.uniform(-0.7, 0.7, n) * z, rng.uniform(-0.7, 0.7, n) * z, z], axis=1)
    quats = rng.normal(size=(n, 4))
    quats /= np.linalg.norm(quats, axis=1, keepdims=True)
    scene = make_scene(means, np.full((n, 3), 0.06), quats, rng.uniform(0.02, 0.08, n))
    cams = [axis_camera(W, H, 50.0), axis_camera(W, H, 45.0)]
    maps, offs, rpv, R = synth.scenes._pack_maps(synth.scenes._draw_seeds(rng, cams, [5, 12]), cams, "cpu")
    ci, cv = synth.region_codes(rng, R, C, K)
    return synth.UpliftWorkload("sheets", scene, cams, maps, offs, ci, cv, C, K, K, rpv)


def test_uplift(gb, oracle_lib, sheets):  # noqa: F811
    acc, risk, cnt = oracle_lib.uplift(sheets)
    for kw in (dict(chunked=True), dict(compensated=True)):
        up = gb.Uplift(sheets, **kw)
        st = up.run()
        assert st["status"] == 0 and st["split_windows"] > 0, st
        info = check_accum(up.accum_value().cpu().numpy(), acc, risk)
        assert info["n_bad"] == 0, (kw, info)
        tk = check_topk(up.topk_idx.cpu().numpy(), up.topk_val.cpu().numpy(), acc, risk, K)
        assert tk["n_problems"] == 0, (kw, tk)
        assert abs(st["contributions"] - cnt["contributions"]) <= 2 * cnt["at_risk"]


@pytest.mark.parametrize("kernel", ["tensor", "simt"])
def test_render(gb, oracle_lib, monkeypatch, sheets, kernel):  # noqa: F811
    if kernel == "simt":
        monkeypatch.setenv("SCOUP_RENDER_SIMT", "1")
    rng = np.random.default_rng(92)
    idx, val = synth.sparse_topk_codes(rng, sheets.scene.n, C, K)
    cam = sheets.cams[0]
    (What, T, _), st = gb.Render(sheets.scene, idx, val, C, [cam]).run(0)
    Wo, To, risk, _ = oracle_lib.render(sheets.scene, idx, val.astype(np.float64), C, cam)
    check_render(What.cpu().numpy(), T.cpu().numpy(), Wo, To, risk)
    assert st["split_windows"] > 0, st


@pytest.mark.parametrize("k", [4, 17])
def test_backward(gb, oracle_lib, sheets, k):  # noqa: F811
    import torch
    rng = np.random.default_rng(93)
    idx, val = synth.sparse_topk_codes(rng, sheets.scene.n, C, k)
    cam, n = sheets.cams[0], sheets.scene.n
    g = rng.normal(size=(cam.height, cam.width, C)).astype(np.float32)
    _, _, risk, _ = oracle_lib.render(sheets.scene, idx, val.astype(np.float64), C, cam)
    g[risk] = 0.0
    r = gb.Render(sheets.scene, idx, val, C, [cam])
    d_val, d_op = torch.zeros((n, k), device="cuda"), torch.zeros(n, device="cuda")
    gb.scoup_render_backward(r.scene, r.topk_idx, r.topk_val, k, C, cam, torch.as_tensor(g, device="cuda"), d_val, d_op,
                             r.workspace)
    dv_o, do_o = oracle_lib.render_backward(sheets.scene, idx, val.astype(np.float64), C, cam, g.astype(np.float64))
    _compare(d_val.cpu().numpy(), dv_o, "d_val")
    _compare(d_op.cpu().numpy(), do_o, "d_opacity")
