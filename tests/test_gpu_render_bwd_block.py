"""Render backward at the edges of its two kernels (codes of up to 16 entries
and longer ones): code lengths around 4, 8 and 16, rows whose width is not a
multiple of four words, padding entries, ragged images, against the oracle."""
import numpy as np
import pytest

import synth
from test_gpu_render_bwd import _case, _compare, gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,C,W,H,n", [
    (1, 8, 17, 9, 200),
    (4, 21, 40, 33, 600),
    (5, 64, 33, 30, 500),
    (8, 256, 48, 35, 900),
    (9, 30, 31, 47, 500),
    (16, 513, 24, 20, 300),
    (17, 40, 24, 20, 300),
])
def test_code_lengths_and_row_widths(gb, oracle_lib, K, C, W, H, n):  # noqa: F811
    import torch
    scene, cam, idx, val, g = _case(80 + K, n, W, H, C, K, -2.4)
    rng = np.random.default_rng(K)
    pad = rng.random(idx.shape) < 0.2  # padding entries anywhere in a code
    idx = np.where(pad, -1, idx).astype(np.int32)
    _, _, risk, _ = oracle_lib.render(scene, idx, val.astype(np.float64), C, cam)
    g[risk] = 0.0
    r = gb.Render(scene, idx, val, C, [cam])
    d_val = torch.zeros((n, K), device="cuda")
    d_op = torch.zeros(n, device="cuda")
    gd = torch.as_tensor(g, device="cuda")
    gb.scoup_render_backward(r.scene, r.topk_idx, r.topk_val, K, C, cam, gd, d_val, d_op, r.workspace)
    dv_o, do_o = oracle_lib.render_backward(scene, idx, val.astype(np.float64), C, cam, g.astype(np.float64))
    _compare(d_val.cpu().numpy(), dv_o, "d_val")
    _compare(d_op.cpu().numpy(), do_o, "d_opacity")
    assert (d_val.cpu().numpy()[pad] == 0.0).all()


def test_gradient_rows_off_16_bytes(gb, oracle_lib):  # noqa: F811
    """A gradient that starts 4 bytes past a 16-byte boundary takes word copies."""
    import torch
    scene, cam, idx, val, g = _case(99, 400, 30, 20, 32, 4, -2.4)
    _, _, risk, _ = oracle_lib.render(scene, idx, val.astype(np.float64), 32, cam)
    g[risk] = 0.0
    r = gb.Render(scene, idx, val, 32, [cam])
    buf = torch.empty(g.size + 1, device="cuda")
    gd = buf[1:].view(g.shape)
    gd.copy_(torch.as_tensor(g))
    d_val, d_op = torch.zeros((400, 4), device="cuda"), torch.zeros(400, device="cuda")
    gb.scoup_render_backward(r.scene, r.topk_idx, r.topk_val, 4, 32, cam, gd, d_val, d_op, r.workspace)
    dv_o, do_o = oracle_lib.render_backward(scene, idx, val.astype(np.float64), 32, cam, g.astype(np.float64))
    _compare(d_val.cpu().numpy(), dv_o, "d_val")
    _compare(d_op.cpu().numpy(), do_o, "d_opacity")
