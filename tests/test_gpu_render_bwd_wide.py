"""Render backward for wide code rows, at the code lengths where its two kernels
meet: 16 entries (a warp per pixel block, one CTA per SM at C = 1024) and longer
codes with their window's codes staged and not (32 and 33), against the oracle."""
import numpy as np
import pytest

from test_gpu_render_bwd import _case, _compare, gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,C", [(8, 512), (16, 1024), (17, 1024), (32, 512), (33, 513)])
def test_wide_rows(gb, oracle_lib, K, C):  # noqa: F811
    import torch
    n, W, H = 700, 43, 26
    scene, cam, idx, val, g = _case(120 + K, n, W, H, C, K, -2.4)
    _, _, risk, _ = oracle_lib.render(scene, idx, val.astype(np.float64), C, cam)
    g[risk] = 0.0
    r = gb.Render(scene, idx, val, C, [cam])
    d_val, d_op = torch.zeros((n, K), device="cuda"), torch.zeros(n, device="cuda")
    gb.scoup_render_backward(r.scene, r.topk_idx, r.topk_val, K, C, cam, torch.as_tensor(g, device="cuda"), d_val, d_op,
                             r.workspace)
    dv_o, do_o = oracle_lib.render_backward(scene, idx, val.astype(np.float64), C, cam, g.astype(np.float64))
    _compare(d_val.cpu().numpy(), dv_o, "d_val")
    _compare(d_op.cpu().numpy(), do_o, "d_opacity")
