"""The region loss with its matrices or its workspace off a 16-byte boundary: the
call takes any 4-byte aligned workspace and gives the same gradients as with an
aligned one (the difference and its doubling are rounded the same in both
kernels, so they are equal bit for bit; the targets are summed by one kernel)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _shifted(t, by):
    """A copy of t that starts `by` bytes past an allocation's boundary."""
    buf = torch.empty(t.numel() * t.element_size() + 16, dtype=torch.uint8, device=t.device)
    out = buf[by:by + t.numel() * t.element_size()].view(t.dtype).view(t.shape)
    out.copy_(t)
    return out


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("F_by,dF_by,ws_by", [(0, 0, 4), (0, 0, 8), (0, 0, 12), (4, 0, 0), (0, 8, 0), (8, 4, 4)])
def test_offsets(dtype, F_by, dF_by, ws_by):
    import paper_2605_13600_gb300 as gb
    from paper_2605_13600_gb300 import _lib
    P, D, R, s, C = 301, 72, 9, 5, 40
    g = torch.Generator(device="cuda").manual_seed(ws_by + 16 * F_by + dF_by)
    F = torch.randn(P, D, generator=g, device="cuda").to(dtype)
    rmap = torch.randint(-1, R, (P,), generator=g, device="cuda", dtype=torch.int32)
    ci = torch.randint(0, C, (R, s), generator=g, device="cuda", dtype=torch.int32)
    cv = torch.rand(R, s, generator=g, device="cuda")
    book = torch.randn(C, D, generator=g, device="cuda")

    def run(F, dF, ws):
        loss = torch.zeros((), dtype=torch.float64, device="cuda")
        gb.scoup_region_l2_grad(F, rmap, ci, cv, book, dF, loss, workspace=ws)
        return dF.clone(), float(loss)

    size = int(_lib.load().scoup_region_l2_grad_workspace_size(R, D))
    want, loss = run(F, torch.empty_like(F), torch.empty(size, dtype=torch.uint8, device="cuda"))
    ws = torch.empty(size + 16, dtype=torch.uint8, device="cuda")[ws_by:ws_by + size]
    got, loss2 = run(_shifted(F, F_by), _shifted(torch.zeros_like(F), dF_by), ws)
    assert torch.equal(got, want)
    # a row's squares are summed in FP32 in another order: D 2^-24 of a sum of positive terms, each side
    assert abs(loss2 - loss) <= 2 * D * 2.0 ** -24 * loss
