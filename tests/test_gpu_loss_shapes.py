"""The region loss at the row lengths where its kernels split the work differently:
one lane to a row up to a whole warp, rows that end inside a step, one region to
a CTA and several, codes longer than a staged chunk, every pair of types.

Targets and differences against FP64: s products and sums of the target
(s 2^-24 of the terms' magnitudes) and the rounding of the difference; gradients
in bf16 round by 2^-8.  The loss: FP32 sums of at most 64 squares."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("types", [(torch.float32, torch.float32), (torch.float32, torch.bfloat16),
                                   (torch.bfloat16, torch.float32), (torch.bfloat16, torch.bfloat16)])
@pytest.mark.parametrize("P,D,R,s", [(1, 8, 1, 1), (33, 16, 5, 3), (1000, 24, 70, 2), (257, 56, 9, 70), (129, 64, 300, 4),
                                     (77, 136, 3, 130), (65, 136, 9, 2), (65, 200, 2, 8), (41, 512, 4, 8), (9, 776, 2, 3), (50, 12, 6, 3)])
def test_against_fp64(types, P, D, R, s):
    import paper_2605_13600_gb300 as gb
    C = 37
    g = torch.Generator(device="cuda").manual_seed(P + D)
    F = torch.randn(P, D, generator=g, device="cuda").to(types[0])
    rmap = torch.randint(-1, R, (P,), generator=g, device="cuda", dtype=torch.int32)
    ci = torch.randint(-1, C, (R, s), generator=g, device="cuda", dtype=torch.int32)
    cv = torch.rand(R, s, generator=g, device="cuda") / s
    book = torch.randn(C, D, generator=g, device="cuda")
    dF = torch.full((P, D), float("nan"), device="cuda").to(types[1])
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    ws = gb.scoup_region_l2_grad(F, rmap, ci, cv, book, dF, loss)
    assert gb.scoup_read_stats(ws)["status"] == 0
    w = torch.where(ci >= 0, cv, torch.zeros_like(cv)).double()
    rows = book.double()[ci.clamp_min(0).long()]
    tgt, mag = (w[..., None] * rows).sum(1), (w[..., None] * rows.abs()).sum(1)
    on = (rmap >= 0)[:, None]
    r = rmap.clamp_min(0).long()
    diff = torch.where(on, F.double() - tgt[r], torch.zeros((), dtype=torch.float64, device="cuda"))
    err = torch.where(on, (s + 1) * 2.0 ** -24 * mag[r] + 2.0 ** -24 * diff.abs(), torch.zeros_like(diff))
    tol = 2 * err + (2.0 ** -8 * 2 * diff.abs() if types[1] == torch.bfloat16 else 0.0)
    assert ((dF.double() - 2 * diff).abs() <= tol).all()
    want = diff.square().sum()
    bound = (2 * diff.abs() * err + err.square()).sum() + 64 * 2.0 ** -24 * want
    assert abs(float(loss) - float(want)) <= float(bound) + 1e-30
