"""FP32 rows that are rounded to bf16 chunk by chunk in the workspace (features of
at most 128 columns, codes of more than 256 atoms, gradients of a backward), over
more rows than a chunk holds.  The chunk a row falls into changes nothing: every
row equals that of a call with the row among a few hundred others, bit for bit,
and such a call is held to FP64."""
import pytest
import torch

pytestmark = pytest.mark.gpu

CHUNK = 262144  # rows


def _slices(P):
    return [slice(0, 300), slice(CHUNK - 200, CHUNK + 213), slice(P - 300, P)]


@pytest.mark.parametrize("C,D,Q,canon", [(256, 128, 32, 4), (264, 272, 16, 4), (264, 128, 16, 0)])
def test_decode_and_query(C, D, Q, canon):
    import paper_2605_13600_gb300 as gb
    P = CHUNK + 3001
    g = torch.Generator(device="cuda").manual_seed(C + D + Q)
    codes = torch.rand(P, C, generator=g, device="cuda") * (torch.rand(P, C, generator=g, device="cuda") < 0.1)
    book = torch.randn(C, D, generator=g, device="cuda")
    text = torch.randn(Q, D, generator=g, device="cuda")

    def run(rows):
        n = rows.shape[0]
        feats = torch.full((n, D), float("nan"), dtype=torch.bfloat16, device="cuda")
        n2 = torch.full((n,), -1.0, device="cuda")
        out = torch.full((n, Q - canon), float("nan"), device="cuda")
        ws = gb.scoup_decode_query(rows, book, text, out, n_canon=canon, features=feats, feat_norm2=n2)
        assert gb.scoup_read_stats(ws)["status"] == 0
        plain, p2 = torch.full_like(feats, float("nan")), torch.full_like(n2, -1.0)
        ws = gb.scoup_decode(rows, book, plain, feat_norm2=p2)
        assert gb.scoup_read_stats(ws)["status"] == 0
        f32 = torch.full((n, D), float("nan"), device="cuda")
        gb.scoup_decode(rows, book, f32)
        return feats, n2, out, plain, f32

    got = run(codes)
    assert all(torch.isfinite(x).all() for x in got)
    for rows in _slices(P):
        few = run(codes[rows].contiguous())
        for a, b in zip(got, few):
            assert torch.equal(a[rows], b)
        w, bk = codes[rows].bfloat16().double(), book.bfloat16().double()
        ref = w @ bk
        tol = 2.0 ** -22 * C * (w.abs() @ bk.abs()) + 1e-12
        assert ((few[4].double() - ref).abs() <= tol).all()
        assert ((few[0].double() - ref).abs() <= tol + 2.0 ** -8 * ref.abs()).all()
        torch.testing.assert_close(few[1].double(), few[0].double().square().sum(1), rtol=2.0 ** -23 * D, atol=0.0)


def test_decode_backward():
    import paper_2605_13600_gb300 as gb
    P, C, D = CHUNK + 3001, 64, 136
    g = torch.Generator(device="cuda").manual_seed(5)
    dF = torch.randn(P, D, generator=g, device="cuda")
    book = torch.randn(C, D, generator=g, device="cuda")
    out = torch.full((P, C), float("nan"), device="cuda")
    gb.scoup_decode_backward(dF, book, out)
    for rows in _slices(P):
        few = torch.empty((rows.stop - rows.start, C), device="cuda")
        gb.scoup_decode_backward(dF[rows].contiguous(), book, few)
        assert torch.equal(out[rows], few)
        a, b = dF[rows].bfloat16().double(), book.bfloat16().double()
        assert ((few.double() - a @ b.T).abs() <= 2.0 ** -22 * D * (a.abs() @ b.abs().T) + 1e-12).all()
