"""The decode GEMM that keeps its rows in shared memory (FP32 codes, and bf16
codes of large fused queries), at ragged row blocks, column tiles and slabs.

Features: against FP64 products of the bf16-rounded operands, with the bound of
the FP32 accumulation (2^-22 C sum |w||b|) and the output's rounding.  Norms:
against the stored rows.  Similarities: against the same rows in a small call
with bf16 codes, which takes the general kernel; the two sum a row's squared
norm in different orders, and D FP32 additions of positive terms are off by at
most D 2^-24 each side, half of that in the norm.
"""
import pytest
import torch

pytestmark = pytest.mark.gpu

CASES = [  # rows, codes, features, phrases, canonical phrases, code type
    (1, 8, 144, 16, 0, torch.float32), (129, 72, 272, 32, 4, torch.float32), (300, 128, 512, 16, 4, torch.float32),
    (19457, 64, 768, 32, 0, torch.float32), (77825, 200, 144, 16, 0, torch.float32),
    (77999, 256, 528, 32, 4, torch.float32), (155649, 136, 144, 32, 0, torch.bfloat16),
    (155905, 256, 272, 16, 4, torch.bfloat16),
]


@pytest.mark.parametrize("P,C,D,Q,canon,dtype", CASES)
def test_rows(P, C, D, Q, canon, dtype):
    import paper_2605_13600_gb300 as gb
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(P + C + D)
    codes = torch.rand(P, C, generator=g, device=dev) * (torch.rand(P, C, generator=g, device=dev) < 0.3)
    codes[0] = 0.0
    codes = codes.to(dtype)
    book = torch.randn(C, D, generator=g, device=dev)
    text = torch.randn(Q, D, generator=g, device=dev)
    text[-1] = 0.0

    def query(rows):
        n = rows.shape[0]
        feats = torch.full((n, D), float("nan"), dtype=torch.bfloat16, device=dev)
        n2 = torch.full((n,), -1.0, device=dev)
        out = torch.full((n, Q - canon), float("nan"), device=dev)
        ws = gb.scoup_decode_query(rows, book, text, out, n_canon=canon, features=feats, feat_norm2=n2)
        assert gb.scoup_read_stats(ws)["status"] == 0
        return feats, n2, out

    feats, n2, out = query(codes)
    plain = torch.full((P, D), float("nan"), device=dev)
    gb.scoup_decode(codes, book, plain)
    assert torch.isfinite(out).all() and torch.isfinite(n2).all()
    w, b = codes.bfloat16(), book.bfloat16().double()
    for at in range(0, P, 40000):
        rows = slice(at, min(P, at + 40000))
        ref = w[rows].double() @ b
        tol = 2.0 ** -22 * C * (w[rows].double().abs() @ b.abs()) + 1e-12
        assert ((plain[rows].double() - ref).abs() <= tol).all()
        assert ((feats[rows].double() - ref).abs() <= tol + 2.0 ** -8 * ref.abs()).all()
        torch.testing.assert_close(n2[rows].double(), feats[rows].double().square().sum(1), rtol=2.0 ** -23 * D, atol=0.0)
    for rows in (slice(0, 300), slice(max(0, P - 300), P)):
        f0, _, o0 = query(w[rows].contiguous())
        assert torch.equal(feats[rows], f0)
        if canon == 0:
            assert ((out[rows] - o0).abs() <= 2.0 ** -23 * D * o0.abs() + 1e-6).all()
        else:  # relevancy: the temperature (10) times the similarities' bound, on values up to 1
            assert ((out[rows] - o0).abs() <= 10 * (2.0 ** -23 * D + 1e-6) * 2).all()
