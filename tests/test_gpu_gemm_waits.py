"""Bounded waits of the decode kernels: with a producer that issues no loads, every
form (general kernel and rows kernel, plain and with the query unit, bf16 and
FP32 rows) gives up, whole warps at a time, and the next call computes."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_every_form_gives_up():
    import paper_2605_13600_gb300 as gb
    from paper_2605_13600_gb300._lib import SCOUP_ERR_TIMEOUT
    before, t0 = gb.scoup_launch_count(), time.perf_counter()
    rc, msg = gb.scoup_selftest_gemm_timeout()
    assert rc == SCOUP_ERR_TIMEOUT, (rc, msg)
    assert gb.scoup_launch_count() - before == 5  # one launch in each form
    assert time.perf_counter() - t0 < 30.0
    # bf16 and FP32 rows, with and without phrases, right afterwards (powers of two: exact products and sums)
    codes = torch.zeros(300, 64, device="cuda")
    codes[:, 3], codes[:, 60] = 0.5, 0.25
    book = torch.ones(64, 144, device="cuda")
    text = torch.ones(16, 144, device="cuda")
    for rows in (codes, codes.bfloat16()):
        feats = torch.empty(300, 144, device="cuda")
        ws = gb.scoup_decode(rows, book, feats)
        assert gb.scoup_read_stats(ws)["status"] == 0 and (feats == 0.75).all()
        out = torch.empty(300, 16, device="cuda")
        ws = gb.scoup_decode_query(rows, book, text, out)
        # parallel rows: 1 up to the roundings of two norms, two quotients and a product
        assert gb.scoup_read_stats(ws)["status"] == 0 and ((out - 1.0).abs() <= 2.0 ** -20).all()
