"""Top-K rows at the edges of the kernel's two selections (candidates above the
K-th lane maximum, rounds of arg-max): many equal entries, few positive ones,
subnormals, negatives and huge ones, around K = 16, over row counts that end
inside a warp's span.  Ids and order are exact; the coefficients are the
binary32 quotients by the sum in that order."""
import numpy as np
import pytest

from test_gpu_uplift import gb  # noqa: F401

pytestmark = pytest.mark.gpu


def _expected(a, K):
    idx = np.full((a.shape[0], K), -1, np.int32)
    val = np.zeros((a.shape[0], K), np.float32)
    for r, row in enumerate(a):
        order = np.lexsort((np.arange(row.size), -row.astype(np.float64)))
        top = [j for j in order[:K] if row[j] > 0]
        s = np.float32(0)
        for j in top:
            s = np.float32(s + row[j])
        with np.errstate(invalid="ignore"):
            for k, j in enumerate(top):
                idx[r, k], val[r, k] = j, np.float32(row[j] / s)
    return idx, val


@pytest.mark.parametrize("C,K", [(5, 3), (32, 16), (33, 4), (64, 4), (64, 17), (128, 8), (256, 8), (256, 5),
                                 (300, 16), (1024, 8)])
@pytest.mark.parametrize("n", [1, 37, 6000])
def test_edge_rows(gb, C, K, n):  # noqa: F811
    import torch
    rng = np.random.default_rng(C + K)
    a = (rng.exponential(1.0, (n, C)) * (rng.random((n, C)) < rng.random((n, 1)))).astype(np.float32)
    special = [np.zeros(C), np.full(C, 0.5), np.where(np.arange(C) % 2, 1.0, 0.0), -np.ones(C),
               np.where(np.arange(C) < 2, 3e-39, 0.0), np.where(np.arange(C) % 7 == 0, 2.0, rng.random(C)),
               np.where(np.arange(C) == C - 1, 1e38, 1e-30)]
    for r, row in enumerate(special[:n]):
        a[r] = row
    acc = torch.as_tensor(a, device="cuda")
    idx = torch.empty((n, K), dtype=torch.int32, device="cuda")
    val = torch.empty((n, K), device="cuda")
    ent = torch.empty(n, device="cuda")
    gb.scoup_topk(acc, K, idx, val)
    want_i, want_v = _expected(a[:64], K)
    assert (idx.cpu().numpy()[:64] == want_i).all()
    assert (val.cpu().numpy()[:64] == want_v).all()
    i2, v2 = torch.empty_like(idx), torch.empty_like(val)
    gb.scoup_topk_entropy(acc, K, i2, v2, ent)
    assert torch.equal(i2, idx) and torch.equal(v2, val)
    p = a.astype(np.float64) * (a > 0)
    p = p / np.maximum(p.sum(1, keepdims=True), 1e-300)
    want = -np.where(p > 0, p * np.log(np.maximum(p, 1e-300)), 0.0).sum(1)
    assert np.abs(ent.cpu().numpy() - want).max() <= 1e-5
