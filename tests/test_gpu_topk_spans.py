"""Top-K over whole arrays: row counts that give a warp spans of 1, 3 and 32 rows
with a short last span, runs of rows with many equal entries (rounds of arg-max,
also for the rows behind them), one entry and more than 16, with and without
compensation terms.  Every row is exact: ids in the order of (value descending,
id ascending), coefficients the binary32 quotients by the sum in that order."""
import pytest
import torch

from test_gpu_uplift import gb  # noqa: F401

pytestmark = pytest.mark.gpu


def _expected(a, K):
    top, idx = torch.sort(a, dim=1, descending=True, stable=True)
    top, idx = top[:, :K], idx[:, :K].to(torch.int32)
    idx = torch.where(top > 0, idx, torch.full_like(idx, -1))
    top = torch.where(top > 0, top, torch.zeros_like(top))
    s = torch.zeros_like(top[:, 0])
    for k in range(K):
        s = s + top[:, k]
    return idx, torch.where(top > 0, top / s[:, None], top)


@pytest.mark.parametrize("C,K", [(20, 1), (64, 1), (64, 2), (96, 4), (200, 6), (256, 8), (33, 16), (96, 17), (1024, 3)])
@pytest.mark.parametrize("per_warp,more", [(0, 133), (3, 5), (32, 17)])
def test_every_row(gb, C, K, per_warp, more):  # noqa: F811
    n = torch.cuda.get_device_properties(0).multi_processor_count * 32 * per_warp + more
    if C == 1024 and per_warp == 32:
        n = n // 2  # spans of 16 rows
    g = torch.Generator(device="cuda").manual_seed(C + K + per_warp)
    a = torch.empty(n, C, device="cuda").exponential_(generator=g)
    a *= torch.rand(n, C, generator=g, device="cuda") < torch.rand(n, 1, generator=g, device="cuda")
    for first, count in ((40, 19), (n - 21, 14), (n - 3, 3)):  # equal entries; rows of the usual kind between and behind
        a[first:first + count] = torch.randint(-1, 3, (count, C), generator=g, device="cuda").float()
    a[n - 1, :] = 0.0
    a[n - 2, C - 1] = 7.0
    idx = torch.full((n, K), -7, dtype=torch.int32, device="cuda")
    val = torch.full((n, K), -7.0, device="cuda")
    ent = torch.empty(n, device="cuda")
    want = _expected(a, K)
    gb.scoup_topk(a, K, idx, val)
    assert torch.equal(idx, want[0]) and torch.equal(val, want[1])
    gb.scoup_topk_entropy(a, K, idx, val, ent)
    assert torch.equal(idx, want[0]) and torch.equal(val, want[1])
    p = a.double().clamp_min(0.0)
    p = p / p.sum(1, keepdim=True).clamp_min(1e-300)
    H = -torch.special.xlogy(p, p).sum(1)
    assert (ent.double() - H).abs().max() <= 1e-5
    comp = torch.randn(n, C, generator=g, device="cuda") * 2.0 ** -20
    want = _expected(a + comp, K)
    gb.scoup_topk_entropy(a, K, idx, val, ent, comp=comp)
    assert torch.equal(idx, want[0]) and torch.equal(val, want[1])
