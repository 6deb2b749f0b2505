"""The alpha-threshold exponent against its definition, -log(255 o) rounded up to
binary32, over the opacities' range and beyond it: random bit patterns, and of many
more those whose exponent comes nearest to a binary32 value from either side, where
the sum of two floats decides the rounding or hands over to FP64.  Equal bit for bit
(patterns within 8 binary64 units of a binary32 value are left out: there the two
binary64 logarithms may round apart)."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _expected(o):
    t = -np.log(255.0 * o.astype(np.float64))
    th = t.astype(np.float32)
    near = np.abs(t - th.astype(np.float64)) <= 8 * np.spacing(np.abs(t))
    return np.where(th.astype(np.float64) < t, np.nextafter(th, np.float32(np.inf)), th), near, t


def _run(o):
    import paper_2605_13600_gb300 as gb
    d = torch.as_tensor(o, device="cuda")
    tau = torch.empty_like(d)
    gb.scoup_selftest_alpha_threshold(d, tau)
    return tau.cpu().numpy()


def _bits(lo, hi, n, rng):
    a, b = np.array([lo, hi], np.float32).view(np.int32)
    return rng.integers(a, b, n, dtype=np.int32).view(np.float32)


@pytest.mark.parametrize("lo,hi", [(2.0 ** -31, 32.0), (1.0 / 256, 1.0), (1e-38, 1e38)])
def test_random_and_nearest(lo, hi):
    rng = np.random.default_rng(int(hi))
    o = _bits(lo, hi, 8_000_000, rng)
    want, near, t = _expected(o)
    with np.errstate(over="ignore"):
        off = (t - t.astype(np.float32).astype(np.float64)) / np.spacing(np.abs(t).astype(np.float32)).astype(np.float64)
    pick = np.concatenate([np.argsort(np.abs(off))[:200_000], np.argsort(-np.abs(off))[:50_000],
                           rng.integers(0, o.size, 500_000)])
    pick = pick[~near[pick]]
    got = _run(o[pick])
    assert np.array_equal(got.view(np.int32), want[pick].view(np.int32)), o[pick][got != want[pick]][:5]


def test_around_the_threshold_and_outside():
    c = np.float32(1.0 / 255.0)
    o = [c]
    for _ in range(2000):
        o.append(np.nextafter(o[-1], np.float32(1)))
    down = [c]
    for _ in range(2000):
        down.append(np.nextafter(down[-1], np.float32(0)))
    o = np.array(o + down + [1.0, 0.5, 0.99, 2.0 ** -31, 32.0, 1e-30, 1e30], np.float32)
    want, near, _ = _expected(o)
    got = _run(o)
    assert np.array_equal(got[~near].view(np.int32), want[~near].view(np.int32))
    edge = _run(np.array([0.0, -0.0, -1.0, -np.inf, np.nan, np.inf], np.float32))
    assert (edge[:5] == np.inf).all() and edge[5] == -np.inf
