"""Lane workspaces of a batched plan when memory is short: one view part each in
place of four, with the same counters and results.  (The device's memory is
filled up by one allocation, which is given back at the end.)"""
import numpy as np
import pytest
import torch

import synth
from test_gpu_batch import gb  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def batch():
    """Two scenes whose four-view lanes take a few hundred MB each."""
    wls = [synth.tiny_workload(400 + k, n=500_000, width=640, height=480, V=5, R=8, C=16, s=3, K=3,
                               log_scale_mean=-4.0) for k in range(2)]
    return wls


class _Filled:
    """Leaves about `leave` bytes of the device's memory free."""
    def __init__(self, leave):
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        self.hold = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")

    def __enter__(self):
        return self

    def __exit__(self, *a):
        torch.cuda.synchronize()
        self.hold = None
        torch.cuda.empty_cache()


def _run(bu):
    bu.run()
    stats = bu.stats()
    assert all(st["status"] == 0 for st in stats)
    return stats, [a.cpu().numpy() for a in bu.accum]


def _equal(got, want):
    assert got[0] == want[0]
    for a, b in zip(got[1], want[1]):  # sums of positive FP32 terms in another order
        assert np.allclose(a, b, rtol=1e-4, atol=1e-6 * b.max())


def test_lanes_shrink_to_one_view(gb, batch):  # noqa: F811
    bu = gb.BatchedUplift(batch)
    want = _run(bu)
    info = bu.info()
    four = info["workspace_bytes"] // info["lanes"]
    assert four > 200 << 20
    # room for the lanes that it has and one more, but not for eight
    with _Filled(four + four // 2):
        bu.set(8, 8)
        small = bu.info()
        assert small["lanes"] == 8 and small["workspace_bytes"] // 8 < four // 2
        _equal(_run(bu), want)
        bu.close()
    # at creation: four views a lane fit, but not into an eighth of what is free
    with _Filled(6 * four):
        bu = gb.BatchedUplift(batch)
        assert bu.info()["workspace_bytes"] // bu.info()["lanes"] == small["workspace_bytes"] // 8
        _equal(_run(bu), want)
        bu.close()
