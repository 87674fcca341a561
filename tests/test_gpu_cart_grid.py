"""Stratifier training by one resident grid: shares of one to eight samples per thread, the last share short, the most a grid takes and one
more; feature values that differ in a few bits, in up to thirty (three passes of the sort) and in all of them (four); a second call finds the
counters at zero."""
import numpy as np
import pytest
import torch

from paper_2505_13254_b200 import binding as hb
from test_gpu_cart_sizes import sums_fit

pytestmark = pytest.mark.gpu

SMS = torch.cuda.get_device_properties(0).multi_processor_count if torch.cuda.is_available() else 148


def feature(kind, n, rng):
    x = rng.gamma(4.0, 2.0, n).astype(np.float32)
    if kind == "signed":                                           # both signs: all 32 bits
        return (x - 8).astype(np.float32)
    if kind == "narrow":                                           # neighbouring floats: ten bits
        return (np.float32(1.0).view(np.int32) + rng.integers(0, 1000, n)).astype(np.int32).view(np.float32)
    if kind == "pair":                                             # two values, one bit
        return np.where(rng.random(n) < 0.3, np.float32(2.0), np.nextafter(np.float32(2.0), np.float32(3.0))).astype(np.float32)
    return x


@pytest.mark.parametrize("n,depth,kind", [(8193, 3, "positive"), (8704, 3, "signed"), (SMS * 1024, 4, "positive"), (SMS * 1024 + 1, 3, "positive"),
                                          (200003, 5, "signed"), (99999, 6, "narrow"), (50000, 1, "pair"),
                                          (SMS * 2 * 4096, 3, "positive"), (SMS * 2 * 4096 + 1, 3, "positive")])
def test_thresholds_of_one_grid(n, depth, kind):
    rng = np.random.default_rng(n + depth)
    x = feature(kind, n, rng)
    y = np.clip(np.round(3.0 * np.abs(x) + rng.normal(0, 3, n)), 0, 59).astype(np.float32)
    if kind in ("narrow", "pair"):
        y = np.clip(np.round((x.view(np.int32) - x.view(np.int32).min()) * 0.05 + rng.normal(0, 3, n)), 0, 59).astype(np.float32)
    want = sums_fit(x, y, depth)
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    for _ in range(2):
        th, status = hb.hs_cart_fit(ctx, xd, yd, depth)
        torch.cuda.synchronize()
        assert int(status) == 0 and hb.hs_device_error(ctx) == 0
        # ranks are whole numbers: the sums are exact, and a threshold is the fp32 rounding of the same midpoint
        assert np.array_equal(th.cpu().numpy(), want.astype(np.float32))
    ctx.close()


def test_the_grid_in_a_graph_and_behind_other_work():
    n = 30000
    rng = np.random.default_rng(1)
    x = feature("positive", n, rng)
    y = np.clip(np.round(3.0 * x + rng.normal(0, 3, n)), 0, 59).astype(np.float32)
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    xd, yd = torch.zeros(n, device="cuda"), torch.from_numpy(y).cuda()
    hb.hs_cart_fit(ctx, torch.from_numpy(x).cuda(), yd, 3)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        th, status = hb.hs_cart_fit(ctx, xd, yd, 3)
    xd.copy_(torch.from_numpy(x))                                  # the feature is written by the kernel ahead of the replay
    graph.replay()
    torch.cuda.synchronize()
    assert int(status) == 0 and np.array_equal(th.cpu().numpy(), sums_fit(x, y, 3).astype(np.float32))
    ctx.close()
