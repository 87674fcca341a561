"""Stratifier training by one resident grid: shares of one to eight samples per thread, the last share short, the most a grid takes and one
more; feature values that differ in a few bits, in up to thirty (three passes of the sort) and in all of them (four); a second call finds the
counters at zero, also behind a wait that ran out."""
import ctypes
import os
import re

import numpy as np
import pytest
import torch

from paper_2505_13254_b200 import binding as hb
from paper_2505_13254_b200 import build
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


def arrivals(ctx, workspace):
    """Device address of the two words in which the CTAs of the training count their arrivals (the workspace pointer lies behind the device, the
    SM count and the workspace's size in the context)."""
    layout = open(os.path.join(build.CSRC, "hs_layout.h")).read()
    head = ctypes.cast(ctx.handle, ctypes.POINTER(ctypes.c_uint64))
    assert head[1] == workspace
    return head[2] + 4 * int(re.search(r"#define HS_CNT_CART (\d+)", layout).group(1))


def words(address, value=None):
    rt = pytest.importorskip("cuda.bindings.runtime")
    host = np.zeros(2, np.uint32) if value is None else np.array(value, np.uint32)
    kinds = rt.cudaMemcpyKind
    to, of, kind = (host.ctypes.data, address, kinds.cudaMemcpyDeviceToHost) if value is None else (address, host.ctypes.data, kinds.cudaMemcpyHostToDevice)
    err, = rt.cudaMemcpy(to, of, 8, kind)
    assert int(err) == 0
    return host.tolist()


@pytest.mark.parametrize("n", [9000, 60000])                       # the counts of all shares added up by every CTA, and 32 digits to a CTA
def test_a_wait_that_runs_out_is_the_status_and_leaves_nothing_behind(n):
    rng = np.random.default_rng(n)
    x = feature("positive", n, rng)
    y = np.clip(np.round(3.0 * x + rng.normal(0, 3, n)), 0, 59).astype(np.float32)
    size = hb.hs_cart_workspace_bytes(n)
    ctx = hb.Context(0, size)
    at = arrivals(ctx, size)
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    words(at, [2 ** 32 - 1, 0])                         # one arrival is missing: the first barrier's wait runs out (one second)
    _, status = hb.hs_cart_fit(ctx, xd, yd, 3)
    torch.cuda.synchronize()
    assert int(status) == hb.HS_ERR_TIMEOUT and words(at) == [0, 0]
    th, status = hb.hs_cart_fit(ctx, xd, yd, 3)                    # the error word has not been read yet
    torch.cuda.synchronize()
    assert int(status) == 0 and np.array_equal(th.cpu().numpy(), sums_fit(x, y, 3).astype(np.float32))
    assert hb.hs_device_error(ctx) == hb.HS_ERR_TIMEOUT and hb.hs_device_error(ctx) == 0
    ctx.close()


def test_two_trainings_and_decode_steps_on_streams_of_their_own():
    """Every CTA of a training holds an SM and waits for the others: what else is resident may only delay it."""
    rng = np.random.default_rng(5)
    jobs = []
    for n in (60000, SMS * 2000):
        x = feature("positive", n, rng)
        y = np.clip(np.round(3.0 * x + rng.normal(0, 3, n)), 0, 59).astype(np.float32)
        ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
        jobs.append((ctx, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), torch.cuda.Stream(), sums_fit(x, y, 3).astype(np.float32)))
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    tree = hb.TreeBatch(i32([0, 60]), i32([-1] + [0] * 59), i32([0] * 60), 1, 60)
    policy = dict(thresholds=[1.0] * 7, d_base=8, alpha=4, n_default=60, top_k=10, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0, entropy_mode=0)
    logits = torch.randn(60, 128256, device="cuda", dtype=torch.bfloat16)
    step = hb.Context(0, hb.hs_workspace_bytes(1, 60, 128256, 32, 8))
    want, _ = hb.hs_entropy_quantify_prune(step, tree, logits, policy)
    torch.cuda.synchronize()
    got = []
    for _ in range(30):
        for ctx, x, y, stream, thresholds in jobs:
            with torch.cuda.stream(stream):
                got.append((hb.hs_cart_fit(ctx, x, y, 3), thresholds))
        quant, _ = hb.hs_entropy_quantify_prune(step, tree, logits, policy)
    torch.cuda.synchronize()
    for (th, status), thresholds in got:
        assert int(status) == 0 and np.array_equal(th.cpu().numpy(), thresholds)
    assert torch.equal(quant.topk_idx, want.topk_idx) and torch.equal(quant.h_full, want.h_full)
    for ctx in [step] + [j[0] for j in jobs]:
        assert hb.hs_device_error(ctx) == 0
        ctx.close()
