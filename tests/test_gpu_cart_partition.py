"""Stratifier training on a stream that belongs to a partition of the device with fewer SMs than the resident grid has CTAs: the launches of one
pass each take it, also under capture, where nothing would refuse a cooperative launch that is too large.  Their sizes: tiles of 4096 keys, the last
one full, nearly empty and short by one, one layer to six, heavy ties, a single feature value."""
import numpy as np
import pytest
import torch

from paper_2505_13254_b200 import binding as hb
from test_gpu_cart_sizes import sums_fit

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stream():
    drv = pytest.importorskip("cuda.bindings.driver")

    def call(name, *args):
        err, *out = getattr(drv, name)(*args)
        assert int(err) == 0, (name, err)
        return out[0] if len(out) == 1 else out

    torch.zeros(1, device="cuda")                                  # (the primary context)
    device = call("cuDeviceGet", torch.cuda.current_device())
    whole = call("cuDeviceGetDevResource", device, drv.CUdevResourceType.CU_DEV_RESOURCE_TYPE_SM)
    groups, _, _ = call("cuDevSmResourceSplitByCount", 1, whole, 0, 8)
    assert groups[0].sm.smCount == 8                               # (8193 samples are nine CTAs)
    part = call("cuGreenCtxCreate", call("cuDevResourceGenerateDesc", [groups[0]], 1), device,
                drv.CUgreenCtxCreate_flags.CU_GREEN_CTX_DEFAULT_STREAM)
    handle = call("cuGreenCtxStreamCreate", part, drv.CUstream_flags.CU_STREAM_NON_BLOCKING, 0)
    yield torch.cuda.ExternalStream(int(handle))
    torch.cuda.synchronize()
    call("cuStreamDestroy", handle)
    call("cuGreenCtxDestroy", part)


def pairs(n, levels=0):
    rng = np.random.default_rng(n)
    x = rng.gamma(4.0, 2.0, n).astype(np.float32)
    if levels:
        x = np.round(x / x.max() * levels).astype(np.float32)      # heavy ties
    return x, np.clip(np.round(0.4 * x ** 1.5 + rng.normal(0, 3, n)), 0, 59).astype(np.float32)


@pytest.mark.parametrize("n", [8193, 60000])
def test_a_captured_training_fits_the_partition(stream, n):
    x, y = pairs(n)
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        hb.hs_cart_fit(ctx, xd, yd, 3)
        stream.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            th, status = hb.hs_cart_fit(ctx, xd, yd, 3)
        status.fill_(-1)
        graph.replay()
    torch.cuda.synchronize()
    assert int(status) == 0 and hb.hs_device_error(ctx) == 0
    assert np.array_equal(th.cpu().numpy(), sums_fit(x, y, 3).astype(np.float32))
    ctx.close()


@pytest.mark.parametrize("n,depth,levels", [(8193, 1, 0), (12288, 6, 0), (12289, 3, 300), (16384, 5, 0), (20480 - 1, 4, 0), (300001, 3, 0)])
def test_launches_of_one_pass_each(stream, n, depth, levels):
    x, y = pairs(n, levels)
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
    torch.cuda.synchronize()
    for there in (True, False, True):                              # between them the resident grid, which finds the same words at zero
        with torch.cuda.stream(stream if there else torch.cuda.current_stream()):
            th, status = hb.hs_cart_fit(ctx, xd, yd, depth)
        torch.cuda.synchronize()
        assert int(status) == 0 and hb.hs_device_error(ctx) == 0
        assert np.array_equal(th.cpu().numpy(), sums_fit(x, y, depth).astype(np.float32))
    ctx.close()


def test_a_constant_feature_is_reported_there(stream):
    n = 9000
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    x, y = torch.full((n,), 2.5, device="cuda"), torch.arange(n, device="cuda", dtype=torch.float32)
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        th, status = hb.hs_cart_fit(ctx, x, y, 3)
    torch.cuda.synchronize()
    assert int(status) == hb.HS_ERR_SHAPE and torch.isnan(th).all() and hb.hs_device_error(ctx) == 0
    ctx.close()
