"""Stratifier training at the sizes where its kernels change: one CTA up to 8192 samples, a resident grid beyond (the same sizes through
the launches of one pass each: test_gpu_cart_partition); features with heavy ties and with a single value per layer."""
import numpy as np
import pytest
import torch

from oracle import cart as ocart
from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


def sums_fit(x, y, depth):
    """Eq. 2 by running sums in integers (ranks are whole numbers): exact, and fast enough for many samples."""
    order = np.argsort(x, kind="stable")
    xs, ys = x[order], y[order].astype(np.int64)
    sy, syy = np.concatenate(([0], np.cumsum(ys))), np.concatenate(([0], np.cumsum(ys * ys)))
    nodes, out = [(0, len(xs))], []
    for _ in range(depth):
        nxt = []
        for lo, hi in nodes:
            i = np.arange(lo + 1, hi)
            i = i[xs[i - 1] < xs[i]]
            yl, yr = sy[i] - sy[lo], sy[hi] - sy[i]
            loss = (i - lo) * (syy[i] - syy[lo]) - yl * yl + (hi - i) * (syy[hi] - syy[i]) - yr * yr
            k = int(i[np.argmin(loss)])
            out.append(0.5 * (float(xs[k - 1]) + float(xs[k])))
            nxt += [(lo, k), (k, hi)]
        nodes = nxt
    return np.sort(np.array(out))


@pytest.mark.parametrize("n,depth,levels", [(8, 1, 0), (33, 2, 0), (1023, 3, 0), (1025, 2, 40), (8192, 5, 0), (8193, 3, 0),
                                            (12288, 6, 0), (12289, 3, 300), (20480 - 1, 4, 0), (300001, 3, 0)])
def test_thresholds_at_the_edges_of_the_kernels(n, depth, levels):
    rng = np.random.default_rng(n)
    x = rng.gamma(4.0, 2.0, n).astype(np.float32)
    if n < 100:
        x = (np.arange(n) + rng.random(n) * 0.5).astype(np.float32)
    if levels:
        x = np.round(x / x.max() * levels).astype(np.float32)               # heavy ties
    y = np.clip(np.round(0.4 * x ** 1.5 + rng.normal(0, 3, n)), 0, 59).astype(np.float32)
    want = sums_fit(x, y, depth)
    if n == 1023:
        assert np.allclose(want, ocart.fit_thresholds(x, y, depth))
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    for _ in range(2):                                                        # (the second call finds the counters as the first left them)
        th, status = hb.hs_cart_fit(ctx, torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda(), depth)
        torch.cuda.synchronize()
        assert int(status) == 0
        assert np.allclose(th.cpu().numpy(), want, rtol=1e-6, atol=1e-6)
    assert hb.hs_device_error(ctx) == 0
    ctx.close()


@pytest.mark.parametrize("n", [5000, 9000])
def test_a_constant_feature_is_reported(n):
    ctx = hb.Context(0, hb.hs_cart_workspace_bytes(n))
    th, status = hb.hs_cart_fit(ctx, torch.full((n,), 2.5, device="cuda"), torch.arange(n, device="cuda", dtype=torch.float32), 3)
    torch.cuda.synchronize()
    assert int(status) == hb.HS_ERR_SHAPE and torch.isnan(th).all()
    ctx.close()
