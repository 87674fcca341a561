"""The entropy pass with few rows: rows in two to eight parts and whole, one to sixteen keys, parts of one and several items with the row's end
inside a vector, and as many equal logits as the list of candidates holds, one warp ranks, or neither."""
import numpy as np
import pytest
import torch

from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


def check(x, k):
    """x: [rows, vocab] on the device (a view of padded rows).  Statistics against fp64, the K best exactly (ties: the lower index)."""
    n, vocab = x.shape
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    star = hb.TreeBatch(i32([0, n]), i32([-1] + [0] * (n - 1)), i32([0] * n), 1, n)
    policy = dict(thresholds=[1.0] * 7, d_base=8, alpha=4, n_default=60, top_k=k, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0, entropy_mode=0)
    ctx = hb.Context(0, hb.hs_workspace_bytes(1, n, vocab, 1, 1))
    out = hb.hs_entropy_quantify(ctx, star, x, policy)
    torch.cuda.synchronize()
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
    h = x.double().cpu().numpy()
    order = np.argsort(-h, axis=1, kind="stable")[:, :k]
    want = np.take_along_axis(h, order, 1)
    fin = want > -np.inf
    val, idx = out.topk_val.cpu().numpy().reshape(n, k), out.topk_idx.cpu().numpy().reshape(n, k)
    assert np.array_equal(val[fin], want[fin].astype(np.float32)) and np.array_equal(idx[fin], order[fin])
    assert (idx[~fin] == -1).all()
    m = h.max(1)
    e = np.exp(h - m[:, None])
    lse = m + np.log(e.sum(1))
    p = e / e.sum(1)[:, None]
    ent = lse - (p * np.where(np.isfinite(h), h, 0.0)).sum(1)
    z = np.where(fin, np.exp(want - want[:, :1]), 0.0)
    q = z / z.sum(1)[:, None]
    itk = -np.where(q > 0, q * np.log(np.where(q > 0, q, 1.0)), 0.0).sum(1)
    assert np.array_equal(out.row_max.cpu().numpy(), m.astype(np.float32))
    # 32-bit sums of exponentials with 2^-22 each; the entropies are differences of values up to |lse|
    np.testing.assert_allclose(out.row_lse.cpu().numpy(), lse, rtol=1e-5, atol=1e-5)
    np.testing.assert_allclose(out.h_full.cpu().numpy(), ent, rtol=1e-4, atol=1e-4)
    np.testing.assert_allclose(out.i_topk.cpu().numpy(), itk, rtol=1e-4, atol=1e-5)


def padded(rows, vocab, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.zeros(rows, (vocab + 7) // 8 * 8, device="cuda", dtype=dtype)[:, :vocab]
    x.copy_(torch.randn(rows, vocab, device="cuda", generator=g) * 3)
    return x


@pytest.mark.parametrize("rows", [1, 18, 21, 24, 29, 36, 49, 74])             # eight, eight, seven, six, five, four, three, two parts on 148 SMs
@pytest.mark.parametrize("vocab, dtype, k", [(128256, torch.bfloat16, 10), (32003, torch.float32, 16), (9001, torch.bfloat16, 1)])
def test_rows_in_parts(rows, vocab, dtype, k):
    check(padded(rows, vocab, dtype, rows + vocab), k)


@pytest.mark.parametrize("equal", [9, 60, 70, 400, 3000])
@pytest.mark.parametrize("rows", [2, 60])
def test_equal_logits_at_the_top(rows, equal):
    x = padded(rows, 64000, torch.bfloat16, equal)
    g = torch.Generator().manual_seed(equal)
    for r in range(rows):
        x[r, torch.randperm(64000, generator=g)[:equal].cuda()] = 20.0
    check(x, 16)


def test_fewer_finite_logits_than_keys_and_a_short_vocabulary():
    x = padded(5, 40000, torch.float32, 3)
    x[:] = -float("inf")
    x[:, 17], x[:, 39999], x[1, 20000] = 1.0, 0.5, 2.0
    check(x, 10)
    check(padded(3, 700, torch.bfloat16, 4), 16)
