"""The entropy pass where its geometry changes: rows around half the number of SMs (parts of a row per cluster, or a share of
the matrix per warp), rows that end in the middle of a round of 128 vectors, shares of many rounds and of several rows, more
candidates than a list holds, rows with -inf; against double-precision row statistics."""
import pytest
import torch

from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


def check(rows, vocab, dtype, make, K=10, workspace=None):
    g = torch.Generator(device="cuda").manual_seed(rows * 7 + vocab)
    ve = 8 if dtype == torch.bfloat16 else 4
    wide = torch.full((rows, (vocab + ve - 1) // ve * ve), 50.0, dtype=dtype, device="cuda")      # what lies past the vocabulary
    wide[:, :vocab] = make(torch.randn(rows, vocab, generator=g, device="cuda")).to(dtype)
    x = wide[:, :vocab]
    B = (rows + 99) // 100
    off = [min(100 * b, rows) for b in range(B + 1)]
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    parent = [-1 if r in off else 0 for r in range(rows)]
    tree = hb.TreeBatch(i32(off), i32(parent), i32([0] * rows), B, rows)
    policy = dict(thresholds=[1.0] * 7, d_base=8, alpha=4, n_default=60, top_k=K, gamma_pct=[30, 60, 100], phi_mode=0,
                  pstar_mode=0, entropy_mode=0)
    ctx = hb.Context(0, workspace or hb.hs_workspace_bytes(B, rows, vocab, 1, 1))
    for _ in range(2):                                        # (the arrival counters have reset themselves)
        q = hb.hs_entropy_quantify(ctx, tree, x, policy)
    d = x.double()
    lse = torch.logsumexp(d, 1)
    lp = d - lse[:, None]
    H = -(lp.exp() * lp.masked_fill(lp == -float("inf"), 0)).sum(1)
    key = d - 1e-11 * torch.arange(vocab, device="cuda", dtype=torch.float64) * d.abs().clamp_min(1.0)
    key = torch.where(d == -float("inf"), d, key)
    val, idx = torch.topk(key, min(K, vocab), 1)
    top = d.gather(1, idx)
    assert torch.equal(q.row_max.double(), d.max(1).values)
    assert torch.allclose(q.row_lse.double(), lse, rtol=1e-5, atol=1e-5)
    assert torch.allclose(q.h_full.double(), H, rtol=1e-4, atol=1e-5)
    got_val, got_idx = q.topk_val.double()[:, : top.shape[1]], q.topk_idx.long()[:, : top.shape[1]]
    fin = torch.isfinite(top)
    assert torch.equal(got_val[fin], top[fin]) and (got_idx[~fin] == -1).all()
    assert torch.equal(d.gather(1, got_idx.clamp_min(0))[fin], top[fin])          # the ids carry these values, each once, ties in order
    same = (top[:, 1:] == top[:, :-1]) & fin[:, 1:]
    assert (got_idx[:, 1:] > got_idx[:, :-1])[same].all()
    assert hb.hs_device_error(ctx) == 0
    ctx.close()


@pytest.mark.parametrize("rows", [1, 18, 19, 74, 75, 148, 149, 400])
@pytest.mark.parametrize("vocab,dtype", [(128256, torch.bfloat16), (32003, torch.float32), (1031, torch.bfloat16)])
def test_rows_and_vocabularies(rows, vocab, dtype):
    check(rows, vocab, dtype, lambda z: 3.0 * z)


@pytest.mark.parametrize("rows,vocab,dtype", [(600, 9, torch.bfloat16), (90, 4, torch.float32), (2000, 1024, torch.bfloat16),
                                              (80, 1000000, torch.bfloat16), (76, 8191, torch.float32)])
def test_small_and_large_rows(rows, vocab, dtype):
    check(rows, vocab, dtype, lambda z: z, K=16)


@pytest.mark.parametrize("rows", [20, 200])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
def test_ties_and_minus_infinity(rows, dtype):
    check(rows, 20000, dtype, lambda z: torch.zeros_like(z))                                       # every logit a candidate
    check(rows, 20000, dtype, lambda z: torch.where(z > 1.5, torch.full_like(z, 2.0), z))
    check(rows, 20000, dtype, lambda z: torch.where(z < 1.0, torch.full_like(z, -float("inf")), z))
    check(rows, 20000, dtype, lambda z: torch.where(z < z.topk(4, 1).values[:, 3:], torch.full_like(z, -float("inf")), z))


def test_a_small_workspace_makes_longer_shares():
    check(500, 50000, torch.bfloat16, lambda z: z, workspace=(256 << 10) + (64 << 10))
