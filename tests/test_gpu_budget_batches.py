"""The token budget over batches around the size up to which one launch does request, reallocation and pruning (a thread per
sequence): kept nodes against the oracle's reallocation of the policy's own requests, flagged sequences among them."""
import numpy as np
import pytest
import torch

from oracle import budget as obudget
from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch", [1, 2, 15, 17, 127, 128, 129, 200])
def test_budget_over_batches(batch):
    rng = np.random.default_rng(batch)
    sizes = rng.integers(1, 61, batch)
    sizes[0] = 128
    off = np.concatenate([[0], np.cumsum(sizes)])
    parent = np.concatenate([[-1] + [int(rng.integers(max(0, i - 6), i)) for i in range(1, n)] for n in sizes])
    bad = batch // 3 if batch > 2 else -1
    if bad >= 0:
        parent[off[bad]] = 0                                # a root that is its own parent: the sequence is flagged
    N = int(off[-1])
    i32 = lambda a: torch.tensor(np.asarray(a), dtype=torch.int32, device="cuda")
    tree = hb.TreeBatch(i32(off), i32(parent), i32(rng.integers(0, 64, N)), batch, N)
    policy = dict(thresholds=[float(t) for t in np.linspace(0.5, 6.0, 7)], d_base=6, alpha=4, n_default=24, top_k=10, gamma_pct=[30, 60, 100],
                  phi_mode=0, pstar_mode=0, entropy_mode=0)
    ctx = hb.Context(0, hb.hs_workspace_bytes(batch, N, 64, 1, 1))
    g = torch.Generator(device="cuda").manual_seed(batch)
    quant = hb.hs_entropy_quantify(ctx, tree, 3 * torch.randn(N, 64, device="cuda", generator=g), policy)
    plain = hb.hs_stratify_prune(ctx, tree, quant, policy)
    status = quant.status.cpu().numpy()
    assert (status != 0).nonzero()[0].tolist() == ([bad] if bad >= 0 else [])
    good = [b for b in range(batch) if status[b] == 0]
    depth, score = quant.depth.cpu().numpy(), quant.score.cpu().numpy()
    d_prime, n_prime = plain.d_prime.tolist(), plain.n_prime.tolist()
    elig = [[i for i in range(sizes[b]) if depth[off[b] + i] <= d_prime[b]] for b in range(batch)]
    slo = rng.integers(0, 3, batch)
    base = sum(min(n_prime[b], len(elig[b])) for b in good)
    for budget in (base + 11 * batch, base, max(1, base - 5 * batch), 3):
        want = [0] * batch
        for b, n in zip(good, obudget.reallocate([n_prime[b] for b in good], [len(elig[b]) for b in good], slo[good].tolist(), budget)):
            want[b] = n
        pr = hb.hs_stratify_prune_budget(ctx, tree, quant, policy, i32(slo), budget)
        assert pr.n_keep.tolist() == want
        assert pr.keep_off.tolist() == np.concatenate([[0], np.cumsum(want)]).tolist()
        keep_idx = pr.keep_idx.tolist()
        for b in good:
            S = score[off[b]:off[b + 1]]
            best = sorted(sorted(elig[b], key=lambda i: (-S[i], i))[:want[b]])
            k0 = sum(want[:b])
            assert keep_idx[k0:k0 + want[b]] == best
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
