"""Tree attention in launches of more query blocks than SMs, and of fewer with long prefixes, where two CTAs share an SM: prefixes around the edges of a key tile and
none at all, trees of 1 to 128 nodes (one or two tree tiles, dead query blocks), grouped heads that do not divide a block, split
prefixes, both row layouts and both cache layouts; against fp32 attention.  (`kernel`: see attn_route; the launches of the other kernel's instance
that stands for this one are among them.)"""
import math
import random

import pytest
import torch

from attn_route import route
from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,nodes,hq,hkv,kv,layout,head_first,prefetch,kernel", [
    (40, (1, 128), 32, 8, [0, 1, 63, 64, 65, 127, 128, 129, 191, 192, 193, 320], hb.HS_ROWS_COMPACT, False, True, 1),
    (40, (30, 128), 21, 3, [0, 7, 64, 200, 700], hb.HS_ROWS_ORIGINAL, True, False, 1),
    (12, (60, 128), 64, 4, [2500, 64, 3000, 1], hb.HS_ROWS_COMPACT, True, True, 1),
    (10, (40, 60), 32, 8, [4096, 4097, 130], hb.HS_ROWS_ORIGINAL, False, True, -1),
    (10, (40, 60), 32, 8, [1500, 1, 640], hb.HS_ROWS_COMPACT, True, False, -1),
    (10, (40, 60), 32, 8, [512, 449, 130], hb.HS_ROWS_ORIGINAL, False, True, 1),
    (4, (50, 62), 64, 8, [16500, 70, 0, 12000], hb.HS_ROWS_ORIGINAL, False, False, 2),
    (4, (50, 62), 64, 8, [100, 16385, 8200, 64], hb.HS_ROWS_COMPACT, True, True, 2),
    (8, (33, 60), 32, 8, [16400, 8256, 63, 16321], hb.HS_ROWS_ORIGINAL, True, True, 2),
])
def test_two_ctas_per_sm(batch, nodes, hq, hkv, kv, layout, head_first, prefetch, kernel):
    rng = random.Random(batch + hq)
    g = torch.Generator(device="cuda").manual_seed(hq)
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    ns = [nodes[0] if b == 0 else nodes[1] if b == 1 else rng.randint(*nodes) for b in range(batch)]
    off, kvo, parent = [0], [0], []
    for b, n in enumerate(ns):
        off.append(off[-1] + n)
        kvo.append(kvo[-1] + kv[b % len(kv)])
        parent += [-1] + [rng.randint(max(0, i - 12), i - 1) for i in range(1, n)]
    assert route(batch, max(ns), hq, hkv, max(kv)) == kernel
    N, T, G = off[-1], kvo[-1], hq // hkv
    tree = hb.TreeBatch(i32(off), i32(parent), i32([rng.randrange(64) for _ in range(N)]), batch, N)
    policy = dict(thresholds=[-1e9] * 7, d_base=100, alpha=4, n_default=128, top_k=10, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0,
                  entropy_mode=0)
    ctx = hb.Context(0, hb.hs_workspace_bytes(batch, N, 64, hq, hkv))
    hb.hs_set_prefetch(ctx, 2 if prefetch else 0)
    _, pr = hb.hs_entropy_quantify_prune(ctx, tree, torch.randn(N, 64, device="cuda", generator=g), policy)
    rn = lambda *s: torch.randn(*s, device="cuda", generator=g, dtype=torch.bfloat16)
    q, kt, vt = rn(N, hq, 128), rn(N, hkv, 128), rn(N, hkv, 128)
    kc, vc = [rn(hkv, T, 128).permute(1, 0, 2) if head_first else rn(T, hkv, 128) for _ in range(2)]
    outs = []
    for _ in range(2):
        out, lse = torch.zeros_like(q), torch.zeros(N, hq, device="cuda")
        hb.hs_tree_verify_attention(ctx, pr, q, kt, vt, kc, vc, i32(kvo), batch=batch, max_nodes=max(ns), max_kv_len=max(kv), layout=layout,
                                    node_off=tree.node_off, out=out, lse_out=lse)
        outs.append(out)
    assert torch.equal(outs[0], outs[1]) and hb.hs_device_error(ctx) == 0
    keep_off, n_keep = pr.keep_off.tolist(), pr.n_keep.tolist()
    for b in range(batch):
        n, k0 = n_keep[b], keep_off[b]
        rows = (off[b] + pr.keep_idx[k0:k0 + n].long()) if layout == hb.HS_ROWS_ORIGINAL else torch.arange(k0, k0 + n, device="cuda")
        m = pr.anc_mask[k0:k0 + n]
        bits = torch.stack([((m[:, j // 64] >> (j % 64)) & 1).bool() for j in range(n)], 1)
        L = kvo[b + 1] - kvo[b]
        mask = torch.cat([torch.ones(n, L, dtype=torch.bool, device="cuda"), bits], 1)
        K = torch.cat([kc[kvo[b]:kvo[b + 1]], kt[rows]]).float().repeat_interleave(G, 1)
        V = torch.cat([vc[kvo[b]:kvo[b + 1]], vt[rows]]).float().repeat_interleave(G, 1)
        s = torch.einsum("nhd,khd->hnk", q[rows].float(), K) * 128 ** -0.5
        s = s.masked_fill(~mask, -math.inf)
        ref = torch.einsum("hnk,khd->nhd", torch.softmax(s, 2), V)
        # (bf16 P, partials and output: 2^-8 of the size of the values, which a row with one visible key hands through)
        assert (outs[0][rows].float() - ref).abs().max() < 1e-2 + 2 ** -7 * ref.abs().max()
        assert torch.allclose(lse[rows], torch.logsumexp(s, 2).T, atol=2e-3)
    ctx.close()
