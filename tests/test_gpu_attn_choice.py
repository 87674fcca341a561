"""Which attention kernel takes a launch follows from what the caller states (blocks, longest prefix), not from the size of the cache
arrays: a cache with room to spare gives the same bits.  Shapes on both sides of the lines (`kernel`: which one takes the launch, see
attn_route), prefixes of very different lengths with two splits among them (a split may then have nothing of a short prefix)."""
import math

import pytest
import torch

from attn_route import route
from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,hq,hkv,lens,kernel", [
    (60, 32, 8, [2048 - 103 * b for b in range(16)], 0),                   # two full waves
    (60, 32, 8, [2048 - 151 * b for b in range(10)], -1),                  # a last wave that is nearly empty
    (60, 32, 8, [1024 - 61 * b for b in range(16)], 1),                    # 16 tiles
    (60, 32, 8, [1025 - 61 * b for b in range(16)], 0),                    # 17
    (60, 32, 8, [6000 - 601 * b for b in range(10)], -1),               # a last wave that is nearly empty, longer
    (62, 64, 8, [16400, 0, 64, 9000], 2),                               # two splits, some of them empty
    (62, 64, 8, [16320, 16300, 1, 8000], 0),                            # one tile less: the other kernel, one split or more
    (62, 64, 8, [300 + 17 * b for b in range(20)], 1),                  # more than three waves
])
def test_room_in_the_cache_does_not_matter(nodes, hq, hkv, lens, kernel):
    B, G = len(lens), hq // hkv
    assert route(B, nodes, hq, hkv, max(lens)) == kernel
    g = torch.Generator(device="cuda").manual_seed(sum(lens))
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    tree = hb.TreeBatch(i32([b * nodes for b in range(B + 1)]), i32(list(range(-1, nodes - 1)) * B), i32([0] * (B * nodes)), B, B * nodes)
    policy = dict(thresholds=[-1e9] * 7, d_base=200, alpha=4, n_default=128, top_k=10, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0,
                  entropy_mode=0)
    ctx = hb.Context(0, hb.hs_workspace_bytes(B, B * nodes, 64, hq, hkv))
    hb.hs_set_prefetch(ctx, hb.HS_PREFETCH_KV)
    _, pr = hb.hs_entropy_quantify_prune(ctx, tree, torch.zeros(B * nodes, 64, device="cuda"), policy)
    rn = lambda *s: torch.randn(*s, device="cuda", generator=g, dtype=torch.bfloat16)
    q, kt, vt = rn(B * nodes, hq, 128), rn(B * nodes, hkv, 128), rn(B * nodes, hkv, 128)
    kc, vc = rn(3 * sum(lens), hkv, 128), rn(3 * sum(lens), hkv, 128)
    off = [0]
    for n in lens:
        off.append(off[-1] + n)
    outs = []
    for total in (sum(lens), 2 * sum(lens), 3 * sum(lens)):
        lse = torch.zeros(B * nodes, hq, device="cuda")
        outs.append((hb.hs_tree_verify_attention(ctx, pr, q, kt, vt, kc[:total], vc[:total], i32(off), batch=B, max_nodes=nodes,
                                                 max_kv_len=max(lens), lse_out=lse), lse))
    assert hb.hs_device_error(ctx) == 0
    for out, lse in outs[1:]:
        assert torch.equal(out, outs[0][0]) and torch.equal(lse, outs[0][1])
    tri = torch.tril(torch.ones(nodes, nodes, device="cuda")).bool()
    for b in range(B):
        r = slice(b * nodes, (b + 1) * nodes)
        K = torch.cat([kc[off[b]:off[b + 1]], kt[r]]).float().repeat_interleave(G, 1)
        V = torch.cat([vc[off[b]:off[b + 1]], vt[r]]).float().repeat_interleave(G, 1)
        s = torch.einsum("nhd,khd->hnk", q[r].float(), K) * 128 ** -0.5
        s = s.masked_fill(~torch.cat([torch.ones(nodes, lens[b], dtype=torch.bool, device="cuda"), tri], 1), -math.inf)
        ref = torch.einsum("hnk,khd->nhd", torch.softmax(s, 2), V)
        assert (outs[0][0][r].float() - ref).abs().max() < 1e-2 + 2 ** -7 * ref.abs().max()      # (bf16 P, partials and output)
        assert torch.allclose(outs[0][1][r], torch.logsumexp(s, 2).T, atol=2e-3)
    ctx.close()
