"""Rows by drafted node id may lie anywhere in the batch's rows: behind a sequence that is too large (flagged and skipped) they lie past
both max_rows, which bounds the kept ones, and 128 rows per sequence.  Both attention kernels read them all the same."""
import pytest
import torch

from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,big,kv", [(3, 700, 900), (24, 3000, 900)])
def test_rows_behind_an_oversized_sequence(batch, big, kv):
    nodes, hq, hkv = 60, 32, 8
    g = torch.Generator(device="cuda").manual_seed(batch)
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device="cuda")
    off = [0, big] + [big + nodes * b for b in range(1, batch)]
    parent = [-1] + [0] * (big - 1) + list(range(-1, nodes - 1)) * (batch - 1)
    N = off[-1]
    tree = hb.TreeBatch(i32(off), i32(parent), i32([0] * N), batch, N)
    policy = dict(thresholds=[-1e9] * 7, d_base=200, alpha=4, n_default=128, top_k=10, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0,
                  entropy_mode=0)
    ctx = hb.Context(0, hb.hs_workspace_bytes(batch, N, 64, hq, hkv))
    _, pr = hb.hs_entropy_quantify_prune(ctx, tree, torch.zeros(N, 64, device="cuda"), policy)
    assert pr.n_keep.tolist() == [0] + [nodes] * (batch - 1)
    rn = lambda *s: torch.randn(*s, device="cuda", generator=g, dtype=torch.bfloat16)
    q, kt, vt = rn(N, hq, 128), rn(N, hkv, 128), rn(N, hkv, 128)
    kc, vc = rn(batch * kv, hkv, 128), rn(batch * kv, hkv, 128)
    outs = []
    for rows in (N, nodes * (batch - 1)):                        # the binding passes the first dimension of q as max_rows
        out = torch.zeros_like(q)
        hb.hs_tree_verify_attention(ctx, pr, q[:rows], kt, vt, kc, vc, i32([b * kv for b in range(batch + 1)]), batch=batch, max_nodes=nodes,
                                    max_kv_len=kv, layout=hb.HS_ROWS_ORIGINAL, node_off=tree.node_off, out=out)
        outs.append(out)
    assert torch.equal(outs[0], outs[1]) and bool((outs[0][big:].abs().sum((1, 2)) > 0).all())
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
