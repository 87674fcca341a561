"""kv_off of the attention call may be written by the launch directly ahead of it (here the reranking, whose last store it is): without
the caller's word for the cache nothing of it may be read before that launch has ended.  Both attention kernels."""
import pytest
import torch

from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,nodes,hq", [(3, 20, 32), (40, 96, 32)])
def test_offsets_written_by_the_launch_ahead(batch, nodes, hq):
    dev, hkv = torch.device("cuda:0"), 8
    g = torch.Generator(device="cuda").manual_seed(batch)
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device=dev)
    lens = [40 + (37 * b) % 700 for b in range(batch)]
    tree = hb.TreeBatch(i32([b * nodes for b in range(batch + 1)]), i32(([-1] + list(range(nodes - 1))) * batch),
                        i32([0] * (batch * nodes)), batch, batch * nodes)
    policy = dict(thresholds=[-1e9] * 7, d_base=200, alpha=4, n_default=128, top_k=10, gamma_pct=[30, 60, 100], phi_mode=0,
                  pstar_mode=0, entropy_mode=0)
    ctx = hb.Context(0, hb.hs_workspace_bytes(batch, batch * nodes, 64, hq, hkv))
    _, pr = hb.hs_entropy_quantify_prune(ctx, tree, torch.randn(batch * nodes, 64, device=dev, generator=g), policy)
    rn = lambda *s: torch.randn(*s, device=dev, generator=g, dtype=torch.bfloat16)
    q, kt, vt = rn(batch * nodes, hq, 128), rn(batch * nodes, hkv, 128), rn(batch * nodes, hkv, 128)
    kc, vc = rn(sum(lens), hkv, 128), rn(sum(lens), hkv, 128)
    # candidate trees whose reranking keeps lens[b] nodes: its node_off is the attention's kv_off
    st = hb.ExpandState(batch, 2048, 10, dev)
    hb.hs_expand_init(ctx, st)
    st.n_cand.fill_(2048)
    n_top, rest = i32(lens), [torch.zeros(sum(lens), dtype=torch.int32, device=dev) for _ in range(4)]

    def attend(kv_off):
        return hb.hs_tree_verify_attention(ctx, pr, q, kt, vt, kc, vc, kv_off, batch=batch, max_nodes=nodes, max_kv_len=max(lens))

    off = [0]
    for n in lens:
        off.append(off[-1] + n)
    want = attend(i32(off))
    for _ in range(5):
        kv_off = torch.zeros(batch + 1, dtype=torch.int32, device=dev)
        torch.cuda.synchronize()
        stream = torch.cuda.current_stream().cuda_stream
        assert hb.native().rerank(ctx.handle.value, st, n_top, 1, kv_off, *rest, stream) == 0
        got = attend(kv_off)
        assert kv_off.tolist() == off and torch.equal(got, want)
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
