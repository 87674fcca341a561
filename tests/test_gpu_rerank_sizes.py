"""Reranking and expansion where the selection can go wrong: ties at the cut, fewer candidates than asked for, one
candidate, candidate counts around a warp, a block of threads and the two candidates a thread holds."""
import numpy as np
import pytest
import torch

from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


def expected(S, parent, n):
    order = sorted(range(len(S)), key=lambda c: (-S[c], c))[:n]
    keep = sorted(order)
    new = {c: i for i, c in enumerate(keep)}
    return keep, [-1 if parent[c] < 0 else new[int(parent[c])] for c in keep]


@pytest.mark.parametrize("counts,cap,n_top", [((1, 2, 33), 40, 5), ((31, 32, 64), 64, 32), ((711, 700, 5), 711, 60), ((1023, 1024), 1024, 100),
                                              ((1025, 2048, 1100), 2048, 128), ((900, 900), 2048, 2000)])
@pytest.mark.parametrize("levels", [0, 6])
def test_reranking_selects_by_value_then_creation(counts, cap, n_top, levels):
    rng = np.random.default_rng(cap + levels)
    B = len(counts)
    ctx = hb.Context(0, 8 << 20)
    st = hb.ExpandState(B, cap, min(16, cap - 1), "cuda")
    want, trees = [], []
    for b, n in enumerate(counts):
        parent = np.array([-1] + [rng.integers(0, i) for i in range(1, n)], dtype=np.int32)
        step = -rng.random(n).astype(np.float32)
        if levels:
            step = np.round(step * levels) / np.float32(levels)              # many ties, zeros among them
        S, dep = np.zeros(n, dtype=np.float32), np.zeros(n, dtype=np.int32)
        for i in range(1, n):
            S[i], dep[i] = S[parent[i]] + step[i], dep[parent[i]] + 1
        tok = rng.integers(0, 1000, n).astype(np.int32)
        for name, a in (("parent", parent), ("score", S), ("depth", dep), ("token", tok)):
            getattr(st, name)[b, :n] = torch.from_numpy(a).cuda()
        st.n_cand[b] = n
        trees.append((S, parent, dep, tok))
    node_off, parent, token, cand_id, depth = (t.cpu().numpy() for t in hb.hs_rerank(ctx, st, None, n_top))
    for b, (S, par, dep, tok) in enumerate(trees):
        keep, new = expected(S, par, min(n_top, counts[b]))
        sl = slice(node_off[b], node_off[b + 1])
        assert cand_id[sl].tolist() == keep and parent[sl].tolist() == new
        assert np.array_equal(depth[sl], dep[keep]) and np.array_equal(token[sl], tok[keep])
    ctx.close()
