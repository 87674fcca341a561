"""The workloads this library is measured on, through the calls a user's program makes.

A verification step (`VerifyStep.run`, or its captured form `GraphedStep.replay`) is what a decode loop does once per
target forward pass; the attention call alone is what every layer of that forward pass does; growing the draft tree is
what happens ahead of it; the budgeted step is a serving batch under a token budget; the training of the stratifier is
the offline part.  Shapes are those of the benchmark configurations and what lies between and around them.

Inputs follow the recipe of the synthetic batches the tests use (peaked and flat draft rows, a tree grown by the top-k
children of the k most confident nodes per level and reranked, target rows = noisy draft rows with the most confident
child raised), made on the device so that a batch takes milliseconds.
"""

import math
import random

import numpy as np
import torch

from paper_2505_13254_b200 import binding as hb
from paper_2505_13254_b200 import step as hs_step

HEAD_DIM = 128
TOP_K = 10
N_DEFAULT = 60
# octiles of Phi(P*) of calibration trees: one tree at a time, and a ragged batch (trees of 8 - 60 nodes)
THRESHOLDS = (5.3, 5.7, 6.1, 6.4, 6.7, 7.0, 7.3)
THRESHOLDS_RAGGED = (3.8, 4.6, 5.2, 5.6, 5.9, 6.5, 7.1)
# most bytes and operations of a drawn case: those of the largest listed ones
MOST_BYTES, MOST_FLOPS = 8.0e8, 2.6e11


def _step(name, **kw):
    case = dict(name=name, kind="step", batch=1, nodes_lo=60, nodes_hi=60, depth=8, d_base=8, vocab=128256, logits="bf16",
                hq=32, hkv=8, kv_lo=2048, kv_hi=2048, accept="greedy", temperature=0.0, call="eager")
    case.update(kw)
    return case


def listed():
    return [
        # the smallest model: 32000 tokens, fp32 logits, no grouped heads; nothing here takes the GPU longer than a few us
        _step("step_tiny_f32", depth=6, d_base=6, vocab=32000, logits="f32", hkv=32, kv_lo=512, kv_hi=512),
        # one interactive sequence of an 8B-shaped model, temperature 0, the calls made one by one ...
        _step("step_8b"),
        # ... and the same step replayed as one CUDA graph
        _step("step_8b_graph", call="graph"),
        # one sequence of a 70B-shaped model, sampling
        _step("step_70b_sampling", hq=64, kv_lo=4096, kv_hi=4096, accept="rejection", temperature=1.0),
        # a ragged serving batch, greedy and sampling requests mixed
        _step("step_ragged", batch=16, nodes_lo=8, kv_lo=1024, kv_hi=8192, accept="mixed", temperature=1.0),
        # long contexts, trees drafted deeper than the base depth
        _step("step_long", batch=4, nodes_lo=96, nodes_hi=96, depth=12, hq=64, kv_lo=32768, kv_hi=32768,
              accept="rejection", temperature=0.7),
        # sampling from trees whose candidates are the draft model's top-k tokens (point-mass proposals)
        _step("step_topk_drafts", batch=8, nodes_lo=24, kv_lo=512, kv_hi=4096, accept="deterministic", temperature=1.0),
        # many small requests that share a token budget and have service classes
        _step("step_budget", batch=32, nodes_lo=8, vocab=32000, kv_lo=256, kv_hi=2048, accept="mixed3", temperature=1.0,
              call="budget"),
        # the attention of one target forward pass: a call per layer, rows compacted to the kept nodes
        dict(name="layers_8b", kind="layers", layers=32, batch=1, nodes_lo=60, nodes_hi=60, hq=32, hkv=8, kv_lo=2048,
             kv_hi=2048, cache="token"),
        # the same for a batch of a 70B-shaped model, cache laid out head by head (a few of its layers)
        dict(name="layers_70b_batch", kind="layers", layers=4, batch=4, nodes_lo=40, nodes_hi=60, hq=64, hkv=8, kv_lo=1024,
             kv_hi=8192, cache="head"),
        # growing the draft trees of four sequences level by level and reranking them
        dict(name="grow_trees", kind="grow", batch=4, depth=8, top_k=10, n_top=60, vocab=128256, logits="bf16"),
        # training the stratifier on a million verified trees
        dict(name="train_stratifier", kind="cart", pairs=1 << 20, depth=3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _within(case):
    w = work(case)
    return w["bytes"] <= MOST_BYTES and w["flops"] <= MOST_FLOPS


def draw(rng):
    while True:
        kind = rng.choice(("step", "step", "step", "step", "layers", "layers", "grow", "cart"))
        if kind == "cart":
            return dict(kind="cart", pairs=_log(rng, 600, 1 << 20), depth=rng.choice((2, 3, 3, 4, 5)))
        if kind == "grow":
            case = dict(kind="grow", batch=_log(rng, 1, 12), depth=rng.randint(4, 10), top_k=rng.choice((4, 8, 10, 10, 16)),
                        n_top=rng.randint(20, 100), vocab=_log(rng, 32000, 131072), logits=rng.choice(("bf16", "bf16", "f32")))
        else:
            hq, hkv = rng.choice(((32, 32), (32, 8), (32, 8), (64, 8)))
            batch, kv = _log(rng, 1, 16), _log(rng, 512, 32768)
            lo = rng.randint(8, 60)
            case = dict(kind=kind, batch=batch, nodes_lo=lo, nodes_hi=rng.randint(lo, 60), hq=hq, hkv=hkv,
                        kv_lo=max(256, int(kv * rng.uniform(0.2, 1.0))), kv_hi=kv)
            if kind == "layers":
                case.update(layers=_log(rng, 2, 32), cache=rng.choice(("token", "head")))
            else:
                call = rng.choice(("eager", "eager", "graph", "budget"))
                accept = rng.choice(("greedy", "greedy", "rejection", "deterministic", "mixed", "mixed3"))
                deep = rng.random() < 0.25
                case.update(depth=12 if deep else 8, d_base=8, vocab=_log(rng, 32000, 131072), accept=accept,
                            logits=rng.choice(("bf16", "bf16", "bf16", "f32")), call=call,
                            temperature=0.0 if accept == "greedy" else rng.choice((0.7, 1.0)))
                if deep:
                    case["nodes_hi"] = rng.randint(case["nodes_hi"], 96)
        if _within(case):
            return case


# ---- inputs --------------------------------------------------------------------------------------------------


def _policy(case):
    ragged = case["nodes_lo"] < 40
    d_base = case.get("d_base", 8)
    return dict(thresholds=list(THRESHOLDS_RAGGED if ragged else THRESHOLDS), d_base=d_base, alpha=(d_base + 1) // 2,
                n_default=N_DEFAULT, top_k=TOP_K, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0, entropy_mode=0)


class _Rows:
    """Draft rows on the device: scale * N(0, 1), and for a peaked row a head of three tokens on top of it."""

    def __init__(self, gen, vocab, dtype):
        self.gen, self.vocab, self.dtype, self.dev = gen, vocab, dtype, torch.device("cuda")

    def rand(self, *shape):
        return torch.rand(*shape, generator=self.gen, device=self.dev)

    def __call__(self, peaked):
        n = peaked.numel()
        x = torch.randn(n, self.vocab, generator=self.gen, device=self.dev)
        x *= torch.where(peaked, 1.0 / 0.3, 1.0 / 3.0)[:, None]
        lse = torch.logsumexp(x, dim=1)
        v0 = lse + 3.5 * self.rand(n)
        v1 = v0 - (1.0 + 2.0 * self.rand(n))
        v2 = v1 - (0.5 + 1.5 * self.rand(n))
        third = self.vocab // 3                                       # three distinct tokens
        head = (self.rand(n, 3) * third).long() + torch.arange(3, device=self.dev) * third
        x.scatter_(1, head, torch.where(peaked[:, None], torch.stack((v0, v1, v2), 1), x.gather(1, head)))
        return x.to(self.dtype)


def _padded(rows):
    """A view of `rows` whose row stride is a multiple of eight elements, as an LM head with a padded output has it."""
    n, v = rows.shape
    if v % 8 == 0:
        return rows.contiguous()
    buf = torch.zeros(n, (v + 7) // 8 * 8, dtype=rows.dtype, device=rows.device)
    buf[:, :v] = rows
    return buf[:, :v]


def _top(x, k):
    """The k largest of every row, ties to the lower index."""
    key = x.double() - 1e-12 * torch.arange(x.shape[1], device=x.device, dtype=torch.float64)
    idx = torch.topk(key, k, dim=1).indices
    return x.float().gather(1, idx), idx


def _trees(gen, sizes, depth, vocab, dtype, ragged):
    """One draft tree per sequence: (node_off, parent, token) on the host, draft rows on the device and which of them are
    peaked.  Levels are grown for the whole batch at once."""
    rows, B, k, dev = _Rows(gen, vocab, dtype), len(sizes), TOP_K, torch.device("cuda")
    frac = rows.rand(B) if ragged else torch.full((B,), 0.6, device=dev)
    peaked = rows.rand(B, 1) < frac[:, None]
    S = torch.zeros(B, 1, device=dev)
    ids = torch.zeros(B, 1, dtype=torch.long, device=dev)             # candidate ids of the frontier
    par, tok, val, pk = [torch.full((B, 1), -1, device=dev)], [torch.zeros(B, 1, dtype=torch.long, device=dev)], [S], [peaked]
    kept_rows, n_cand = [], 1
    where = {}                                                       # (level, frontier ids) of the rows made so far
    for level in range(depth):
        f = ids.shape[1]
        x = rows(peaked.reshape(-1))
        kept_rows.append(x)
        where[level] = ids
        v, t = _top(x, k)
        logc = v - torch.logsumexp(x.float(), dim=1, keepdim=True)
        lead = torch.zeros(B, f, k, dtype=torch.bool, device=dev)
        lead[:, :, 0] = peaked
        child = (S[:, :, None] + logc.reshape(B, f, k)).reshape(B, f * k)
        u = rows.rand(B, f * k)
        cpk = u < torch.where(lead.reshape(B, f * k), torch.tensor(0.95, device=dev), frac[:, None])
        par.append(ids[:, :, None].expand(B, f, k).reshape(B, f * k)); tok.append(t.reshape(B, f * k))
        val.append(child); pk.append(cpk)
        order = torch.sort(child, dim=1, descending=True, stable=True).indices[:, :k]
        S, peaked, ids = child.gather(1, order), cpk.gather(1, order), n_cand + order
        n_cand += f * k
    par, tok, pk = torch.cat(par, 1).cpu().numpy(), torch.cat(tok, 1).cpu().numpy(), torch.cat(pk, 1).cpu().numpy()
    rank = torch.sort(torch.cat(val, 1), dim=1, descending=True, stable=True).indices.cpu().numpy()
    row_of = np.full((B, n_cand), -1)
    base = 0
    for level, x in enumerate(kept_rows):
        fid = where[level].cpu().numpy()
        for b in range(B):
            row_of[b, fid[b]] = base + b * fid.shape[1] + np.arange(fid.shape[1])
        base += x.shape[0]
    off, parent, token, src, flags = [0], [], [], [], []
    for b, n in enumerate(sizes):
        keep = np.sort(rank[b, :n])
        local = np.full(n_cand, -1)
        local[keep] = np.arange(len(keep))
        p = par[b, keep]
        parent.append(np.where(p < 0, -1, local[p])); token.append(tok[b, keep]); src.append(row_of[b, keep]); flags.append(pk[b, keep])
        off.append(off[-1] + len(keep))
    parent, token, src, flags = (np.concatenate(a) for a in (parent, token, src, flags))
    fresh = np.nonzero(src < 0)[0]                                   # nodes that were never expanded get rows of their own
    draft = torch.empty(len(src), vocab, dtype=dtype, device=dev)
    old = np.nonzero(src >= 0)[0]
    level_of = np.searchsorted(np.cumsum([x.shape[0] for x in kept_rows]), src[old], side="right")
    starts = np.concatenate(([0], np.cumsum([x.shape[0] for x in kept_rows])))
    for level, x in enumerate(kept_rows):
        sel = old[level_of == level]
        if len(sel):
            draft[torch.from_numpy(sel).cuda()] = x[torch.from_numpy(src[sel] - starts[level]).cuda()]
    if len(fresh):
        draft[torch.from_numpy(fresh).cuda()] = rows(torch.from_numpy(flags[fresh]).cuda())
    return off, parent, token, draft, flags


def _target(gen, draft, parent, token, off, flags):
    """Draft rows plus noise of half their scale; with probability 0.9 the first child's token on top."""
    dev = draft.device
    t = torch.randn(draft.shape, generator=gen, device=dev)
    t *= torch.where(torch.from_numpy(flags).to(dev), 0.5 / 0.3, 0.5 / 3.0)[:, None]
    t += draft
    first = np.full(len(parent), -1)
    for b in range(len(off) - 1):
        for i in range(off[b + 1] - 1, off[b], -1):
            first[off[b] + parent[i]] = token[i]
    lift = (torch.rand(len(parent), generator=gen, device=dev) < 0.9) & torch.from_numpy(first >= 0).to(dev)
    at = torch.from_numpy(np.maximum(first, 0)).to(dev)[:, None]
    t.scatter_(1, at, torch.where(lift[:, None], t.max(1, keepdim=True).values + 2.0, t.gather(1, at)))
    return t.to(draft.dtype)


def _i32(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.int32, device="cuda")


def _normal(gen, *shape):
    return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)


def _sizes(case):
    """Tree sizes and prefix lengths of the sequences: part of the case, not of the seed."""
    rng = random.Random(1000003 * case["batch"] + 1009 * case["nodes_lo"] + case["kv_hi"])
    ns = [rng.randint(case["nodes_lo"], case["nodes_hi"]) for _ in range(case["batch"])]
    return ns, [rng.randint(case["kv_lo"], case["kv_hi"]) for _ in range(case["batch"])]


def _setup(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    return gen, random.Random(seed)


def _batch(case, seed):
    """A DeviceBatch of the case: trees, logits and, for a step, query / key / value rows and the cache."""
    gen, rng = _setup(seed)
    B, step = case["batch"], case["kind"] == "step"
    sizes, lens = _sizes(case)
    vocab, dtype = (case["vocab"], torch.float32 if case["logits"] == "f32" else torch.bfloat16) if step else (32000, torch.bfloat16)
    off, parent, token, draft, flags = _trees(gen, sizes, case.get("depth", 8), vocab, dtype, case["nodes_lo"] < 40)
    kv_off = np.concatenate(([0], np.cumsum(lens)))
    accept = case.get("accept", "greedy")
    mode = np.array([{"greedy": 0, "rejection": 1, "deterministic": 2, "mixed": b % 2, "mixed3": b % 3}[accept] for b in range(B)])
    n, total = len(parent), int(kv_off[-1])
    heads = lambda rows, h: _normal(gen, rows, h, HEAD_DIM)
    return hs_step.DeviceBatch(
        tree=hb.TreeBatch(_i32(off), _i32(parent), _i32(token), B, n), draft=_padded(draft),
        target=_padded(_target(gen, draft, parent, token, off, flags)) if step else None,
        q=heads(n, case["hq"]) if step else None, k_tree=heads(n, case["hkv"]) if step else None,
        v_tree=heads(n, case["hkv"]) if step else None, k_cache=heads(total, case["hkv"]) if step else None,
        v_cache=heads(total, case["hkv"]) if step else None, kv_off=_i32(kv_off), mode=_i32(mode),
        temperature=torch.tensor(np.where(mode != 0, case.get("temperature", 0.0), 0.0), dtype=torch.float32, device="cuda"),
        seed=(seed * 0x9E3779B97F4A7C15 + 0x1234567) & (2 ** 64 - 1), offset=0, max_nodes=max(sizes), max_kv_len=max(lens),
        any_sampling=bool((mode == 1).any())), gen, rng


def _context(batch, rows, vocab, hq=1, hkv=1, prefetch=0):
    ctx = hb.Context(0, hb.hs_workspace_bytes(batch, rows, vocab, hq, hkv))
    hb.hs_set_prefetch(ctx, prefetch)
    return ctx


def prepare(case, seed):
    return {"step": _prepare_step, "layers": _prepare_layers, "grow": _prepare_grow, "cart": _prepare_cart}[case["kind"]](case, seed)


def _prepare_step(case, seed):
    db, gen, rng = _batch(case, seed)
    # the cache was appended a step ago; in a captured step the logits are in place long before the replay as well
    prefetch = hb.HS_PREFETCH_KV | (hb.HS_PREFETCH_LOGITS if case["call"] == "graph" else 0)
    ctx = _context(case["batch"], db.tree.n_nodes_total, case["vocab"], case["hq"], case["hkv"], prefetch)
    st = hs_step.VerifyStep(ctx, db, _policy(case))
    state = dict(kind="step", call=case["call"], ctx=ctx, db=db, step=st)
    if case["call"] == "graph":
        state["graph"] = hs_step.GraphedStep(st, db)
    if case["call"] == "budget":
        state["budget"] = max(case["batch"], int(0.75 * db.tree.n_nodes_total))
        state["slo"] = _i32([rng.randint(0, 2) for _ in range(case["batch"])])
    return state


def _prepare_layers(case, seed):
    db, gen, _ = _batch(case, seed)
    n, total, policy, layers = db.tree.n_nodes_total, int(db.kv_off[-1]), _policy(case), []
    ctx = _context(case["batch"], n, 32000, case["hq"], case["hkv"], hb.HS_PREFETCH_KV)
    quant, pruned = hb.QuantOut(n, case["batch"], TOP_K, "cuda"), hb.PrunedTree(n, case["batch"], "cuda")
    hb.hs_entropy_quantify_prune(ctx, db.tree, db.draft, policy, out=quant, pruned_out=pruned)
    for _ in range(case["layers"]):
        q, kt, vt = _normal(gen, n, case["hq"], HEAD_DIM), _normal(gen, n, case["hkv"], HEAD_DIM), _normal(gen, n, case["hkv"], HEAD_DIM)
        if case["cache"] == "head":
            kc, vc = (_normal(gen, case["hkv"], total, HEAD_DIM).permute(1, 0, 2) for _ in range(2))
        else:
            kc, vc = (_normal(gen, total, case["hkv"], HEAD_DIM) for _ in range(2))
        layers.append((q, kt, vt, kc, vc, torch.zeros_like(q)))
    db.draft = None
    return dict(kind="layers", ctx=ctx, db=db, pruned=pruned, layers=layers, bound=hs_step.keep_bound(policy, db.max_nodes))


def _prepare_grow(case, seed):
    gen, _ = _setup(seed)
    B, k = case["batch"], case["top_k"]
    rows = _Rows(gen, case["vocab"], torch.float32 if case["logits"] == "f32" else torch.bfloat16)
    levels = []
    for level in range(case["depth"]):                # the draft model's rows after the frontier of every level
        x = rows(rows.rand(B * k) < 0.6)
        levels.append(_padded(x.reshape(B, k, -1)[:, :1].expand(B, k, x.shape[1]).reshape(B * k, -1) if level == 0 else x))
    star = hb.TreeBatch(_i32([b * k for b in range(B + 1)]), _i32(([-1] + [0] * (k - 1)) * B), _i32([0] * (B * k)), B, B * k)
    policy = dict(thresholds=list(THRESHOLDS), d_base=case["depth"], alpha=(case["depth"] + 1) // 2, n_default=N_DEFAULT,
                  top_k=k, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0, entropy_mode=0)
    return dict(kind="grow", ctx=_context(B, B * k, case["vocab"]), levels=levels, star=star, policy=policy, n_top=case["n_top"],
                tree=hb.ExpandState(B, 1 + k + (case["depth"] - 1) * k * k, k, "cuda"), quant=hb.QuantOut(B * k, B, k, "cuda"))


def _prepare_cart(case, seed):
    gen, _ = _setup(seed)
    n = case["pairs"]
    u = torch.rand(4, n, generator=gen, device="cuda").clamp_min(1e-7)
    x = -2.0 * torch.log(u).sum(0)                     # entropies: positive, skewed; ranks 0 .. 59 that grow with them
    x = torch.where(torch.rand(n, generator=gen, device="cuda") < 0.1, x.roll(1), x)          # some values repeat
    y = torch.clamp(torch.round(0.4 * x ** 1.5 + 3.0 * torch.randn(n, generator=gen, device="cuda")), 0, 59)
    return dict(kind="cart", ctx=hb.Context(0, hb.hs_cart_workspace_bytes(n) + (1 << 20)), x=x, y=y, depth=case["depth"])


# ---- one pass --------------------------------------------------------------------------------------------------


def run(state):
    return {"step": _run_step, "layers": _run_layers, "grow": _run_grow, "cart": _run_cart}[state["kind"]](state)


_QUANT = ("row_max", "row_lse", "h_full", "i_topk", "i_trunc", "topk_val", "topk_idx", "logc", "score", "phi", "depth",
          "pstar_node", "phi_star", "status")
_PRUNED = ("bin", "d_prime", "n_prime", "n_keep", "keep_off", "keep_idx", "new_parent", "new_depth", "keep_rank", "anc_mask",
           "status")
_ACCEPT = ("accept_len", "path_nodes", "path_compact", "path_tokens", "bonus_token", "terminal_rank", "status")
_TREE = ("n_cand", "parent", "token", "depth", "logc", "score", "frontier", "n_frontier", "status")


def _run_step(state):
    st, db = state["step"], state["db"]
    if state["call"] == "graph":
        state["graph"].replay()
    elif state["call"] == "budget":
        st.quantify(db)
        hb.hs_stratify_prune_budget(state["ctx"], db.tree, st.quant, st.policy, state["slo"], state["budget"], out=st.pruned)
        st.attention(db, max_nodes=db.max_nodes)
        st.accept_path(db)
    else:
        st.run(db)
    return {"quant": [getattr(st.quant, n) for n in _QUANT], "pruned": [getattr(st.pruned, n) for n in _PRUNED],
            "accept": [getattr(st.accept, n) for n in _ACCEPT], "out": st.attn_out, "lse": st.attn_lse}


def _run_layers(state):
    db, outs = state["db"], []
    for q, kt, vt, kc, vc, out in state["layers"]:
        outs.append(hb.hs_tree_verify_attention(state["ctx"], state["pruned"], q, kt, vt, kc, vc, db.kv_off, batch=db.tree.batch,
                                                max_nodes=state["bound"], max_kv_len=db.max_kv_len, out=out))
    return outs


def _run_grow(state):
    ctx, tree = state["ctx"], state["tree"]
    hb.hs_expand_init(ctx, tree)
    for logits in state["levels"]:
        hb.hs_entropy_quantify(ctx, state["star"], logits, state["policy"], out=state["quant"])
        hb.hs_expand_level(ctx, tree, state["quant"])
    return {"rows": [getattr(state["quant"], n) for n in _QUANT], "tree": [getattr(tree, n) for n in _TREE],
            "reranked": hb.hs_rerank(ctx, tree, None, state["n_top"])}


def _run_cart(state):
    return hb.hs_cart_fit(state["ctx"], state["x"], state["y"], state["depth"])


# ---- what a pass cannot do without, and how far another correct implementation may be off ------------------------


def work(case):
    """Bytes: every logits row, the cache and the rows of the kept nodes once, the outputs once.  Operations: the two
    products of the attention; for the rest a handful per value read (exponential, sums) counts as nothing beside it."""
    if case["kind"] == "cart":
        return {"bytes": 8.0 * case["pairs"], "flops": 4.0 * case["depth"] * case["pairs"]}
    if case["kind"] == "grow":
        size = 4 if case["logits"] == "f32" else 2
        rows = case["batch"] * (1 + (case["depth"] - 1) * case["top_k"])
        return {"bytes": float(rows * case["vocab"] * size), "flops": 4.0 * rows * case["vocab"]}
    nodes, kv = _sizes(case)
    # of the eight regimes one keeps 30 % of the default, one 60 %, the others all of it (at most the tree)
    kept = [min(n, 0.86 * N_DEFAULT) for n in nodes]
    attn_bytes = sum((4.0 * (l + k) * case["hkv"] + 4.0 * k * case["hq"]) * HEAD_DIM for k, l in zip(kept, kv))
    attn_flops = sum(4.0 * k * (l + k) * case["hq"] * HEAD_DIM for k, l in zip(kept, kv))
    if case["kind"] == "layers":
        return {"bytes": case["layers"] * attn_bytes, "flops": case["layers"] * attn_flops}
    size = 4 if case["logits"] == "f32" else 2
    # the acceptance reads the target row of every kept node; a rejection-sampling sequence the draft rows of its inner nodes
    share = {"greedy": 0.0, "deterministic": 0.0, "rejection": 1.0, "mixed": 0.5, "mixed3": 1 / 3}[case["accept"]]
    rows = sum(nodes) + (1 + 0.4 * share) * sum(kept)
    return {"bytes": rows * case["vocab"] * size + attn_bytes, "flops": 4.0 * rows * case["vocab"] + attn_flops}


def tolerance(case):
    if case["kind"] in ("step", "layers"):
        # the attention's output is bf16 and so are its probabilities; everything else is 32-bit sums or whole numbers
        return {"rel": 1e-2, "max": 0.1}
    return {"rel": 1e-5}
