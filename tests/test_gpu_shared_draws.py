"""The bonus draw of a deterministic-proposal sequence is cut into slices that idle CTAs of the row pass take; the sampling
walk uses clusters of 16 or of 8 CTAs.  Cases where the rules for that change: one sequence and many, more sequences
than the sharing keeps counters for, a vocabulary of one slice and of all 64, many siblings with repeated tokens."""
import pytest
import torch

from paper_2505_13254_b200 import binding as hb
from paper_2505_13254_b200 import step as gstep
from paper_2505_13254_b200 import synth

import parity_util as pu

pytestmark = pytest.mark.gpu

BASE = synth.CONFIGS["c4_ragged"].scaled(kv_len=(1, 1), temperature=1.0)
CASES = {
    "one": (BASE.scaled(batch=1, vocab=40000, accept="deterministic"), None),
    "few_f32_odd": (BASE.scaled(batch=3, vocab=12345, n_nodes=(8, 20), logits_dtype="f32", accept="deterministic"), 12348),
    "one_slice": (BASE.scaled(batch=12, vocab=3001, n_nodes=(8, 16), accept="mixed3"), 3008),
    "all_slices": (BASE.scaled(batch=1, vocab=260000, n_nodes=(4, 4), draft_depth=2, logits_dtype="f32", accept="deterministic"), None),
    "many": (BASE.scaled(batch=40, vocab=2500, n_nodes=(8, 14), accept="mixed3"), 2504),
    "unshared": (BASE.scaled(batch=260, vocab=600, n_nodes=(3, 6), draft_depth=2, accept="mixed3"), None),
}


def star(batch):
    """Sequence 0 becomes a root whose other nodes are all its children, every third with its left neighbour's token."""
    lo, hi = batch["node_off"][0], batch["node_off"][1]
    batch["parent"][lo + 1:hi] = 0
    batch["token"][lo + 3:hi:3] = batch["token"][lo + 2:hi - 1:3]


@pytest.mark.parametrize("variant", [hb.HS_ROW_PASS_CHUNK, hb.HS_ROW_PASS_STREAM])
@pytest.mark.parametrize("name", sorted(CASES) + ["star"])
def test_draws_match_the_oracle(name, variant):
    cfg, stride = CASES.get(name) or (BASE.scaled(batch=2, vocab=5000, n_nodes=(60, 60), accept="deterministic"), None)
    policy = pu.policy_for(cfg, "c4_ragged")
    batch, res = pu.oracle_case(cfg, policy, 9100, attention="none", mutate=star if name == "star" else None)
    db = gstep.upload(batch)
    if stride:                                                   # odd vocabularies: rows padded to whole vectors
        for field in ("draft", "target"):
            t = getattr(db, field)
            wide = torch.full((t.shape[0], stride), 9.0, dtype=t.dtype, device=t.device)
            wide[:, : t.shape[1]] = t
            setattr(db, field, wide[:, : t.shape[1]])
    ctx = hb.Context(0, 64 << 20)
    hb.hs_set_row_pass(ctx, variant)
    st = gstep.VerifyStep(ctx, db, policy)
    for _ in range(3):                                            # the counters of the draws have reset themselves
        st.quantify(db); st.prune(db); st.accept_path(db)
        torch.cuda.synchronize()
        pu.check_accept(st.accept, res)
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
