"""The sampling walk where a thread's run of a vocabulary row is nothing, less than a vector, one piece held in registers or several, with clusters of
sixteen and of eight CTAs, and with many siblings to reject before the draw."""
import pytest
import torch

from paper_2505_13254_b200 import binding as hb
from paper_2505_13254_b200 import step as gstep
from paper_2505_13254_b200 import synth

import parity_util as pu

pytestmark = pytest.mark.gpu

BASE = synth.CONFIGS["c4_ragged"].scaled(kv_len=(1, 1), temperature=1.0, accept="rejection", draft_depth=2)
CASES = {
    "short": (BASE.scaled(batch=3, vocab=700, n_nodes=(6, 12)), 704),
    "one_piece_bf16": (BASE.scaled(batch=2, vocab=131072, n_nodes=(5, 8)), None),
    "two_pieces_bf16": (BASE.scaled(batch=2, vocab=131081, n_nodes=(5, 8)), 131088),
    "two_pieces_f32": (BASE.scaled(batch=1, vocab=140001, n_nodes=(5, 8), logits_dtype="f32"), 140004),
    "eight_ctas": (BASE.scaled(batch=40, vocab=70001, n_nodes=(3, 4)), 70008),
}


def star(batch):
    """The first sequence's nodes are all children of its root."""
    lo, hi = batch["node_off"][0], batch["node_off"][1]
    batch["parent"][lo + 1:hi] = 0


@pytest.mark.parametrize("name", sorted(CASES) + ["star"])
def test_the_walk_matches_the_oracle(name):
    cfg, stride = CASES.get(name) or (BASE.scaled(batch=2, vocab=40000, n_nodes=(40, 40), draft_depth=8), None)
    policy = pu.policy_for(cfg, "c4_ragged")
    batch, res = pu.oracle_case(cfg, policy, 9300, attention="none", mutate=star if name == "star" else None)
    db = gstep.upload(batch)
    if stride:                                                   # odd vocabularies: rows padded to whole vectors
        for field in ("draft", "target"):
            t = getattr(db, field)
            wide = torch.full((t.shape[0], stride), 9.0, dtype=t.dtype, device=t.device)
            wide[:, : t.shape[1]] = t
            setattr(db, field, wide[:, : t.shape[1]])
    ctx = hb.Context(0, 64 << 20)
    st = gstep.VerifyStep(ctx, db, policy)
    for _ in range(2):
        st.quantify(db); st.prune(db); st.accept_path(db)
        torch.cuda.synchronize()
        pu.check_accept(st.accept, res)
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
