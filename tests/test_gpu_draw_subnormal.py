"""The bonus draw of a deterministic-proposal sequence counts every token of positive probability, those below fp32's normal range
included: with u = 0 the drawn token is the first whose mass is not zero (2^-137 here), as in the fp64 definition."""
import numpy as np
import pytest
import torch

from oracle import accept as oacc
from paper_2505_13254_b200 import binding as hb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [hb.HS_ROW_PASS_CHUNK, hb.HS_ROW_PASS_STREAM])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
@pytest.mark.parametrize("first", [0, 1100, 2999])
def test_masses_below_the_normal_range_are_drawn(variant, dtype, first):
    vocab, dev = 3000, torch.device("cuda:0")
    i32 = lambda a: torch.tensor(a, dtype=torch.int32, device=dev)
    tree = hb.TreeBatch(i32([0, 1]), i32([-1]), i32([0]), 1, 1)
    row = torch.full((1, vocab), -float("inf"))
    row[0, first] = -95.0
    row[0, 2999] = 0.0                                          # all the mass that a sum in fp32 would notice
    row = row.to(dtype).to(dev)
    policy = dict(thresholds=[1.0] * 7, d_base=8, alpha=4, n_default=60, top_k=2, gamma_pct=[30, 60, 100], phi_mode=0, pstar_mode=0,
                  entropy_mode=0)
    ctx = hb.Context(0, 16 << 20)
    hb.hs_set_row_pass(ctx, variant)
    _, pr = hb.hs_entropy_quantify_prune(ctx, tree, row, policy)
    acc = hb.hs_accept_path(ctx, tree, pr, row, None, i32([hb.HS_ACCEPT_DETERMINISTIC]), torch.ones(1, device=dev),
                            uniforms=torch.zeros(2, device=dev))
    _, want = oacc.deterministic(np.array([-1]), np.array([0]), row.double().cpu().numpy(), 1.0, np.zeros(1), 0.0)
    assert int(acc.status[0]) == 0 and int(acc.accept_len[0]) == 0
    assert int(acc.bonus_token[0]) == want == first
    assert hb.hs_device_error(ctx) == 0
    ctx.close()
