"""The native call module reads the tensor bundles as the ctypes structures do: argument errors surface as Python
errors, everything else reaches the C call (handle 0 there gives HS_ERR_INVALID_ARG, so no device is needed)."""
import pytest
import torch

from paper_2505_13254_b200 import binding as hb

POLICY = dict(thresholds=[1.0] * 7, d_base=8, alpha=4, n_default=60, top_k=10, gamma_pct=(30, 60, 100), phi_mode=0,
              pstar_mode=0, entropy_mode=0)


def bundles(dtype=torch.bfloat16):
    z = torch.zeros(2, dtype=torch.int32)
    tree = hb.TreeBatch(z, z, z, 1, 1)
    return tree, torch.zeros(1, 64, dtype=dtype), hb.QuantOut(1, 1, 10, "cpu"), hb.PrunedTree(1, 1, "cpu")


def test_calls_reach_the_library():
    nat = hb.native()
    tree, x, q, pr = bundles()
    assert nat.entropy_quantify(0, tree, x, POLICY, q, 0) == hb.HS_ERR_INVALID_ARG
    assert nat.entropy_quantify_prune(0, tree, x, POLICY, q, pr, 0) == hb.HS_ERR_INVALID_ARG
    acc = hb.AcceptOut(1, 4, "cpu")
    assert nat.accept_path(0, tree, pr, x, 0, None, tree.parent, q.score, (1 << 64) - 1, 0, None, acc, 0) == hb.HS_ERR_INVALID_ARG
    assert nat.expand_init(0, hb.ExpandState(1, 11, 10, "cpu"), 0) == hb.HS_ERR_INVALID_ARG


@pytest.mark.parametrize("change,error", [(dict(d_base="x"), TypeError), (dict(thresholds=[0.0] * 8), IndexError),
                                          (dict(gamma_pct=None), TypeError), (None, KeyError)])
def test_a_bad_policy_is_a_python_error(change, error):
    tree, x, q, _ = bundles()
    policy = dict(POLICY, **change) if change else {k: v for k, v in POLICY.items() if k != "top_k"}
    with pytest.raises(error):
        hb.native().entropy_quantify(0, tree, x, policy, q, 0)


def test_a_bad_dtype_and_a_bad_call_are_python_errors():
    tree, x, q, _ = bundles(torch.float16)
    with pytest.raises(TypeError):
        hb.native().entropy_quantify(0, tree, x, POLICY, q, 0)
    with pytest.raises(AttributeError):
        hb.native().entropy_quantify(0, object(), x, POLICY, q, 0)
    with pytest.raises(TypeError):
        hb.native().entropy_quantify(0, tree)
