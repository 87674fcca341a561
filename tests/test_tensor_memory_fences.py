"""Tensor memory handed from one warp to another across a barrier needs tcgen05.fence::before_thread_sync ahead of it and
tcgen05.fence::after_thread_sync behind it; no result shows a missing one reliably, so the sources are read."""
import os
import re

import pytest

from paper_2505_13254_b200 import build


def text(name):
    return re.sub(r"//.*", "", open(os.path.join(build.CSRC, name)).read())


def test_the_pair_barrier_carries_both_fences():
    body = re.search(r"void pair_sync\(int quad\) \{(.*?)\n\}", text("tree_attn_duo.cuh"), re.S).group(1)
    first, last = body.find("named_bar_sync"), body.rfind("named_bar_sync")
    assert 0 <= body.find("tc_fence_before_sync()") < first
    assert body.find("tc_fence_after_sync()") > last


@pytest.mark.parametrize("name", ["tree_attention.cu", "tree_attn_duo.cuh"])
def test_tensor_memory_is_freed_behind_a_fenced_barrier(name):
    last = text(name).rindex("tmem_dealloc(")
    tail = re.sub(r"\s+", "", text(name)[:last])
    assert re.search(r"tc_fence_before_sync\(\);__syncthreads\(\);tc_fence_after_sync\(\);if\(warp==\w+\)$", tail)


def test_lanes_that_waited_alone_meet_again_ahead_of_tensor_memory():
    # `if (!ok) mbar_wait(...)`: a lane waits by its own answer, and tcgen05.ld / st (.sync.aligned) need all lanes of the warp
    body = text("tree_attention.cu")
    waits = [m.end() for m in re.finditer(r"if \(!ok_\w+\) mbar_wait\(", body)]
    assert len(waits) == 2
    for at in waits:
        assert re.search(r"\btmem_\w+\(|__syncwarp\(\)|__any_sync\(HS_FULL_MASK", body[at:]).group(0).startswith("__")


def test_the_query_rows_are_handed_to_the_issuer_behind_both_fences():
    body = re.sub(r"\s+", " ", text("tree_attention.cu"))
    written = re.search(r"tmem_st32\(tQ (.*?)bar\.arrive 3, %0;\" ::\"r\"\(UM_SM_THREADS \+ 32\)", body).group(1)
    assert 0 < written.find("tmem_wait_st()") < written.find("tc_fence_before_sync()")
    # the issuer meets the 256 softmax threads once, ahead of the first product that reads them
    assert re.search(r"if \(i == UM_Q_FIRST\) \{ named_bar_sync\(3, UM_SM_THREADS \+ 32\); tc_fence_after_sync\(\); \} "
                     r"issue_qk\(i, \[\]\(int t\) \{ return t >= UM_Q_FIRST; \}\)", body)
    assert body.count("named_bar_sync(3,") == body.count("bar.arrive 3,") == 1
