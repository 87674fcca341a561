"""Which attention kernel the lines give to a launch, and where its query rows come from, on the 148 SMs of the device that they are drawn for."""
import shutil

import pytest

from attn_route import route, splits_with_q_in_tensor_memory


@pytest.mark.skipif(not shutil.which("g++"), reason="no host compiler")
@pytest.mark.parametrize("batch, nodes, hq, hkv, longest, kernel", [
    (4, 62, 64, 8, 255 * 64, 0), (4, 62, 64, 8, 255 * 64 + 1, 2),         # 128 blocks: two splits that share SMs from 256 tiles on
    (18, 30, 32, 8, 448 * 64, 2),                                         # 144, one per head: from 448
    (10, 60, 32, 8, 9 * 64, -1), (10, 60, 32, 8, 128 * 64, -1), (10, 60, 32, 8, 8 * 64, 1), (10, 60, 32, 8, 129 * 64, 0),     # 160
    (20, 30, 32, 8, 9 * 64, 0), (20, 30, 32, 8, 128 * 64, 0), (18, 30, 32, 8, 447 * 64, 0),      # one query block per head: plain
    (3, 62, 64, 8, 32768, 0),                                             # 96: never
])
def test_lines(batch, nodes, hq, hkv, longest, kernel):
    assert route(batch, nodes, hq, hkv, longest, 148) == kernel


@pytest.mark.skipif(not shutil.which("g++"), reason="no host compiler")
@pytest.mark.parametrize("batch, nodes, hq, hkv, longest, splits", [
    (7, 60, 32, 8, 33 * 64, 0), (7, 60, 32, 8, 33 * 64 + 1, 1), (7, 60, 32, 8, 8192, 1),    # 112 blocks: from 34 prefix tiles and the tree's on
    (4, 100, 32, 8, 32 * 64, 0), (4, 100, 32, 8, 32 * 64 + 1, 1),         # two tiles of the tree
    (2, 60, 32, 8, 4 * 33 * 64, 0), (2, 60, 32, 8, 4 * 33 * 64 + 1, 4), (1, 60, 64, 8, 16384, 4),    # of a split's share
    (16, 60, 32, 8, 8192, 0),                   # more than one wave: not
    (10, 60, 32, 8, 60 * 64, 0), (10, 60, 32, 8, 60 * 64 + 1, 1), (12, 60, 32, 8, 4096, 0), (5, 60, 64, 8, 8192, 1), (10, 60, 32, 8, 8193, 0),    # but FOLLOW's above 60 tiles
    (5, 60, 32, 8, 12800, 0),                                             # 80 blocks in three splits: two waves
    (10, 30, 32, 8, 47 * 64, 0), (10, 30, 32, 8, 47 * 64 + 1, 1), (1, 30, 32, 8, 8 * 33 * 64, 0), (1, 30, 32, 8, 8 * 33 * 64 + 1, 8), (9, 30, 32, 8, 8192, 0),    # one query block per head: 80, 64, 144 CTAs
    (16, 30, 32, 8, 12000, 0), (2, 60, 32, 32, 8192, 0),
    (4, 62, 64, 8, 16384, 0),                                             # two CTAs per SM
])
def test_query_operand(batch, nodes, hq, hkv, longest, splits):
    assert splits_with_q_in_tensor_memory(batch, nodes, hq, hkv, longest, 148) == splits
