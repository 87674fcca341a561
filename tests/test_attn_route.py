"""Which attention kernel the lines give to a launch, on the 148 SMs of the device that they are drawn for."""
import shutil

import pytest

from attn_route import route


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
