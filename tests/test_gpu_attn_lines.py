"""The lines between one attention kernel and the other and between split and unsplit prefixes, a launch on either side of each (`kernel`: see attn_route): blocks of
one and of two waves, one query block per head, the longest prefix one tile longer; same bits whatever room the cache has, and against
fp32 attention (bound there)."""
import pytest

import test_gpu_attn_choice as choice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,hq,hkv,lens,kernel", [
    (40, 32, 32, [512, 70], 0), (40, 32, 32, [513, 70], 0),               # 64 blocks, 8 and 9 tiles: one split, two
    (60, 32, 8, [256], 0), (60, 32, 8, [385], 0),                         # 16 blocks, 4 and 7 tiles: one split, several
    (60, 32, 8, [4096 - 31 * b for b in range(5)], 0),                    # 80 blocks, 64 tiles: two waves of splits do not pay
    (40, 32, 32, [512, 0, 1, 65, 300], 1), (40, 32, 32, [513, 0, 1, 65, 300], 0),    # 160 blocks of one each: two CTAs per SM, one
    (40, 32, 32, [2048, 5, 1024, 64, 1999, 640], 1), (40, 32, 32, [2049, 5, 1024, 64, 1999, 640], 0),    # 192 blocks, 32 and 33 tiles
    (16, 32, 32, [1024 - 64 * b for b in range(8)], 1), (16, 32, 32, [1025 - 64 * b for b in range(8)], 0),    # 256 blocks, 16 and 17
    (62, 64, 8, [16320, 1, 640, 0], 0), (62, 64, 8, [16321, 1, 640, 0], 2),    # 128 blocks, 255 and 256 tiles
    (62, 64, 8, [28609, 1, 640, 0], 2),                                   #   448 tiles
    (100, 32, 32, [28608, 1, 640, 0], 0), (100, 32, 32, [28609, 1, 640, 0], 2),    # the same of one each: 447 and 448
    (60, 32, 8, [3200 - 300 * b for b in range(10)], -1), (60, 32, 8, [8193 - 800 * b for b in range(10)], 0),    # 160: 50 tiles, 129
])
def test_both_sides_of_a_line(nodes, hq, hkv, lens, kernel):
    choice.test_room_in_the_cache_does_not_matter(nodes, hq, hkv, lens, kernel)
