"""The lines between one attention kernel and the other and between split and unsplit prefixes, a launch on either side of each: blocks of
one and of two waves, one query block per head, the longest prefix one tile longer; same bits whatever room the cache has, and against
fp32 attention (bound there)."""
import pytest

import test_gpu_attn_choice as choice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,hq,hkv,lens", [
    (40, 32, 32, [512, 70]), (40, 32, 32, [513, 70]),                     # 64 blocks, 8 and 9 tiles: one split, two
    (60, 32, 8, [256]), (60, 32, 8, [385]),                               # 16 blocks, 4 and 7 tiles: one split, several
    (60, 32, 8, [4096 - 31 * b for b in range(5)]),                       # 80 blocks, 64 tiles: two waves of splits do not pay
    (40, 32, 32, [512, 0, 1, 65, 300]), (40, 32, 32, [513, 0, 1, 65, 300]),          # 160 blocks of one each: two CTAs per SM, one
    (40, 32, 32, [2048, 5, 1024, 64, 1999, 640]), (40, 32, 32, [2049, 5, 1024, 64, 1999, 640]),    # 192 blocks, 32 and 33 tiles
    (16, 32, 32, [1024 - 64 * b for b in range(8)]), (16, 32, 32, [1025 - 64 * b for b in range(8)]),    # 256 blocks, 16 and 17
    (62, 64, 8, [16320, 1, 640, 0]), (62, 64, 8, [16321, 1, 640, 0]),     # 128 blocks, 255 and 256 tiles
    (62, 64, 8, [28609, 1, 640, 0]),                                      #   448 tiles
])
def test_both_sides_of_a_line(nodes, hq, hkv, lens):
    choice.test_room_in_the_cache_does_not_matter(nodes, hq, hkv, lens)
