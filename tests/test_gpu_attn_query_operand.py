"""Where a CTA of tree_attn_umma_kernel takes the query rows from: shared memory up to 24 tiles, tensor memory from the ninth tile on above.  Prefixes on both
sides of that line in one launch and tree tiles at its end (ten trees of two query blocks: one split, the tree is a tile of its own), against the
reference and bounds of the launches that other tests make."""
import pytest

from test_gpu_attn_choice import test_room_in_the_cache_does_not_matter as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,hq,hkv,lens,kernel", [
    (60, 32, 8, [1472] * 5 + [1471, 1410, 64, 1, 0], -1),             # at most 23 + 1 tiles
    (60, 32, 8, [1473, 1536, 1537, 1600, 1472, 64, 1, 0, 500, 512], -1),    # 25 .. 27 tiles, and fewer
    (100, 32, 8, [1473, 1472, 1408, 1409, 3000], -1),                 # two tree tiles
    (60, 32, 32, [1473, 1472, 4000], 0),                              # one query block, splits
])
def test_query_rows_from_either_memory(nodes, hq, hkv, lens, kernel):
    check(nodes, hq, hkv, lens, kernel)
