"""Where a CTA of tree_attn_umma_kernel takes the query rows from: shared memory up to 34 tiles, tensor memory from the ninth tile on above, in the launches for
which that is faster (`splits`: of such a launch, 0 for the others; see attn_route).  CTAs on both sides of that line in
one launch, tree tiles at the end, splits of which some are long, against the reference and bounds of the launches that other tests make."""
import pytest

from attn_route import splits_with_q_in_tensor_memory
from test_gpu_attn_choice import test_room_in_the_cache_does_not_matter as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,hq,hkv,lens,kernel,splits", [
    (60, 32, 8, [2112] * 3 + [2111, 64, 1, 0], 0, 0),                 # at most 33 tiles and the tree's
    (60, 32, 8, [2176, 2113, 2112, 2048, 64, 1, 0], 0, 1),            # 35 and 34 with the tree's, and fewer
    (100, 32, 8, [2049, 2048, 4000, 5], 0, 1),                        # two tree tiles
    (60, 32, 8, [20000, 8449], 0, 4),                                 # 79 tiles a split; 34, the last one 31 and the tree's
    (60, 64, 8, [28000], 0, 4),                                       # 110 tiles a split
    (60, 32, 8, [6000 - 601 * b for b in range(10)], -1, 1),          # more than one wave, FOLLOW
    (60, 32, 8, [1473, 1536, 1537, 1600, 1472, 64, 1, 0, 500, 512], -1, 0),    # the same, shorter
    (60, 32, 32, [1473, 1472, 4000], 0, 1),                           # one query block per head: 96 CTAs
    (30, 32, 8, [28000], 0, 8), (30, 32, 8, [4000 - 400 * b for b in range(10)], 0, 1),    # 64 and 80
    (30, 32, 8, [3008] * 10, 0, 0), (16, 32, 32, [3100, 2400, 1, 64], 0, 0),    # 48 tiles; 128 CTAs
])
def test_query_rows_from_either_memory(nodes, hq, hkv, lens, kernel, splits):
    assert splits_with_q_in_tensor_memory(len(lens), nodes, hq, hkv, max(lens)) == splits
    check(nodes, hq, hkv, lens, kernel)
