"""Where a CTA of tree_attn_umma_kernel takes the query rows from: shared memory up to 31 tiles, tensor memory from the ninth tile on above, in the launches for
which that is faster (`splits`: of such a launch, 0 for the others; see attn_route).  CTAs on both sides of that line in
one launch, tree tiles at the end, splits of which some are long, against the reference and bounds of the launches that other tests make."""
import pytest

from attn_route import splits_with_q_in_tensor_memory
from test_gpu_attn_choice import test_room_in_the_cache_does_not_matter as check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nodes,hq,hkv,lens,kernel,splits", [
    (60, 32, 8, [1920] * 3 + [1919, 64, 1, 0], 0, 0),                 # at most 30 tiles and the tree's
    (60, 32, 8, [1984, 1921, 1920, 1856, 64, 1, 0], 0, 1),            # 32 and 31 with the tree's, and fewer
    (100, 32, 8, [1857, 1856, 4000, 5], 0, 1),                        # two tree tiles
    (60, 32, 8, [20000, 7681], 0, 4),                                 # 79 tiles a split; 31, the last one 28 and the tree's
    (60, 64, 8, [28000], 0, 4),                                       # 110 tiles a split
    (60, 32, 8, [6000 - 601 * b for b in range(10)], -1, 1),          # more than one wave, FOLLOW
    (60, 32, 8, [1473, 1536, 1537, 1600, 1472, 64, 1, 0, 500, 512], -1, 0),    # the same, shorter
    (60, 32, 32, [1473, 1472, 4000], 0, 0),                           # one query block per head
])
def test_query_rows_from_either_memory(nodes, hq, hkv, lens, kernel, splits):
    assert splits_with_q_in_tensor_memory(len(lens), nodes, hq, hkv, max(lens)) == splits
    check(nodes, hq, hkv, lens, kernel)
