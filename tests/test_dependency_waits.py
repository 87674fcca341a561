"""The entropy pass merges the parts of a row in shared memory; the first CTA of the row waits for the others with a limit, so none of them may
wait for the kernel ahead before it has sent its part.  That shows only behind a kernel that takes a second: the source is read."""
import os
import re

from paper_2505_13254_b200 import build


def test_no_part_waits_for_the_kernel_ahead_before_it_is_sent():
    text = re.sub(r"//.*", "", open(os.path.join(build.CSRC, "row_stats.cu")).read())
    body = text[text.index("quantify_cluster_kernel(const __grid_constant__"):]
    body = body[:body.index("\n}")]
    waits = [m.start() for m in re.finditer(r"pdl_wait\(\)", body)]
    sent, merged = body.index("st_async_v4"), body.index("mbar_wait_cluster(")
    # one ahead of the row's first load where the rows are not prefetched, one behind the merge where they are
    assert len(waits) == 2 and sent < merged < waits[1]
    assert re.search(r"if \(!p\.prefetch\) $", body[:waits[0]]) and re.search(r"if \(p\.prefetch\) $", body[:waits[1]])
