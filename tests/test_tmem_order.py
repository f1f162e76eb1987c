"""Tensor memory that MMAs have read is written again only behind a fence: tcgen05 operations are not ordered by the wait on a barrier
that a tcgen05.commit signals, but by tcgen05.fence::after_thread_sync behind it.  Nothing shows when the order happens to hold, so
the sources are read."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1706_09453_b200", "csrc")


def test_stores_behind_a_wait_on_a_free_slot_are_fenced():
    seen = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        lines = [line.split("//")[0] for line in open(path)]
        for i, line in enumerate(lines):
            if not re.search(r"\btmem_st\d+\(", line) or "__device__" in line:
                continue
            waits = [j for j in range(max(0, i - 60), i) if "warp_wait(" in lines[j] and "empty" in lines[j]]
            if not waits:        # the block scales, which are written once
                continue
            seen += 1
            assert any("tc_fence_after_sync()" in x for x in lines[waits[-1]:i]), "%s:%d" % (os.path.basename(path), i + 1)
    assert seen >= 6
