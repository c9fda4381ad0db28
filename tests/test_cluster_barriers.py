"""The cluster's barrier in its aligned form is one instruction of a whole warp: wherever the kernels issue it, the lanes are gathered first."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_10848_b200", "csrc")


def test_lanes_are_gathered_before_every_aligned_cluster_barrier():
    found = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu*"))):
        for i, line in enumerate(open(path).read().split("\n"), 1):
            at = line.find("barrier.cluster.")
            if at < 0:
                continue
            found += 1
            # on the same line: nothing can come between
            assert re.search(r"(__syncwarp\(\)|cluster_arrive(_relaxed)?\(\));\s*asm volatile\(\"$", line[:at]), (os.path.basename(path), i)
    assert found >= 4
