"""A kernel releases the launches behind it only after its own dependent-launch wait: what it releases earlier becomes resident before its
input is on its way, beside a kernel that is two launches before it."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_10848_b200", "csrc")


def test_no_kernel_releases_its_successors_before_its_wait():
    kernels = 0
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        for body in re.split(r"__global__", open(path).read())[1:]:
            wait, trigger = body.find("pdl_wait();"), body.find("pdl_trigger();")
            if trigger >= 0:
                kernels += 1
                assert 0 <= wait < trigger, (os.path.basename(path), body[:120])
    assert kernels > 10
