"""The argument types the binding declares are those of include/sfs.h, and a call without a stream takes the current one."""
import os
import re

import pytest

from paper_2506_10848_b200 import binding as sfs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_declared_arguments_are_the_headers():
    text = re.sub(r"/\*.*?\*/", "", open(os.path.join(ROOT, "include", "sfs.h")).read(), flags=re.S)
    kind = {"int32_t": "i", "uint32_t": "i", "int64_t": "l", "float": "f"}
    seen = 0
    for m in re.finditer(r"\w+\s*\*?\s*\b(sfs_\w+)\(([^;]*?)\);", text):
        args = [a.replace("const ", "").strip() for a in m.group(2).split(",") if a.strip() not in ("", "void")]
        want = "".join("p" if "*" in a else kind[a.split()[0]] for a in args)
        if want:
            assert sfs._PROTOTYPES[m.group(1)] == want, m.group(1)
            seen += 1
    assert seen == len(sfs._PROTOTYPES)


@pytest.mark.gpu
def test_no_stream_means_the_current_one():
    import torch
    default = torch.cuda.current_stream().cuda_stream
    other = torch.cuda.Stream()
    for _ in range(2):                                      # the first call, and those after it
        assert sfs._stream(None) == default
        with torch.cuda.stream(other):
            assert sfs._stream(None) == other.cuda_stream
    assert sfs._stream(other) == other.cuda_stream and sfs._stream(7) == 7
