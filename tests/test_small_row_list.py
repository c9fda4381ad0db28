"""Which entries of a row list the small models' LM head reads: a caller's list may have exactly as many entries as the device's row
count says, far fewer than the call's bound.  The index functions of the kernel, compiled for the host."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_10848_b200", "csrc")
CODE = r"""
#include "small_gemm.cuh"
extern "C" void entries(int known, int M, int m, int has_list, int *out)
{
    static int32_t list[1];
    sfs::SmallGemmArgs g{};
    g.rows = has_list ? list : nullptr; g.rows_known = known;
    out[0] = sfs::list_entry_early(g, m); out[1] = sfs::list_entry_late(g, m, M);
}
"""


@pytest.fixture(scope="module")
def entries(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    (d / "e.cpp").write_text(CODE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", "/usr/local/cuda/include", "-o", str(d / "e.so"), str(d / "e.cpp")], check=True)
    lib = ctypes.CDLL(str(d / "e.so"))

    def f(known, M, m, has_list=True):
        out = (ctypes.c_int * 2)()
        lib.entries(known, M, m, int(has_list), out)
        return list(out)
    return f


@pytest.mark.parametrize("bound", [1, 31, 32, 33, 96])
def test_no_entry_beyond_the_count_is_read_and_every_one_below_it_is(entries, bound):
    for M in sorted({0, 1, bound // 2, bound}):
        for known in (0, bound):                               # a caller's list with a count, without one (or the session's own)
            there = max(M, known)
            for m in range((bound + 31) // 32 * 32):           # whole row tiles
                read = [e for e in entries(known, M, m) if e >= 0]
                assert all(e == m and e < there for e in read)
                assert len(read) == 1 if m < M else len(read) <= 1
                assert entries(known, M, m, has_list=False) == [-1, -1]
