"""katz_certify_topk_noalloc after its device array was left in any state (as
calls that overlapped leave it): no word of it is an index outside it.  The
array is not reachable from outside the library, so the entry point's source
is compiled once more here, with a function of its own."""
import ctypes
import os
import subprocess

import pytest

from paper_1807_03847_gb300 import build as B

SOURCE = """
#include "%s"
extern "C" unsigned place(unsigned word) { return place_of(word); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("noalloc")
    (d / "filled.cu").write_text(SOURCE % os.path.join(B.CSRC, "katz_noalloc.cu"))
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", "-o", str(d / "filled.so"), str(d / "filled.cu")],
                   check=True)
    so = ctypes.CDLL(str(d / "filled.so"))
    so.place.argtypes, so.place.restype = [ctypes.c_uint], ctypes.c_uint
    return so


def test_words_of_the_order_stay_within_the_candidates(lib):
    cap = 8192
    assert [lib.place(w) for w in (0, 1, cap - 1)] == [0, 1, cap - 1]
    assert all(lib.place(w) < cap for w in (cap, 3 * 10**9, 0x7fffffff, 0xbff00000, 0xffffffff))
