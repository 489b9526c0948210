"""katz_certify_topk_noalloc after its device array was left in any state (as
calls that overlapped leave it): the next call, alone, is right again, and no
word of the array is an index outside it.  The array is not reachable from
outside the library, so the entry point's source is compiled once more here,
with functions of its own."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_1807_03847_gb300 import build as B

SOURCE = """
#include "%s"
#include <cstddef>
extern "C" unsigned place(unsigned word) { return place_of(word); }
extern "C" int fill_scratch(int byte, unsigned ticket) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc) != cudaSuccess) return 1;
    if (cudaMemset(p, byte, sizeof(NoAllocScratch)) != cudaSuccess) return 2;
    return cudaMemcpy((char*)p + offsetof(NoAllocScratch, ticket), &ticket, sizeof(ticket), cudaMemcpyHostToDevice);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("noalloc")
    (d / "filled.cu").write_text(SOURCE % os.path.join(B.CSRC, "katz_noalloc.cu"))
    subprocess.run([B._nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-shared", "-o", str(d / "filled.so"), str(d / "filled.cu")],
                   check=True)
    so = ctypes.CDLL(str(d / "filled.so"))
    so.katz_certify_topk_noalloc.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64,
                                             ctypes.c_double, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    so.fill_scratch.argtypes = [ctypes.c_int, ctypes.c_uint]
    so.place.argtypes, so.place.restype = [ctypes.c_uint], ctypes.c_uint
    return so


def test_words_of_the_order_stay_within_the_candidates(lib):
    cap = 8192
    assert [lib.place(w) for w in (0, 1, cap - 1)] == [0, 1, cap - 1]
    assert all(lib.place(w) < cap for w in (cap, 3 * 10**9, 0x7fffffff, 0xbff00000, 0xffffffff))


@pytest.mark.gpu
@pytest.mark.parametrize("byte,ticket", [(0, 1), (0, 37), (0, 127), (0xff, 500), (0xff, 0xffffffff)])
@pytest.mark.parametrize("n,k,kind", [(5000, 10, "random"), (300007, 700, "random"), (30000, 50, "equal"),
                                      (100003, 5000, "random")])
def test_first_call_after_any_state(lib, byte, ticket, n, k, kind):
    rng = np.random.default_rng(n)
    lower = rng.random(n) if kind == "random" else np.full(n, 0.5)
    order = np.lexsort((np.arange(n), -lower))
    x = torch.from_numpy(lower).cuda()
    ids = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    cert = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    assert lib.fill_scratch(byte, ticket) == 0
    assert lib.katz_certify_topk_noalloc(x.data_ptr(), x.data_ptr(), n, k, 1e-12, ids.data_ptr(), cert.data_ptr(),
                                         torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    assert np.array_equal(ids.cpu().numpy(), order[:k])
    top, rest = order[:k], order[k:]
    ok = np.all(lower[top[1:]] - 1e-12 < lower[top[:-1]]) and np.all(lower[rest] - 1e-12 < lower[top[-1]])
    assert int(cert) == int(ok)
