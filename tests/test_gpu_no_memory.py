"""Calls that find no device memory return KATZ_ENOMEM and leave the handle as it
was: the same call succeeds once there is memory again.  Each case is a process
of its own that holds nearly all of the device's free memory for a while."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

N = 1 << 24
PAIRS = 1 << 25


def _csr(keys):
    import torch

    rowptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(keys >> 31, minlength=N), 0, out=rowptr[1:])
    return rowptr, (keys & 0x7fffffff).int()


def _both(u, v):
    import torch

    return torch.unique(torch.cat([(u << 31) | v, (v << 31) | u])[torch.cat([u != v, u != v])])


def _pairs(m, seed):
    import torch

    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (torch.randint(0, N, (m,), generator=g, device="cuda") for _ in range(2))


def _fill(leave):
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def child(kind):
    import numpy as np
    import torch

    import paper_1807_03847_gb300 as K

    keys = _both(*_pairs(PAIRS, 1))
    opts = dict(keep_history=1, r_max=16, deg_bound=64)
    h = K.Katz(*_csr(keys), K.katz_default_opts(**opts))
    if kind == "rank":
        held = _fill(64 << 20)
        for _ in range(2):
            with pytest.raises(K.KatzError) as e:
                h.rank(0.0, 100, 1e-9)
            assert e.value.name == "KATZ_ENOMEM"
        del held
        torch.cuda.empty_cache()
        torch.empty(1 << 20, device="cuda").zero_()  # the program's own work goes on
    h.rank(0.0, 100, 1e-9)
    if kind == "update":
        a, b = (x.int().cpu().numpy() for x in _pairs(1000, 2))  # new edges, as good as surely
        one = np.ones(1000, np.uint8)
        held = _fill(64 << 20)
        for _ in range(2):
            with pytest.raises(K.KatzError) as e:
                h.update(a, b, one)
            assert e.value.name == "KATZ_ENOMEM"
        del held
        torch.cuda.empty_cache()
        h.update(a, b, one)
        keys = torch.unique(torch.cat([keys, _both(*_pairs(1000, 2))]))
    ref = K.Katz(*_csr(keys), K.katz_default_opts(**opts))
    ref.rank(0.0, 100, 1e-9)
    assert np.array_equal(h.ranking(100), ref.ranking(100))


@pytest.mark.parametrize("kind", ["rank", "update"])
def test_call_without_memory_then_with_it(kind):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, os.path.abspath(__file__), kind], capture_output=True, text=True, timeout=300,
                       env={**os.environ, "PYTHONPATH": root})
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-3000:]


if __name__ == "__main__":
    child(sys.argv[1])
