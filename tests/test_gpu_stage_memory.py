"""Staged gathers are optional memory: a call that finds no other memory takes
theirs and goes on with plain gathers, with the same results.  Each case is a
process of its own (the library keeps what its handles gave back) that, after
the create, holds all of the device's free memory but `leave` bytes."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

N = (1 << 25) + 5
ARCS = 200_000_000


def _graph():
    import torch

    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    u = torch.randint(0, N, (ARCS,), generator=g, device="cuda")
    keys = torch.unique(u << 31 | torch.randint(0, N, (ARCS,), generator=g, device="cuda"))
    rowptr = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(keys >> 31, minlength=N), 0, out=rowptr[1:])
    return rowptr, (keys & 0x7fffffff).int()


def _fill(leave):
    import torch

    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(max(torch.cuda.mem_get_info()[0] - leave, 0), dtype=torch.uint8, device="cuda")


def child(kind, leave):
    import numpy as np
    import torch

    import paper_1807_03847_gb300 as K

    graph = _graph()
    h = K.Katz(*graph, K.katz_default_opts(undirected=0, r_max=4))
    top = lambda x: (lambda i: (i.r, i.launches, x.ranking(100)))(x.rank(0.0, 100, 1e-9, check=False))
    if kind == "rank":
        held = _fill(leave)
        a = top(h)
        b = top(h)  # and again, on the loop captured anew
        assert a[:2] == b[:2] and np.array_equal(a[2], b[2])
        del held
    else:
        staged = top(h)
        held = _fill(leave)
        if kind == "sort":
            h.rank_by(K.KATZ_CRIT_RANKING, eps=1e-300, check=False)
            order = h.ranking(N)
        else:
            lower, upper, _ = K.katz_get_bounds(h.h, N)
        del held
        a = top(h)
        assert a[1] < staged[1]  # plain from here on
        if kind == "sort":
            assert np.array_equal(np.sort(order), np.arange(N))
        else:
            lo = torch.empty(N, dtype=torch.float64, device="cuda")
            K.katz_get_bounds(h.h, lower=lo, upper=torch.empty_like(lo))
            assert np.array_equal(lower, lo.cpu().numpy()) and np.all(lower <= upper)
    h.close()
    torch.cuda.empty_cache()
    h = K.Katz(*graph, K.katz_default_opts(undirected=0, r_max=4))
    c = top(h)
    h.close()
    print("launches", a[1], c[1])
    assert a[0] == c[0] and a[1] < c[1] and np.array_equal(a[2], c[2])


@pytest.mark.parametrize("kind,leave_mb", [("rank", 64), ("rank", 700), ("rank", 2048), ("sort", 64), ("bounds", 64)])
def test_calls_take_the_staged_gathers_memory(kind, leave_mb):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = subprocess.run([sys.executable, os.path.abspath(__file__), kind, str(leave_mb << 20)], capture_output=True, text=True,
                       timeout=300, env={**os.environ, "PYTHONPATH": root})
    assert p.returncode == 0, p.stdout[-2000:] + p.stderr[-3000:]


if __name__ == "__main__":
    child(sys.argv[1], int(sys.argv[2]))
