"""Staged gathers are for graphs whose gathers miss L2: a graph whose ids are near
its neighbours' keeps plain gathers however large it is, new and restored, and
ranks to the same bits either way.  katz_opts.keep_history = 1 never stages."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MIN_N = 1 << 25  # smallest graph with staged gathers


def _within(n, m, reach, undirected):
    """m pairs (u, u + d mod n), 1 <= d < reach."""
    g = torch.Generator(device="cuda")
    g.manual_seed(reach)
    u = torch.randint(0, n, (m,), generator=g, device="cuda")
    v = (u + torch.randint(1, reach, (m,), generator=g, device="cuda")) % n
    keys = torch.unique(torch.cat([(u << 31) | v, (v << 31) | u]) if undirected else (u << 31) | v)
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(keys >> 31, minlength=n), 0, out=rowptr[1:])
    col = (keys & 0x7fffffff).int()
    torch.cuda.synchronize()
    return rowptr, col


@pytest.mark.parametrize("n,reach,undirected,offsets64,staged", [
    (MIN_N, 2, 1, 0, False), (MIN_N + 3, 100, 1, 0, False), (MIN_N + 8191, 1 << 20, 1, 1, False),
    (MIN_N + 1, 1 << 10, 0, 0, False), (MIN_N + 17, 1 << 24, 1, 0, True), (MIN_N + 5, 1 << 25, 0, 0, True)])
def test_local_graphs_keep_plain_gathers(n, reach, undirected, offsets64, staged):
    import paper_1807_03847_gb300 as K

    rowptr, col = _within(n, 80_000_000, reach, undirected)
    out = []
    for history in (0, 1):
        h = K.Katz(rowptr, col, K.katz_default_opts(undirected=undirected, offsets64=offsets64, keep_history=history,
                                                    r_max=4))
        info = h.rank(0.0, 50, 1e-300, check=False)
        lower = torch.empty(n, dtype=torch.float64, device="cuda")
        upper = torch.empty_like(lower)
        K.katz_get_bounds(h.h, lower=lower, upper=upper)
        out.append((info.r, info.launches, h.ranking(50), lower, upper))
        if not history:
            h2 = K.Katz.restore(h.checkpoint())
            # a restored handle's threshold before the loop takes one kernel more
            assert h2.rank(0.0, 50, 1e-300, check=False).launches == info.launches + 1
            h2.close()
        h.close()
    a, b = out
    assert a[0] == b[0] and np.array_equal(a[2], b[2])
    assert (a[1] > b[1]) == staged
    assert torch.equal(a[3], b[3]) and torch.equal(a[4], b[4])
