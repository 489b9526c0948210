"""Staged gathers (walk vectors far larger than L2): the same bits as plain
gathers, on the smallest graphs that take them, at sizes whose last window is
cut short, whose directed rows leave windows empty, and with int64 offsets.
katz_opts.keep_history = 1 ranks the same graph with plain gathers."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

MIN_N = 1 << 25  # smallest graph with staged gathers


def _arcs(n, m, seed, undirected):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = torch.randint(0, n, (m,), generator=g, device="cuda")
    v = (torch.rand(m, generator=g, device="cuda", dtype=torch.float64).pow(3) * n).long()  # some hubs
    keys = (u << 31) | v
    if undirected:
        keys = torch.cat([keys, (v << 31) | u])
    keys = torch.unique(keys[u != v] if not undirected else keys[torch.cat([u != v, u != v])])
    rowptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(keys >> 31, minlength=n), 0, out=rowptr[1:])
    col = (keys & 0x7fffffff).int()
    torch.cuda.synchronize()  # the library reads them on a stream of its own
    return rowptr, col


@pytest.mark.parametrize("n,undirected,offsets64,precision", [
    (MIN_N, 1, 0, 0), (MIN_N + 8191, 1, 1, 0), (MIN_N + 1, 0, 0, 0), (MIN_N + 4097, 1, 0, 1), (MIN_N + 13, 0, 1, 1)])
def test_staged_levels_have_the_bits_of_plain_ones(n, undirected, offsets64, precision):
    import paper_1807_03847_gb300 as K

    rowptr, col = _arcs(n, 60_000_000, n, undirected)
    out = []
    for history in (0, 1):
        h = K.Katz(rowptr, col, K.katz_default_opts(undirected=undirected, offsets64=offsets64, precision=precision,
                                                    fp32_from=4 if precision else 0, keep_history=history, r_max=7,
                                                    locality=-1))
        info = h.rank(0.0, 50, 1e-300, check=False)
        lower = torch.empty(n, dtype=torch.float64, device="cuda")
        upper = torch.empty_like(lower)
        K.katz_get_bounds(h.h, lower=lower, upper=upper)
        walk = torch.empty_like(lower)
        K.katz_get_walk(h.h, info.r, out=walk)
        out.append((info.r, info.launches, h.ranking(50), lower, upper, walk))
        if not history and not precision:  # a restored handle stages again
            h2 = K.Katz.restore(h.checkpoint())
            again = h2.rank(0.0, 50, 1e-300, check=False)
            assert again.launches >= info.launches and np.array_equal(h2.ranking(50), out[0][2])
            h2.close()
        h.close()
    a, b = out
    assert a[0] == b[0] and np.array_equal(a[2], b[2])
    assert a[1] > b[1]  # the staging kernel ran
    for x, y in zip(a[3:], b[3:]):
        assert torch.equal(x, y)
