"""The top-k of a level around the sizes where the select changes its way: few
candidates (ranked as they are), a filtered list, and more equal bounds than
that list holds.  The order (lower bound desc, id asc) is unique, so the ids
are those of a sort of the returned bounds, exactly."""
import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu

DIRECT, CAP = 1024, 8192


def _ring_with_hub(n):  # n tied nodes and one hub
    u = np.arange(n)
    return gg.from_edges(n + 301, np.concatenate([u, np.full(300, n)]),
                         np.concatenate([(u + 1) % n, np.arange(n + 1, n + 301)]))


@pytest.mark.parametrize("r_max", [1, 2, 4])
@pytest.mark.parametrize("k", [1, 32, DIRECT, CAP])
@pytest.mark.parametrize("n", [3, DIRECT - 1, DIRECT, DIRECT + 1, CAP - 1, CAP, CAP + 1, 30011])
def test_tied_candidates(n, k, r_max):
    _check(_ring_with_hub(n), k, r_max)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k", [10, 1500, CAP])
@pytest.mark.parametrize("graph", ["rmat", "er", "directed", "mostly-empty"])
def test_spread_candidates(graph, k, precision):
    g = {"rmat": lambda: gg.rmat(15, 16, seed=3), "er": lambda: gg.erdos_renyi(40000, 320000, seed=4),
         "mostly-empty": lambda: gg.from_edges(30000, np.arange(900), (np.arange(900) * 7 + 1) % 1000),
         "directed": lambda: gg.orient(gg.rmat(15, 16, seed=5), 6)}[graph]()
    for r_max in (1, 2, 3, 7):
        _check(g, k, r_max, precision, undirected=0 if graph == "directed" else 1)


def _check(g, k, r_max, precision=0, undirected=1):
    import paper_1807_03847_gb300 as K

    h = K.Katz(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.col).cuda(),
               K.katz_default_opts(r_max=r_max, precision=precision, undirected=undirected))
    info = h.rank(0.0, k, 1e-9, check=False)
    lo, _, _ = h.bounds()
    kk = min(k, g.n)
    assert np.array_equal(h.ranking(kk), np.lexsort((np.arange(g.n), -lo))[:kk])
    empty = np.diff(g.rowptr) == 0  # rows the later levels leave alone
    assert not h.walk(info.r)[empty].any() and not lo[empty].any()
    h.close()
