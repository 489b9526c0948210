"""The ranking criterion's order wherever the loop ends: the sort runs only at
the levels that may satisfy the criterion and at r_max, and its order is then
that of the returned lower bounds (ties: smaller id first).  Whole numbers: no
tolerance."""
import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r_max", [1, 2, 3, 4, 5, 9])
@pytest.mark.parametrize("graph", ["er", "rmat-directed", "path", "single"])
def test_the_order_is_that_of_the_lower_bounds_at_any_level(graph, r_max):
    import paper_1807_03847_gb300 as K

    g = {"er": lambda: gg.erdos_renyi(4099, 16000, seed=5), "path": lambda: gg.path(2049),  # path: nearly all tied
         "rmat-directed": lambda: gg.orient(gg.rmat(12, 8, seed=6), 7), "single": lambda: gg.path(1)}[graph]()
    h = K.Katz(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.col).cuda(),
               K.katz_default_opts(r_max=r_max, undirected=0 if graph == "rmat-directed" else 1))
    for _ in range(2):  # a second ranking starts over
        info = h.rank_by(K.KATZ_CRIT_RANKING, eps=1e-12, check=False)
        lo, up, _ = h.bounds()
        order = np.lexsort((np.arange(g.n), -lo))
        assert np.array_equal(h.ranking(g.n), order)
        separated = bool(np.all(up[order[1:]] - 1e-12 < lo[order[:-1]]))
        assert info.converged == separated and info.r <= r_max
        assert separated or info.r == r_max
    h.close()
