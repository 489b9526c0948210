"""The ranking criterion on a handle restored from a checkpoint, whatever the
handle ranked by before it: the order of the handle that was saved."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("first", ["ranking", "pair", "topk"])
@pytest.mark.parametrize("n", [2, 700, 5000])
def test_restored_handle_ranks_again(first, n):
    import paper_1807_03847_gb300 as K

    g = gg.erdos_renyi(n, 8 * n, 5) if n > 2 else gg.path(2)
    h = K.Katz(g.rowptr, g.col, K.katz_default_opts(r_max=40))
    if first == "topk":
        h.rank(0.0, min(n, 10), 1e-9, check=False)
    else:
        h.rank_by(K.KATZ_CRIT_RANKING if first == "ranking" else K.KATZ_CRIT_PAIR, eps=1e-7, pair=(0, 1), check=False)
    h2 = K.Katz.restore(h.checkpoint())
    orders = []
    for x in (h, h2):
        x.rank_by(K.KATZ_CRIT_RANKING, eps=1e-7, check=False)
        orders.append(x.ranking(n).copy())
        x.close()
    np.testing.assert_array_equal(*orders)
