"""The renaming of the column array at create (tiles of rows plus arcs).

s_2 = alpha (A s_1) with s_1 = alpha deg reads every arc once, so it is
checked against the degrees summed in exact integers.  Tolerance: s_1, the
row sum and the last product are rounded once each (2^-53 relative), and the
reference's two products and quotient once each: 6 x 2^-53 < 1e-15.
"""
import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu

TILE = 1024  # rows plus arcs per warp of the renaming kernel


def _graph(kind):
    if kind.startswith("items"):  # a cycle and isolated rows: 3 items a node, 1 a row; totals around tile edges
        total = TILE * 3 + int(kind[5:])
        m = total // 6
        u = np.arange(m)
        g = gg.from_edges(m + total - 3 * m, u, (u + 1) % m)
        assert g.n + g.nnz == total
        return g
    if kind == "hubs-first":  # neighbouring hub rows, far longer than a tile, then short and empty rows
        rng = np.random.default_rng(5)
        hub, leaf = np.repeat(np.arange(7), 5000), rng.integers(7, 40000, 35000)
        return gg.from_edges(60000, hub, leaf)
    if kind == "empty-ends":  # only the middle rows have arcs
        u = np.arange(20000, 20300)
        return gg.from_edges(41000, u, u + 300)
    return gg.rmat(18, 16, seed=gg.SEED_BASE + 18)  # above the size that arrives in slices from host memory


@pytest.mark.parametrize("host", [True, False])
@pytest.mark.parametrize("kind", ["items-1", "items0", "items1", "hubs-first", "empty-ends", "rmat18"])
def test_every_arc_reaches_its_renamed_row(kind, host):
    import paper_1807_03847_gb300 as K

    g = _graph(kind)
    rowptr, col = torch.from_numpy(g.rowptr), torch.from_numpy(g.col)
    if not host:
        rowptr, col = rowptr.cuda(), col.cuda()
    h = K.Katz(rowptr, col, K.katz_default_opts(r_max=2))
    info = h.rank(0.0, 1, 1e-300, check=False)
    assert info.r == 2
    deg = np.diff(g.rowptr)
    rows = np.repeat(np.arange(g.n), deg)
    two = np.zeros(g.n, np.int64)
    np.add.at(two, rows, deg[g.col])
    a = 1.0 / (deg.max() + 1)
    np.testing.assert_allclose(h.walk(1), a * deg, rtol=1e-15)
    np.testing.assert_allclose(h.walk(2), a * a * two, rtol=1e-15)
    h.close()


@pytest.mark.parametrize("at", [0, 700, -1])
def test_a_column_out_of_range_is_still_refused(at):
    import paper_1807_03847_gb300 as K

    g = _graph("items0")
    col = g.col.copy()
    col[at] = g.n
    with pytest.raises(K.KatzError) as e:
        K.Katz(g.rowptr, col)
    assert e.value.name == "KATZ_EINVAL"
