"""The renaming of the column array with tiles of every size its warps take, at
totals of rows plus arcs around a multiple of the tile and of its limits: s_2 =
alpha (A s_1) against the degrees summed in exact integers.  Tolerance: three
roundings of 2^-53 each side, 6 x 2^-53 < 1e-15."""
import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu

WARPS = 152 * 48  # a tile size needs as many tiles of it, or the next smaller one is taken


@pytest.mark.parametrize("tile", [128, 256, 512, 1024])
@pytest.mark.parametrize("extra", [-1, 0, 1, 77])
def test_every_tile_size(tile, extra):
    import paper_1807_03847_gb300 as K

    total = tile * WARPS + extra if tile > 128 else 128 * 5000 + extra
    rng = np.random.default_rng(tile + extra)
    m = total // 3
    n0 = max(m // 8, 2)
    base = gg.from_edges(n0, rng.integers(0, n0, m), (rng.random(m) ** 3 * n0).astype(np.int64))
    n = total - base.nnz  # rows without arcs at the end
    assert n >= n0
    rowptr = torch.from_numpy(np.concatenate([base.rowptr, np.full(n - n0, base.nnz, np.int64)])).cuda()
    col = torch.from_numpy(base.col).cuda()
    h = K.Katz(rowptr, col, K.katz_default_opts(r_max=2))
    assert h.rank(0.0, 1, 1e-300, check=False).r == 2
    deg = rowptr[1:] - rowptr[:-1]
    two = torch.zeros(n, dtype=torch.int64, device="cuda")
    two.index_add_(0, torch.repeat_interleave(torch.arange(n, device="cuda"), deg), deg[col.long()])
    a = 1.0 / (int(deg.max()) + 1)
    np.testing.assert_allclose(h.walk(1), a * deg.cpu().numpy(), rtol=1e-15)
    np.testing.assert_allclose(h.walk(2), a * a * two.cpu().numpy(), rtol=1e-15)
    h.close()
