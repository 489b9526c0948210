"""Row sums at the edges of the row modes (degrees 16/17, 128/129, 2048/2049)
and of the blocks that share rows, FP64 and FP32 levels, one state and two.

FP64: s_2 = alpha (A s_1), s_1 = alpha deg, against exact integer sums;
tolerance 1e-15 (three roundings of 2^-53 each side).  FP32 level 2: the
longest chain of FP32 additions here is below 24, plus the rounding of the
inputs, of alpha and of the product: 27 x 2^-24 < 2e-6.
"""
import numpy as np
import pytest
import torch

import graphgen as gg

pytestmark = pytest.mark.gpu


def _graph(counts, seed):
    """Rows of the given {degree: count}, their neighbours random leaves."""
    rng = np.random.default_rng(seed)
    deg = np.repeat(list(counts), list(counts.values()))
    rng.shuffle(deg)
    m, leaves = len(deg), 6000
    u = np.repeat(np.arange(m), deg)
    v = np.concatenate([m + rng.choice(leaves, d, replace=False) for d in deg])
    return gg.from_edges(m + leaves, u, v)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("counts", [
    {1: 3, 15: 5, 16: 300, 17: 64, 18: 1}, {17: 65, 32: 7, 33: 70, 127: 3, 128: 129, 129: 15},
    {129: 17, 130: 1, 255: 16, 256: 33}, {2047: 2, 2048: 17, 2049: 3, 4096: 2, 4097: 1}, {5999: 1}])
def test_row_sums_at_the_mode_edges(counts, precision):
    import paper_1807_03847_gb300 as K

    g = _graph(counts, 3)
    h = K.Katz(torch.from_numpy(g.rowptr).cuda(), torch.from_numpy(g.col).cuda(),
               K.katz_default_opts(r_max=2, precision=precision, fp32_from=2 if precision else 0))
    h.rank(0.0, 1, 1e-300, check=False)
    deg = np.diff(g.rowptr)
    two = np.zeros(g.n, np.int64)
    np.add.at(two, np.repeat(np.arange(g.n), deg), deg[g.col])
    a = 1.0 / (deg.max() + 1)
    np.testing.assert_allclose(h.walk(2), a * a * two, rtol=2e-6 if precision else 1e-15)
    h.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_two_states_at_the_mode_edges(precision):
    import paper_1807_03847_gb300 as K

    g = _graph({16: 70, 17: 66, 128: 33, 129: 18, 2048: 5, 2049: 3}, 4)
    D = g.deg_max() + 8
    opts = dict(keep_history=1, deg_bound=D, precision=precision)
    first = gg.update_batch(g, 40, 1)
    batches = [first, gg.update_batch(gg.apply_batch(g, *first), 40, 2)]
    walks = []
    for pair in (0, 2):
        h = K.Katz(g.rowptr, g.col, K.katz_default_opts(**opts))
        h.rank(0.0, 20, 1e-9)
        s = K.Server(workers=1, pair_batches=pair)
        s.attach(h, 20)
        answers = [s.wait(t) for t in [s.submit(h, *b) for b in batches]]
        s.close()
        assert all(a[0] == 0 for a in answers)
        r = answers[-1][2].info.r
        walks.append([h.walk(i) for i in range(1, r + 1)] + [np.concatenate([a[1] for a in answers])])
        h.close()
    assert len(walks[0]) == len(walks[1])
    for x, y in zip(*walks):
        assert np.array_equal(x, y)  # the pass over two states has the bits of one by one



@pytest.mark.parametrize("seed,kinds", [(1, "delete"), (2, "both"), (3, "both"), (4, "insert")])
def test_rebuilt_rows_at_the_mode_edges(seed, kinds):
    """A batch that empties whole stretches of hub rows and touches first and
    last rows of every mode: the walk vectors are those of a new handle on the
    updated graph, bit for bit (exact row sums)."""
    import paper_1807_03847_gb300 as K

    g = _graph({1: 5, 16: 33, 17: 34, 128: 17, 129: 3, 2048: 2, 2049: 2, 4600: 2}, seed)
    rng = np.random.default_rng(seed)
    rows = np.repeat(np.arange(g.n), np.diff(g.rowptr))
    keep = rows < g.col
    u, v = rows[keep], g.col[keep]
    hub = int(np.argmax(np.diff(g.rowptr)))
    chosen = np.zeros(len(u), bool)
    if kinds != "insert":
        chosen |= rng.random(len(u)) < 0.05
        chosen |= (u == hub) & (v > np.median(g.col))  # most of a chunk
    src, dst = list(u[chosen]), list(v[chosen])
    ins = [0] * len(src)
    if kinds != "delete":
        present = set(zip(u.tolist(), v.tolist()))
        for a, b in rng.integers(0, g.n, (400, 2)).tolist():
            a, b = min(a, b), max(a, b)
            if a != b and (a, b) not in present:
                present.add((a, b))
                src.append(a), dst.append(b), ins.append(1)
    src, dst, ins = np.array(src, np.int32), np.array(dst, np.int32), np.array(ins, np.uint8)
    D = g.deg_max() + 64
    opts = dict(keep_history=1, deg_bound=D)
    h = K.Katz(g.rowptr, g.col, K.katz_default_opts(**opts))
    h.rank(0.0, 10, 1e-9)
    info = h.update(src, dst, ins)
    new = gg.apply_batch(g, src, dst, ins)
    fresh = K.Katz(new.rowptr, new.col, K.katz_default_opts(r_max=info.r, **opts))
    fresh.rank(0.0, 10, 1e-300, check=False)
    for i in range(1, info.r + 1):
        assert np.array_equal(h.walk(i), fresh.walk(i))
    h.close()
    fresh.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("top", [1, 62, 63, 64, 65, 700])
def test_first_level_on_both_sides_of_its_table(top, precision):
    """Level 1 is alpha deg and its bounds, of degrees in the block's table and
    past it; FP64 bounds are the formula's bits, certified ones contain it and
    are wider by a few dozen roundings at most (1e-13 relative)."""
    import paper_1807_03847_gb300 as K

    g = _graph({d: 400 // d + 2 for d in {1, 2, max(top - 1, 1), top}}, 5)
    deg = np.diff(g.rowptr)
    h = K.Katz(g.rowptr, g.col, K.katz_default_opts(r_max=1, precision=precision))
    k = 5
    for _ in range(2):  # the second pass finds the first one's buffers
        info = h.rank(0.0, k, 1e-300, check=False)
        s = info.alpha * deg.astype(np.float64)
        low, up = s + info.alpha * s, s + (info.alpha * info.gamma) * s
        lo, hi = h.bounds()[:2]
        if precision:
            assert (lo <= low * (1 + 1e-15)).all() and (hi >= up * (1 - 1e-15)).all()  # their own roundings
            np.testing.assert_allclose(lo, low, rtol=1e-13)
            np.testing.assert_allclose(hi, up, rtol=1e-13)
        else:
            assert np.array_equal(lo, low) and np.array_equal(hi, up)
        assert np.array_equal(h.walk(1), s) and np.array_equal(h.walk(0), np.ones(g.n))
        assert np.array_equal(h.ranking(k), np.lexsort((np.arange(g.n), -deg))[:k])
    h.close()
