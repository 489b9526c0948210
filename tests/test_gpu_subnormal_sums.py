"""FP64 row sums whose terms reach from 2^-867 down to subnormals whose upper
word is 0, in every row mode, on full levels and on repaired rows: against
rational arithmetic, rounded once per sum and once per product.

A clique's walk counts grow as (degree alpha)^r, a two-cycle's fall as alpha^r;
rows lead into both.  Such terms are below the sum's last kept bit, so every
level is the rounding of the exact sum."""
from fractions import Fraction

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

# (arcs into the clique, arcs into two-cycles) of rows in every row mode; with these
# multiples no sum below ends in a tie that only a term below the last kept bit breaks
ROWS = [(1, 1), (4, 2), (13, 3), (1, 15), (59, 60), (4, 100), (99, 29), (90, 1500), (99, 1900), (99, 3000), (8, 4500)]


def _graph(clique, cycles, rows):
    first_row = clique + 2 * cycles
    adj = [[j for j in range(clique) if j != i] for i in range(clique)]
    adj += [[clique + (i ^ 1)] for i in range(2 * cycles)]
    rng = np.random.default_rng(1)
    for a, b in rows:
        adj.append(sorted(rng.choice(clique, a, replace=False)) + list(clique + np.arange(b)))
    rowptr = np.concatenate([[0], np.cumsum([len(x) for x in adj])]).astype(np.int64)
    return first_row, rowptr, np.concatenate(adj).astype(np.int32)


def _levels(alpha, r, clique, rows):
    """s_1..s_r of a clique node, a two-cycle node and the rows."""
    mul = lambda x: float(Fraction(alpha) * Fraction(x))
    out = [(1.0, 1.0, [1.0] * len(rows))]
    for _ in range(r):
        c, t, _ = out[-1]
        out.append((mul(float((clique - 1) * Fraction(c))), mul(t),
                    [mul(float(a * Fraction(c) + b * Fraction(t))) for a, b in rows]))
    return out[1:]


def _check(h, expected, clique, first_row):
    for level, (c, t, rows) in enumerate(expected, 1):
        s = h.walk(level)
        assert np.all(s[:clique] == c) and np.all(s[clique:first_row] == t), level
        np.testing.assert_array_equal(s[first_row:], rows, err_msg=f"level {level}")


@pytest.mark.parametrize("clique,exponent,r", [(100, 41, 27), (256, 55, 20)])
def test_terms_far_below_the_sum(clique, exponent, r):
    import paper_1807_03847_gb300 as K

    cycles, alpha = 2300, 2.0 ** -exponent
    first_row, rowptr, col = _graph(clique, cycles, ROWS)
    h = K.Katz(rowptr, col, K.katz_default_opts(undirected=0, r_max=r, keep_history=1, deg_bound=5000))
    info = h.rank(alpha, 1000, 1e-300, check=False)  # the clique's ties keep it from ending early
    assert info.r == r
    _check(h, _levels(alpha, r, clique, ROWS), clique, first_row)
    # one more two-cycle arc per row: the rows are repaired, one by one
    n_rows = len(ROWS)
    info = h.update((first_row + np.arange(n_rows)).astype(np.int32),
                    np.full(n_rows, first_row - 1, np.int32), np.ones(n_rows, np.uint8), check=False)
    assert info.r == r
    _check(h, _levels(alpha, r, clique, [(a, b + 1) for a, b in ROWS]), clique, first_row)
    h.close()
