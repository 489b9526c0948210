"""katz_certify_topk_noalloc on bounds that take its candidate filter and its
radix select to their limits, against numpy on the same arrays: ids and verdict
are whole numbers and compare exactly."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GROUPS = 8192   # groups of the candidate filter
CAP = 8192      # candidates held


def _check(lower, k, eps=1e-9, width=0.0):
    import paper_1807_03847_gb300 as K

    upper = lower + width
    n = len(lower)
    ids = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    cert = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    K.katz_certify_topk_noalloc(torch.from_numpy(lower).cuda(), torch.from_numpy(upper).cuda(), k, eps, ids, cert,
                                torch.cuda.current_stream())
    order = np.lexsort((np.arange(n), -lower))
    assert np.array_equal(ids.cpu().numpy(), order[:k])
    top, rest = order[:k], order[k:]
    ok = np.all(upper[top[1:]] - eps < lower[top[:-1]]) and np.all(upper[rest] - eps < lower[top[-1]])
    assert int(cert) == int(ok)


@pytest.mark.parametrize("n,k", [(1, 1), (2, 2), (31, 7), (GROUPS - 1, 4096), (GROUPS, 4096), (GROUPS + 1, 4097),
                                 (65536, 100), (65537, 1), (8 * 65536 + 3, 1500), (100003, CAP), (CAP, CAP)])
@pytest.mark.parametrize("order", ["random", "rising", "falling"])
def test_distinct_bounds(n, k, order):
    x = np.random.default_rng(n + k).permutation(n).astype(np.float64) / n
    x = {"random": x, "rising": np.sort(x), "falling": np.sort(x)[::-1].copy()}[order]
    _check(x, k)
    _check(x, k, width=2.0 / n)


@pytest.mark.parametrize("kind", ["equal", "few-values", "one-group", "negative", "infinite"])
@pytest.mark.parametrize("k", [1, 700, 4096, CAP])
def test_bounds_that_the_groups_do_not_separate(kind, k):
    n = 300007
    rng = np.random.default_rng(k)
    if kind == "equal":  # the radix select goes down to the ids
        x = np.full(n, 0.25)
    elif kind == "few-values":
        x = rng.integers(0, 5, n).astype(np.float64)
    elif kind == "one-group":  # all large bounds 8192 apart
        x = rng.random(n)
        x[5::GROUPS] += 10.0
    elif kind == "negative":
        x = -rng.random(n) - 1.0
        x[::3] = 0.0
    else:
        x = rng.random(n)
        x[rng.integers(0, n, 50)] = -np.inf
        x[17] = np.inf
    _check(x, k)
