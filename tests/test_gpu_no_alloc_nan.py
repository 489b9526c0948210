"""katz_certify_topk_noalloc on bounds that are mostly NaN with the sign bit set
(x86's default NaN): they order below every number, by id among themselves."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,real,k", [(10000, 50, 100), (10000, 0, 4096), (300007, 400, 700), (8192, 3, 100)])
def test_bounds_that_are_mostly_no_numbers(n, real, k):
    import paper_1807_03847_gb300 as K

    rng = np.random.default_rng(n + k)
    bits = np.full(n, 0xfff8000000000000, np.uint64)
    bits[rng.choice(n, real, replace=False)] = (rng.random(real) + 1.0).view(np.uint64)
    key = np.where(bits >> np.uint64(63), ~bits, bits | np.uint64(1 << 63))
    order = np.lexsort((np.arange(n), -key.astype(np.float64)))  # two kinds of keys far apart: exact enough
    order[:real] = sorted(order[:real], key=lambda v: -int(key[v]))
    x = torch.from_numpy(bits.view(np.float64)).cuda()
    ids = torch.full((k,), -1, dtype=torch.int32, device="cuda")
    cert = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    K.katz_certify_topk_noalloc(x, x, k, 1e-9, ids, cert, torch.cuda.current_stream())
    assert np.array_equal(ids.cpu().numpy(), order[:k])
