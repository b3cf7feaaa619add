"""Step 1's set kernels at the edges of their ranges: log B of every family
against the oracle, and the joint-state counts of large families.

A score is a sum of at most 2 min(cells, m) nonzero terms lgamma(a + N) -
lgamma(a): the oracle rounds each to a few units in the last place of
lgamma(m), the library to 2^-(S+1) (S = 61 - ceil(log2(2 m L + 1)), at most
52, L = max |ln(a + t)|); both sums of that many terms are bounded below.
"""
import math

import numpy as np
import pytest

from oracle import oracle as orc
from paper_1408_1664_gb300 import binding as B
from paper_1408_1664_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with B.Context(0) as c:
        yield c


def _bound(m, cells):
    terms = 2 * min(cells, m) + 2
    ulp = 2.0 ** -52 * max(1.0, m * math.log(m + 2.0))
    L = max(math.log(m + 1.0), math.log(65536.0))
    S = min(52, 61 - math.ceil(math.log2(2 * m * L + 1)))
    return terms * (4 * ulp + 2.0 ** -(S + 1))


@pytest.mark.parametrize("n,m,arity,d", [
    (5, 63, 2, 4), (6, 64, 2, 5), (7, 65, 2, 5),       # a set per thread, the first per warp
    (11, 129, 2, 10), (12, 40, 2, 11),                 # 10 variables by a warp, 11 and 12 by a block
    (2, 1, 2, 1), (3, 0, 2, 2),
    (7, 1001, 3, 5), (8, 33, 3, 7),                    # 729 states by a warp, 2187 and 6561 by a block
    (6, 777, [5, 4, 4, 4, 3, 4], 4),                   # 1280 states: the block histogram
    (6, 257, 7, 4), (6, 120, 8, 4),                    # 16807 and 32768 states: neither histogram
    (4, 500, [255, 2, 3, 30], 1), (5, 50, [1, 2, 1, 3, 4], 3),
    (8, 30000, 3, 2), (6, 30001, 2, 5),                # data beyond one block's shared memory
])
def test_log_scores_and_counts(ctx, n, m, arity, d):
    ds = datagen.random_dag_data(n, m, arity, min(d, 3), 1.0, seed=n * 1000 + m)
    masks, logB = ctx.scores(ds.data, ds.arity, d)
    om, ol = orc.scores(ds.data, ds.arity, d)
    np.testing.assert_array_equal(masks, om)
    cells = int(np.prod(np.sort(ds.arity.astype(np.int64))[::-1][:d + 1]))
    assert np.abs(logB - ol).max() <= _bound(m, cells)
    rng = np.random.default_rng(m)
    job = B.Job(ds.data, ds.arity, d)
    for k in {0, d // 2, d}:
        i = int(rng.integers(n))
        G = sum(1 << int(p) for p in rng.choice([p for p in range(n) if p != i], size=k, replace=False))
        want = orc.family_counts(ds.data, ds.arity, i, G)
        np.testing.assert_array_equal(B.bn_debug_counts(ctx.h, job, i, G, want.shape[0]), want)


def test_invalid_device_data_is_reported(ctx):
    """Device data is checked on the GPU: a value not below its arity gives
    BN_EINVAL, whatever state numbers it would form."""
    import torch
    ds = datagen.random_dag_data(7, 300, 3, 3, 1.0, seed=5)
    bad = ds.data.copy()
    bad[17, 2] = 255
    bad[290, 6] = 3
    with pytest.raises(B.BnError) as e:
        B.bn_scores(ctx.h, B.Job(torch.from_numpy(bad).cuda(), ds.arity, 4))
    assert e.value.code == B.BN_EINVAL
    masks, logB = ctx.scores(ds.data, ds.arity, 4)     # the context still works
    np.testing.assert_allclose(logB, orc.scores(ds.data, ds.arity, 4)[1], atol=1e-10, rtol=0)
