"""Histograms of the joint states over chunks of samples, for data beyond one
block's shared memory: sizes around the first and second chunk, ragged sample
counts, several sets per group and round, warp and block histograms, batch
jobs of unequal sample counts in one group.  Counts are exact; the scores' bound
is that of test_gpu_set_scores.py (the same sums)."""
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
    (20, 9601, 3, 2), (20, 9830, 3, 3), (26, 7540, 3, 1), (26, 7549, 3, 1),
    (8, 24001, 3, 3), (8, 49999, 3, 7), (5, 100002, 3, 4),
    (6, 70003, [5, 4, 4, 4, 3, 4], 4), (5, 50000, 6, 4), (3, 65537, [30, 2, 255], 2),
    (12, 30001, 2, 11),
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


@pytest.mark.parametrize("graph", [True, False])
def test_batch_jobs_of_unequal_sample_counts(ctx, graph):
    jobs = [B.Job(ds.data, ds.arity, 3, precision="fp32")
            for ds in (datagen.random_dag_data(9, m, 3, 3, 1.0, seed=m) for m in (40001, 1, 21900, 300))]
    with B.Context(0, autotune=False, graph_batch=graph) as c, B.Batch(c.h, jobs) as batch:
        batch.run()
        for k, job in enumerate(jobs):
            post, lpd = B.bn_edge_posteriors(ctx.h, job)
            got, got_lpd = batch.results(k)
            np.testing.assert_array_equal(got, post)
            assert got_lpd == lpd
