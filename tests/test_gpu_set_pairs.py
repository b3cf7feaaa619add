"""Counts and scores of binary families whose sets come from bases (7 to 10
variables: bases of 5 to 8), and from m = 65536 on set by set, against the
oracle; the counts are whole numbers, the scores within the set scores'
bound."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_1408_1664_gb300 import binding as B
from paper_1408_1664_gb300 import datagen
from test_gpu_set_scores import _bound

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,d", [(7, 65, 6), (8, 100, 6), (11, 129, 6), (10, 33, 7), (12, 200, 8),
                                   (10, 0, 9), (12, 57, 9), (8, 65535, 6), (8, 65536, 6)])
def test_scores_and_counts(n, m, d):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ds = datagen.random_dag_data(n, m, 2, 3, 1.0, seed=n * 100 + m)
    rng = np.random.default_rng(m)
    with B.Context(0) as ctx:
        masks, logB = ctx.scores(ds.data, ds.arity, d)
        om, ol = orc.scores(ds.data, ds.arity, d)
        np.testing.assert_array_equal(masks, om)
        assert np.abs(logB - ol).max() <= _bound(m, 2 ** (d + 1))
        job = B.Job(ds.data, ds.arity, d)
        for k in (d, d, d - 1, d - 1, d - 2):
            i = int(rng.integers(n))
            G = sum(1 << int(p) for p in rng.choice([p for p in range(n) if p != i], size=k, replace=False))
            want = orc.family_counts(ds.data, ds.arity, i, G)
            np.testing.assert_array_equal(B.bn_debug_counts(ctx.h, job, i, G, want.shape[0]), want)
