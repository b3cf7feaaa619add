"""The persistent up-zeta tiles on both sides of their choice of blocks per SM
(by the number of samples and d): the same bits as the per-tile kernel, which a
batch of two jobs takes."""
import numpy as np
import pytest

from paper_1408_1664_gb300 import binding as B
from paper_1408_1664_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d,m", [(14, 3, 800), (15, 4, 800), (15, 4, 801), (17, 5, 801), (16, 5, 790), (16, 6, 790)])
def test_alone_equals_batch(n, d, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ds = datagen.random_dag_data(n, m, 2, 3, 1.0, seed=m + n)
    job = B.Job(ds.data, ds.arity, d, precision="fp32")
    with B.Context(0, autotune=False, graph_batch=True) as ctx:
        post, lpd = B.bn_edge_posteriors(ctx.h, job)
        with B.Batch(ctx.h, [job, job]) as batch:
            batch.run()
            want, want_lpd = batch.results(1)
    np.testing.assert_array_equal(post, want)
    assert lpd == want_lpd
