"""Column sums of the up-zeta where a column's chunks lie in a cluster's
blocks (13 and more high dimensions): the same job in a batch's persistent
launch (whole columns, one block each) gives the same bits; past the sizes a
batch takes, FP32 against FP64 within the FP32 tolerance."""
import numpy as np
import pytest

from paper_1408_1664_gb300 import binding as B
from paper_1408_1664_gb300 import datagen

pytestmark = pytest.mark.gpu


def _data(n, dependent):
    ds = datagen.random_dag_data(n, 400, 2, 2, 1.0, seed=600 + n)
    data = ds.data.copy()
    if dependent:                     # columns wider than one window
        data[:, n - 1] = data[:, 0]
        data[:, 3] = data[:, 17]
    return data, ds.arity


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,d,dependent", [(26, 2, False), (27, 1, False), (27, 2, True), (27, 3, False)])
def test_chunked_columns_equal_whole_ones(n, d, dependent, precision):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    data, arity = _data(n, dependent)
    with B.Context(0, autotune=False) as ctx:
        alone, lpd = ctx.edge_posteriors(data, arity, d, precision=precision)
        with B.Batch(ctx.h, [B.Job(data, arity, d, precision=precision)]) as batch:
            batch.run()
            post, lpd1 = batch.results(0)
    assert np.all(np.isfinite(alone))
    assert np.array_equal(post, alone) and lpd1 == lpd


@pytest.mark.parametrize("n,d", [(28, 2), (29, 2)])
def test_chunked_columns_fp32_against_fp64(n, d):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    data, arity = _data(n, True)
    p = {}
    for f in ("fp32", "fp64"):
        with B.Context(0) as ctx:
            p[f] = ctx.edge_posteriors(data, arity, d, precision=f)[0]
    np.testing.assert_allclose(p["fp32"], p["fp64"], atol=1e-4, rtol=0)
