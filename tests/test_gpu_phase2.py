"""The down-zeta's second phase and its relevance cuts at their edges, FP32
against the FP64 path (other kernels) within the FP32 tolerance of 1e-4: the
wide column sums (from n = 22), the register transform of short and of many
columns, strongly dependent data (sums hundreds of bits below their column's
largest), and an order prior with zero factors at large sets."""
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


def _both(ctx, data, arity, d, **kw):
    p = {f: B.bn_edge_posteriors(ctx.h, B.Job(data, arity, d, precision=f, **kw))[0] for f in ("fp32", "fp64")}
    assert np.all(np.isfinite(p["fp32"])) and np.all(np.isfinite(p["fp64"]))
    np.testing.assert_allclose(p["fp32"], p["fp64"], atol=1e-4, rtol=0)


@pytest.mark.parametrize("n,d", [(22, 0), (22, 1), (22, 3), (23, 2), (17, 8), (19, 7), (14, 3), (15, 14)])
def test_fp32_against_fp64(ctx, n, d):
    ds = datagen.random_dag_data(n, 300, 2, 3, 1.0, seed=300 + n)
    _both(ctx, ds.data, ds.arity, d)


@pytest.mark.parametrize("n,d", [(22, 2), (18, 4), (16, 8)])
def test_strongly_dependent_data(ctx, n, d):
    ds = datagen.random_dag_data(n, 2000, 2, 2, 1.0, seed=400 + n)
    data = ds.data.copy()
    data[:, n - 1] = data[:, 0]
    data[:, n - 2] = data[:, 5]
    data[:, 1] = data[:, 6]
    _both(ctx, data, ds.arity, d)


@pytest.mark.parametrize("n,size", [(15, 13), (15, 14), (16, 13), (14, 13)])
def test_order_prior_with_zeros_at_large_sets(ctx, n, size):
    """q_i(S) = 0 for one node at |S| = size: the node's other sets count."""
    ds = datagen.random_dag_data(n, 200, 2, 2, 1.0, seed=500 + n)
    log_q = np.zeros((n, n))
    log_q[2, size] = -np.inf
    log_q[5, size] = -80.0
    ref = orc.edge_posteriors(ds.data, ds.arity, 2, log_q=log_q)
    for f, tol in (("fp64", 1e-9), ("fp32", 1e-4)):
        post, _ = B.bn_edge_posteriors(ctx.h, B.Job(ds.data, ds.arity, 2, precision=f, log_q=log_q))
        np.testing.assert_allclose(post, ref["post"], atol=tol, rtol=0)
