"""The down-zeta's relevance cut under an order prior with zero factors at
large sets, against the oracle."""
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
