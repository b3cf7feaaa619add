"""The linear FP64 form (values with a wide exponent instead of logarithms)
at its edges: on both sides of the range rule, on data whose values span
thousands of bits (copied variables, which also need several passes per tile),
with zero weights, and for every small n; against the oracle within the FP64
path's 1e-9.  (The start of every bound is 1e-9, the FP64 path's contract.)"""
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


def _check(ctx, data, arity, d, **kw):
    ref = orc.edge_posteriors(data, arity, d, **kw)
    post, lpd = B.bn_edge_posteriors(ctx.h, B.Job(data, arity, d, precision="fp64", **kw))
    np.testing.assert_allclose(post, ref["post"], atol=1e-9, rtol=0)
    assert abs(lpd - ref["log_PD"]) <= 1e-9 * max(1.0, abs(ref["log_PD"]))


@pytest.mark.parametrize("n,m,d", [(5, 200, 4), (6, 1900, 2), (6, 2200, 2), (12, 900, 3), (12, 1100, 3),
                                   (13, 800, 4), (14, 7500, 2), (14, 9500, 2), (15, 60, 6)])
def test_both_sides_of_the_range_rule(ctx, n, m, d):
    ds = datagen.random_dag_data(n, m, 2, 3, 1.0, seed=n + m)
    _check(ctx, ds.data, ds.arity, d)


@pytest.mark.parametrize("n,m,arity,d", [(8, 1000, 2, 3), (12, 700, 2, 2), (14, 2000, 2, 3), (16, 3000, 2, 2),
                                         (15, 1500, 3, 2)])
def test_copied_variables(ctx, n, m, arity, d):
    """Pairs and triples of identical variables: a node's score moves by
    thousands of bits with one parent, in A, F, R' and Gamma alike."""
    ds = datagen.random_dag_data(n, m, arity, 2, 1.0, seed=n)
    data = ds.data.copy()
    data[:, 1] = data[:, 0]
    data[:, n - 1] = data[:, 2]
    data[:, n - 2] = data[:, 2]
    data[:, n // 2] = data[:, 3]
    _check(ctx, data, ds.arity, d)


@pytest.mark.parametrize("n,d", [(7, 3), (13, 2), (15, 3)])
def test_zero_weights(ctx, n, d):
    """Zero weights (-inf) in the order prior and on families, the empty
    parent set of one node among them (that job keeps the logarithms)."""
    ds = datagen.random_dag_data(n, 300, 2, 2, 1.0, seed=70 + n)
    K = orc.num_families(n, d)
    rng = np.random.default_rng(n)
    log_w = np.where(rng.random((n, K)) < 0.3, -np.inf, rng.normal(0.0, 1.0, (n, K)))
    log_w[:, 0] = 0.5
    log_q = -rng.random((n, n))
    log_q[3, 2] = -np.inf
    _check(ctx, ds.data, ds.arity, d, log_q=log_q, log_w=log_w)
    log_w[2, 0] = -np.inf
    _check(ctx, ds.data, ds.arity, d, log_q=log_q, log_w=log_w)


@pytest.mark.parametrize("n,d", [(9, 3), (13, 4), (14, 4), (16, 7), (18, 5), (20, 3)])
def test_alone_equals_batch(ctx, n, d):
    """One launch for both sweeps (alone) and a launch per level (batch)."""
    ds = datagen.random_dag_data(n, 250, 2, 3, 1.0, seed=90 + n)
    job = B.Job(ds.data, ds.arity, d, precision="fp64")
    with B.Context(0, autotune=False, graph_batch=True) as c:
        post, lpd = B.bn_edge_posteriors(c.h, job)
        with B.Batch(c.h, [job, job]) as batch:
            batch.run()
            for k in range(2):
                want, want_lpd = batch.results(k)
                np.testing.assert_array_equal(post, want)
                assert lpd == want_lpd
