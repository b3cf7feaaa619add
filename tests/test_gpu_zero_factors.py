"""FP64 jobs whose zero factors leave no order or no network, or only networks
without the empty parent sets: the linear form is kept where its lower bound
holds, and the logarithms elsewhere, with e^-1e7 in the zeros' place.

Bounds: 1e-9 (the FP64 contract); where P(D) = 0 the logarithms lie near -1e7,
whose unit is 1.9e-9: 2 n roundings of it enter a posterior, 1e-7 at n = 16."""
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


@pytest.mark.parametrize("n", [6, 12, 14, 16])
def test_order_prior_without_an_order(ctx, n):
    ds = datagen.random_dag_data(n, 120, 2, 2, 1.0, seed=800 + n)
    log_q = -np.random.default_rng(n).random((n, n))
    log_q[4] = -np.inf                                  # node 4 has no place
    soft = np.where(np.isinf(log_q), -1e7, log_q)
    ref = orc.edge_posteriors(ds.data, ds.arity, 2, log_q=soft)
    job = B.Job(ds.data, ds.arity, 2, precision="fp64", log_q=log_q)
    post, lpd = B.bn_edge_posteriors(ctx.h, job)
    np.testing.assert_allclose(post, ref["post"], atol=1e-7, rtol=0)
    assert lpd < -5e6 and abs(lpd - ref["log_PD"]) <= 1e-6
    masks, _ = orc.scores(ds.data, ds.arity, 2)
    log_f = np.zeros(masks.shape)
    log_f[1] = np.where(masks[1] & 1, 0.0, -np.inf)     # the edge 0 -> 1
    p, lpfd = B.bn_feature_posterior(ctx.h, job, log_f)
    assert abs(p - ref["post"][0, 1]) <= 1e-6
    assert math.isfinite(lpfd)
    post32, lpd32 = B.bn_edge_posteriors(ctx.h, B.Job(ds.data, ds.arity, 2, precision="fp32", log_q=log_q))
    assert np.all(np.isfinite(post32)) and lpd32 < -5e6


@pytest.mark.parametrize("n,d,m", [(7, 3, 400), (13, 2, 3000), (14, 2, 7800), (14, 2, 9000), (15, 3, 700)])
def test_features_that_forbid_the_empty_set(ctx, n, d, m):
    """Strongly dependent data on both sides of the range rule: every node but
    the first must have a parent, and three of them the largest number."""
    ds = datagen.random_dag_data(n, m, 2, 2, 1.0, seed=810 + n)
    data = ds.data.copy()
    data[:, n - 1] = data[:, 0]
    data[:, n - 2] = data[:, 3]
    masks, _ = orc.scores(data, ds.arity, d)
    size = np.array([[bin(int(g)).count("1") for g in row] for row in masks])
    log_f = np.zeros(masks.shape)
    log_f[1:][size[1:] == 0] = -np.inf
    log_f[4:7][size[4:7] < d] = -np.inf
    ref, lref = orc.feature_posterior(data, ds.arity, d, log_f)
    p, lpfd = B.bn_feature_posterior(ctx.h, B.Job(data, ds.arity, d, precision="fp64"), log_f)
    assert abs(p - ref) <= 1e-9
    assert abs(lpfd - lref) <= 1e-9 * max(1.0, abs(lref))


@pytest.mark.parametrize("n", [7, 14])
def test_log_rho_that_leaves_no_network(ctx, n):
    """No family of fewer than two parents: no node can come first."""
    ds = datagen.random_dag_data(n, 100, 2, 2, 1.0, seed=820 + n)
    rho = [-6e6, -6e6, 0.0]
    ref = orc.edge_posteriors(ds.data, ds.arity, 2, log_rho=rho)
    post, lpd = B.bn_edge_posteriors(ctx.h, B.Job(ds.data, ds.arity, 2, precision="fp64", log_rho=rho))
    np.testing.assert_allclose(post, ref["post"], atol=1e-7, rtol=0)
    assert abs(lpd - ref["log_PD"]) <= 1e-6
