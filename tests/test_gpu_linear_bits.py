"""The linear FP64 form holds no value to fewer bits than a logarithm would:
what is stored, and the posteriors against sums in extended precision.

Stored values: with no samples every score is its family weight, so A_i({}) is
exp(log_w_i({}) - max_f log_w_i(f)).  Within 2^+-1024 it has 52 fraction bits.
From a weight within 3 nats the exponential rounds by at most 2^-52, the stored
value by 2^-53, and reading its logarithm back by 2^-52 and half a unit of the
result (2^-52): 1e-15.  Below 2^-1024 it has 46 bits: 2^-47, half a unit of
720 nats (2^-44) twice: 1.5e-13.

Posteriors: the roundings of the score table (a logarithm of the families that
matter, below 32 nats, to 2^-49; standard deviation 0.3 of that), of the zeta
sums, A and the level sums (ten of 2^-53 each) enter one of n levels each, so
an error of about sqrt(3 n) (0.3 2^-49 + sqrt(10) 0.3 2^-53) = 5e-15 is
expected at n = 16, and 2e-14 is four times that.  Fractions of 46 bits alone
give sqrt(3 n) 0.3 2^-46 = 3e-14."""
import math

import numpy as np
import pytest

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


def _families(n, d):
    return sum(math.comb(n - 1, k) for k in range(d + 1))


@pytest.mark.parametrize("lo,hi,tol", [(0.0, 3.0, 1e-15), (700.0, 709.0, 1.5e-13), (709.0, 720.0, 1.5e-13)])
@pytest.mark.parametrize("n,d", [(5, 2), (9, 3), (13, 2), (14, 2), (16, 3)])
def test_stored_values(ctx, n, d, lo, hi, tol):
    rng = np.random.default_rng([n, int(hi)])
    log_w = np.full((n, _families(n, d)), -3.0)
    log_w[:, 0] = -rng.uniform(lo, hi, n)
    log_w[:, 1] = 0.0                                   # the node's largest
    job = B.Job(np.zeros((0, n), np.uint8), [2] * n, d, precision="fp64", log_w=log_w)
    B.bn_edge_posteriors(ctx.h, job)
    A = B.bn_debug_stage(ctx.h, B.BN_STAGE_A, (n, 1 << (n - 1)), np.float64)
    np.testing.assert_allclose(A[:, 0], log_w[:, 0], atol=tol, rtol=0)


def _posteriors(n, d, masks, logB):
    """Edge posteriors from the library's own scores, in extended precision."""
    L = np.longdouble
    N = 1 << (n - 1)
    c = logB.max(axis=1)
    A = np.zeros((n, N), L)
    for i in range(n):
        low, mk = (1 << i) - 1, masks[i].astype(np.int64)
        A[i, (mk & low) | (mk >> 1 & ~low)] = np.exp(logB[i].astype(L) - L(c[i]))
        for j in range(n - 1):
            v = A[i].reshape(-1, 2, 1 << j)
            v[:, 1] += v[:, 0]
    full = np.zeros((n, 2 * N), L)                      # A_i(S) over all S without i
    S = np.arange(2 * N)
    without = []
    for i in range(n):
        low = (1 << i) - 1
        without.append(S[(S >> i & 1) == 0])
        full[i, without[i]] = A[i, (without[i] & low) | (without[i] >> 1 & ~low)]
    size = np.array([bin(s).count("1") for s in S])
    F, R = np.zeros(2 * N, L), np.zeros(2 * N, L)
    F[0] = R[-1] = 1
    for k in range(n):
        for i in range(n):
            T = without[i][size[without[i]] == k]
            F[T | 1 << i] += full[i, T] * F[T]
    for k in range(n - 1, -1, -1):
        for i in range(n):
            T = without[i][size[without[i]] == k]
            R[T] += full[i, T] * R[T | 1 << i]
    post = np.zeros((n, n))
    for v in range(n):
        T = without[v]
        W = F[T] * R[T | 1 << v]
        for u in range(n):
            if u != v:
                has = (T >> u & 1) == 1
                post[u, v] = float(np.sum(W[has] * (full[v, T[has]] - full[v, T[has] & ~(1 << u)])) / F[-1])
    return post


@pytest.mark.parametrize("n,d,m,arity", [(12, 3, 200, 2), (14, 3, 200, 2), (15, 2, 500, 3), (16, 4, 100, 2)])
def test_posteriors_against_extended_precision(ctx, n, d, m, arity):
    ds = datagen.random_dag_data(n, m, arity, min(d, 3), 1.0, seed=17 * n + d)
    job = B.Job(ds.data, ds.arity, d, precision="fp64")
    masks, logB = B.bn_scores(ctx.h, job)
    post, _ = B.bn_edge_posteriors(ctx.h, job)
    np.testing.assert_allclose(post, _posteriors(n, d, masks, logB), atol=2e-14, rtol=0)
