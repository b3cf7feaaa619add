"""Modular features with large finite weights, FP32 from n = 14 (the persistent
up-zeta tiles): a constant weight moves a node's values far above one window
of the tiles, and weights on part of its families spread them over several
windows, so every form of a tile runs on values the scores alone never reach.
Against the oracle.

The bound: a value of up to 2^9 bits is stored to 2^-16 bits, and the column
sums, A and F store one per level (n <= 17): 3 * 17 * 2^-16 * ln 2 = 5.4e-4
nats; 1e-3 with the sums' own rounding."""
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


@pytest.mark.parametrize("n,d", [(14, 2), (15, 4), (17, 3)])
@pytest.mark.parametrize("const,some", [(150.0, 0.0), (250.0, 0.0), (0.0, 60.0), (0.0, 200.0), (200.0, 150.0)])
def test_large_feature_weights_match_oracle(ctx, n, d, const, some):
    ds = datagen.random_dag_data(n, 200, 2, min(d, 3), 1.0, seed=41 * n + d)
    masks, _ = orc.scores(ds.data, ds.arity, d)
    log_f = np.zeros(masks.shape)
    log_f[3] += const                                  # every family of node 3
    log_f[n - 2] += const
    log_f[5, masks[5] & 1 == 1] += some                # the families of node 5 with parent 0
    ref, lref = orc.feature_posterior(ds.data, ds.arity, d, log_f)
    p, lpfd = B.bn_feature_posterior(ctx.h, B.Job(ds.data, ds.arity, d, precision="fp32"), log_f)
    assert abs(lpfd - lref) <= 1e-3
    assert abs(math.log(p) - math.log(ref)) <= 2e-3
