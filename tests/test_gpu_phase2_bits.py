"""Phase 2 of the FP32 down-zeta keeps its inputs' bits: on given sums over the
low bits (log2, within 15 bits of 0) its outputs agree with sums in double.

The bound, in bits: an output below 32 rounds by 2^-20 (9.5e-7), its logarithm
by 2^-22 (2.4e-7), the terms' exponentials by 2^-22 of themselves (3.4e-7), and
a sum of at most 17 steps by 17 2^-24 of itself (1.5e-6): 3e-6.  In the scale of
a pass (2^126) a logarithm alone would round by 2^-18 (3.8e-6), and an input by
as much.
"""
import itertools
import math

import numpy as np
import pytest

from paper_1408_1664_gb300 import binding as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.load(build_if_missing=True)


def _families(bits, d):
    """Masks of at most d of the bits, by size, then colexicographically."""
    out = []
    for k in range(d + 1):
        out += sorted(sum(1 << b for b in c) for c in itertools.combinations(range(bits), k))
    return out


# register transform of short columns (h = n - 14 <= 9), of long ones (d = 7),
# lane sums (h < 8), wide sums (h >= 8)
@pytest.mark.parametrize("n,d", [(14, 3), (16, 3), (18, 4), (18, 7), (21, 2), (22, 2), (23, 1), (24, 0), (24, 2)])
def test_outputs_against_double(n, d):
    h = n - 14
    low = _families(13, d)
    rng = np.random.default_rng([n, d])
    W = rng.uniform(-15.0, 15.0, (n, 1 << h, len(low))).astype(np.float32)
    W -= np.float32(h)                                  # the sums stay below 2^16
    got = B.bn_debug_phase2(B.Job(np.zeros((0, n), np.uint8), [2] * n, d, precision="fp32"), W)
    index = {m: f for f, m in enumerate(_families(n - 1, d))}
    for v in (0, n // 2, n - 1):
        x = np.exp2(W[v].astype(np.float64))            # rows x columns
        for j in range(h):
            y = x.reshape(-1, 2, 1 << j, len(low))
            y[:, 0] += y[:, 1]
        want = np.full(got.shape[1], np.nan)
        for c, g in enumerate(low):
            for t in range(1 << h):
                if bin(g).count("1") + bin(t).count("1") <= d:
                    want[index[g | t << 13]] = math.log2(x[t, c])
        np.testing.assert_allclose(got[v].astype(np.float64), want, atol=3e-6, rtol=0)
