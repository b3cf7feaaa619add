"""Rules of the host planner that guard a kernel's limits, read through the
bn_debug_plan hook (no GPU)."""
import numpy as np
import pytest

from paper_1408_1664_gb300 import binding as B


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.load(build_if_missing=True)


def _plan(n, d, m=2, arity=2, precision="fp32", **kw):
    ar = [arity] * n if np.isscalar(arity) else arity
    return B.bn_debug_plan(B.Job(np.zeros((m, n), np.uint8), ar, d, precision=precision, **kw))


@pytest.mark.parametrize("precision,first,last", [("fp32", 5, 32), ("fp64", 5, 31)])
def test_one_launch_sweeps_end_with_their_places(precision, first, last):
    """k_sweeps forms the places of A's n 2^(n-1) values in 32 bits: no group
    of larger jobs may take it, by the flag or by the tuner."""
    for n in range(first, last + 1):
        assert _plan(n, 1, precision=precision)[B.BN_PLAN_SWEEPS] == (n << (n - 1) <= 2 ** 32), n
