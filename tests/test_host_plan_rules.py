"""Rules of the host planner that guard a kernel's limits, read through the
bn_debug_plan hook (no GPU)."""
import itertools

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


@pytest.mark.parametrize("n,m,arity,d", [(20, 10000, 3, 4), (29, 6400, 3, 3), (12, 100000, 4, 5),
                                         (20, 9400, [2 + i % 3 for i in range(20)], 5)])
def test_no_sample_count_takes_the_state_walk(n, m, arity, d):
    """The joint states of a set are counted by a histogram however many
    samples there are; only sets of more than 16384 states are walked."""
    assert _plan(n, d, m=m, arity=arity)[B.BN_PLAN_ANY_SETS] == 0


def test_sets_of_many_states_take_the_state_walk():
    """7^4 = 2401 states fit a histogram, 7^5 = 16807 do not."""
    assert _plan(8, 3, arity=7)[B.BN_PLAN_ANY_SETS] == 0
    assert _plan(8, 4, arity=7)[B.BN_PLAN_ANY_SETS] == 1


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_one_launch_sweeps_fit_the_device(precision):
    """The blocks of the whole-GPU sweeps wait on one another: F's and R's
    together never exceed what the device holds at a time, and a device too
    small for the form keeps a launch per level."""
    for n in range(5, 22):
        job = B.Job(np.zeros((2, n), np.uint8), [2] * n, 2, precision=precision)
        most, _ = B.bn_debug_sweep_blocks(job, 152)
        assert most > 0
        for sms in (1, 4, 8, 20, 76, 132, 148, 152):
            blocks, per_sm = B.bn_debug_sweep_blocks(job, sms)
            if most <= 8:                               # one block, or a cluster
                assert blocks == most
            else:
                assert 2 * blocks <= sms * per_sm and blocks != 1
                assert blocks > 8 or (blocks == 0 and sms * per_sm < 18)


def _linear(**kw):
    return _plan(kw.pop("n", 8), kw.pop("d", 2), m=kw.pop("m", 30), precision="fp64", **kw)[B.BN_PLAN_LINEAR]


def _weights(n, d):
    """log_w over the families of n nodes, and the parents of every family."""
    sets = []
    for k in range(d + 1):
        sets += sorted(itertools.combinations(range(n - 1), k), key=lambda c: sum(1 << b for b in c))
    masks = [[sum(1 << (b + (b >= i)) for b in c) for c in sets] for i in range(n)]
    return np.zeros((n, len(sets))), masks


def test_linear_form_needs_an_order_without_zero_factors():
    n = 8
    assert _linear() == 1
    q = np.zeros((n, n))
    q[3, 2] = q[0, 0] = -np.inf
    assert _linear(log_q=q) == 1
    q = np.zeros((n, n))
    q[5] = -np.inf                                      # node 5 has no place
    assert _linear(log_q=q) == 0
    q = np.zeros((n, n))
    q[1, :3] = q[4, :3] = q[1, 4:] = q[4, 4:] = -np.inf  # two nodes for one place
    assert _linear(log_q=q) == 0
    q[4, 6] = 0.0
    assert _linear(log_q=q) == 1


def test_linear_form_needs_a_network_without_zero_weights():
    n, d = 8, 2
    w, masks = _weights(n, d)
    w[2, 0] = -np.inf                                   # node 2 needs a parent: it has some
    assert _linear(log_w=w) == 1
    w[2] = -np.inf
    assert _linear(log_w=w) == 0
    w, masks = _weights(n, d)
    for i, j in ((0, 1), (1, 0)):                       # 0 needs 1 and 1 needs 0
        w[i] = [0.0 if m >> j & 1 else -np.inf for m in masks[i]]
    assert _linear(log_w=w) == 0
    w[1, 0] = 0.0
    assert _linear(log_w=w) == 1
    # no family sizes but 2: no node can be first; sizes 0 and 2: it can
    assert _linear(log_rho=[-6e6, -6e6, 0.0]) == 0
    assert _linear(log_rho=[0.0, -6e6, 0.0]) == 1
    q = np.zeros((n, n))
    q[3, 2] = -np.inf                                   # with an order prior of zeros: not shown
    w, _ = _weights(n, d)
    w[2, 0] = -np.inf
    assert _linear(log_q=q, log_w=w) == 0


def test_linear_form_counts_the_family_in_reach():
    """A node that may have only large families lies further below 1."""
    n, d, m = 6, 5, 2500
    w, masks = _weights(n, d)
    assert _linear(n=n, d=d, m=m, arity=4, log_w=w) == 1
    w[3] = [0.0 if bin(x).count("1") == d else -np.inf for x in masks[3]]
    assert _linear(n=n, d=d, m=m, arity=4, log_w=w) == 0
