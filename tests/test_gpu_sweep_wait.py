"""The blocks of the whole-GPU sweeps (k_sweeps, n of about 15 to 21) wait on one
another by polls of a counter.  The wait is bounded: with one block missing (a
test hook) the others give up after the given number of polls, leave the timeout
bit in the job's error word and return -- no fault, no endless wait -- and the
context runs the next job of that form correctly."""
import ctypes as C

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
    B.load(build_if_missing=True)
    with B.Context(0, autotune=False) as c:
        yield c


@pytest.mark.parametrize("polls", [1, 1000, 100000])
def test_missing_block_times_out_and_context_survives(ctx, polls):
    w = C.c_int32(-1)
    assert B.load().bn_debug_sweep_wait(polls, C.byref(w)) == 0
    assert w.value == 2                   # the timeout bit, nothing else
    ds = datagen.random_dag_data(n=17, m=200, arity=2, max_parents=3, alpha=1.0, seed=polls % 89)
    ref = orc.edge_posteriors(ds.data, ds.arity, 2)
    for precision, tol in (("fp32", 1e-4), ("fp64", 1e-9)):
        post, _ = ctx.edge_posteriors(ds.data, ds.arity, 2, precision=precision)
        np.testing.assert_allclose(post, ref["post"], atol=tol, rtol=0)
