"""F and R' in one launch (k_sweeps) against the level-by-level row kernels:
a job run alone and in a batch without the tuner (which keeps the level
launches) give the same bits, for every way its blocks meet -- one block (n =
5 to 10), a cluster (to n = 14) and the whole GPU (n = 15 on) -- and both
orders of A's rows (tile-level order from n = 14)."""
import numpy as np
import pytest

from paper_1408_1664_gb300 import binding as B
from paper_1408_1664_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.mark.parametrize("n,d", [(5, 2), (6, 5), (10, 3), (11, 3), (12, 2), (13, 2), (14, 4),
                                 (15, 2), (17, 3), (20, 2), (21, 2), (22, 1)])
def test_alone_equals_level_launches(torch_cuda, n, d):
    ds = datagen.random_dag_data(n, 300, 2, 3, 1.0, seed=40 + n)
    job = B.Job(ds.data, ds.arity, d, precision="fp32")
    with B.Context(0, autotune=False, graph_batch=True) as ctx:
        post, lpd = B.bn_edge_posteriors(ctx.h, job)
        again, _ = B.bn_edge_posteriors(ctx.h, job)
        with B.Batch(ctx.h, [job]) as batch:
            assert " frc=0 " in batch.describe()
            batch.run()
            want, want_lpd = batch.results(0)
    np.testing.assert_array_equal(post, want)
    np.testing.assert_array_equal(post, again)
    assert lpd == want_lpd


@pytest.mark.parametrize("n", [9, 13, 16])
def test_under_capture(torch_cuda, n):
    """A job with device data captured into a CUDA graph (its tables are on the
    device from the call before) gives the direct call's result on replay."""
    torch = torch_cuda
    ds = datagen.random_dag_data(n, 200, 2, 3, 1.0, seed=n)
    with B.Context(0) as ctx:
        data = torch.from_numpy(ds.data).cuda()
        job = B.Job(data, ds.arity, 3, precision="fp32")
        out = torch.zeros(n * n, dtype=torch.float64, device="cuda")
        s = torch.cuda.Stream()
        torch.cuda.synchronize()
        B.bn_edge_posteriors_async(ctx.h, job, out, None, s)
        s.synchronize()
        want = out.clone()
        out.zero_()
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            B.bn_edge_posteriors_async(ctx.h, job, out, None, s)
        for _ in range(2):
            g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
