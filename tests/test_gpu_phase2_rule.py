"""The choice between the two transforms of the down-zeta's second phase, on both
sides of its line (2^7 to 2^12 rows a column, eight and four columns a block):
FP32 within its tolerance of 1e-4 of the FP64 path, which takes another kernel."""
import numpy as np
import pytest

from paper_1408_1664_gb300 import binding as B
from paper_1408_1664_gb300 import datagen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(21, 2), (22, 3), (22, 4), (23, 4), (23, 5), (24, 5), (24, 6), (25, 7),
                                 (26, 6), (26, 7)])
def test_both_sides(n, d):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ds = datagen.random_dag_data(n, 400, 2, 3, 1.0, seed=600 + n + d)
    with B.Context(0) as ctx:
        p = {f: ctx.edge_posteriors(ds.data, ds.arity, d, precision=f)[0] for f in ("fp32", "fp64")}
    assert np.all(np.isfinite(p["fp32"])) and np.all(np.isfinite(p["fp64"]))
    np.testing.assert_allclose(p["fp32"], p["fp64"], atol=1e-4, rtol=0)
