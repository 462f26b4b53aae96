"""Which batches of short curves AUTO leaves to the strip kernels.

Kernel mode 5 is the packed strip, 6 the tensor-core sums (times beside the rule in
lsp_api.cu): a hundred curves of a unit of samples or two are faster by strips, a
few of them, longer ones, or several realizations of each on the tensor cores.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lsp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1007_1658_gb300 import build, lsp as L
    build.build()
    return L


@pytest.mark.parametrize("curves,lo,hi,n_real,mode", [(100, 50, 200, 1, 5), (148, 130, 250, 1, 5), (8, 250, 400, 1, 6),
                                                      (100, 300, 500, 1, 6), (100, 50, 200, 8, 6)])
def test_route_of_short_curves(lsp, curves, lo, hi, n_real, mode):
    rng = np.random.default_rng(9)
    nt = rng.integers(lo, hi, curves)
    off = np.concatenate([[0], np.cumsum(nt)]).astype(np.int64)
    t = np.concatenate([np.sort(rng.uniform(0, 30.0, n)) for n in nt])
    df = np.full(curves, 1.0 / 120.0)
    with lsp.Context(0) as ctx:
        mx = np.empty(curves * n_real, np.float32)
        am = np.empty(curves * n_real, np.int32)
        ctx.batch(off, t, df, df, (2 * nt).astype(np.int64), seed=3, n_real=n_real, maxP=mx, argmax=am)
        assert ctx.test_last_batch_shape()[0] == mode
        assert np.all(mx > 0.0) and np.all(am >= 0)
