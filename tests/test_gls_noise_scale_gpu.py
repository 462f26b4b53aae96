"""The floating-mean Monte Carlo does not depend on the unit of the errors.

X = dy z is normalized by its weighted mean and variance, so a common factor of
dy falls out; by a power of two it does so without rounding, and the maxima are
equal bit for bit.  Factors near the ends of what the errors may be: 2^-63, where
a weight 1/dy^2 is near the largest FP32 value (fluxes in cgs units), and 2^60.
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


# one realization a CTA, and four (from 304 CTAs on)
@pytest.mark.parametrize("curves,n_real", [(3, 2), (80, 17)])
@pytest.mark.parametrize("power", [-63, 60])
def test_scale_of_the_errors_falls_out(lsp, curves, n_real, power):
    rng = np.random.default_rng(curves)
    sizes = np.array([3000 if curves < 10 else 300 + 7 * i for i in range(curves)])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    t = np.concatenate([np.sort(rng.uniform(0, 20.0, n)) for n in sizes])
    dy = np.exp(rng.uniform(np.log(0.6), np.log(2.0), t.size))
    df = np.full(curves, 1.0 / 80.0)
    nf = np.full(curves, 500, np.int64)
    out = []
    for p in (0, power):
        mx = np.empty(n_real * curves, np.float32)
        am = np.empty(n_real * curves, np.int32)
        with lsp.Context(0) as ctx:
            ctx.batch_gls_noise(off, t, df, df, nf, dy=dy * 2.0 ** p, seed=4, n_real=n_real, maxP=mx, argmax=am)
        out.append((mx, am))
    assert np.all(out[0][0] > 0.0)
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
    assert np.array_equal(out[0][1], out[1][1])
