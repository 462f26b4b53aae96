"""The FFT behind the Press & Rybicki periodogram at every split of its bits into
passes: grids too small for two passes (formed bin by bin), two to four passes
with each radix from 16 to 256, and the last bin that a grid can hold (macc = 2
and a power of two of bins: K = n/4 - 1), against the FP64 oracle of the same
approximation.  Bounds as for the other shapes: an FP32 FFT of 2^26 nodes errs by
some 26 roundings of 6e-8 of its outputs' rms, far inside 1e-4 of max P.
"""
import numpy as np
import pytest

from oracle import press_rybicki as pr
from tests.parity import assert_parity

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1007_1658_gb300 import build, lsp as L
    build.build()
    c = L.Context(0)
    yield c
    c.close()


# (log2 of the grid, bins, first bin, macc)
CASES = [(5, 4, 0, 4), (8, 32, 0, 4), (8, 7, 24, 4), (9, 128, 0, 2), (9, 33, 1, 4), (10, 256, 0, 2), (11, 250, 3, 4),
         (12, 511, 1, 4), (13, 1000, 5, 4), (14, 3000, 1095, 2), (15, 4096, 0, 4), (16, 16384, 0, 2), (17, 9000, 1, 4),
         (18, 20000, 1, 4), (19, 64000, 1, 4), (20, 262144, 0, 2), (22, 500000, 1, 4), (25, 4194304, 0, 4),
         (26, 4200000, 3, 4)]


@pytest.mark.parametrize("log2,nf,j0,macc", CASES)
def test_every_split_of_the_grid(ctx, log2, nf, j0, macc):
    assert pr.fft_size(j0 + nf - 1, macc) == 1 << log2
    rng = np.random.default_rng(log2 + nf)
    n = 300 + 41 * log2
    t = np.sort(rng.uniform(0, 50.0, n))
    X = rng.normal(size=n) + np.sin(2 * np.pi * 0.9 * t)
    df = 1.0 / (1.3 * (t.max() - t.min()))
    ref = pr.periodogram(t, X, j0, nf, df, macc)
    P = ctx.press_rybicki(torch.from_numpy(t).cuda(), torch.from_numpy(X).cuda(), j0 * df, df, nf, macc=macc)
    ctx.sync(60.0)
    assert_parity(P.cpu().numpy().astype(np.float64), ref, what="2^%d nodes" % log2)
