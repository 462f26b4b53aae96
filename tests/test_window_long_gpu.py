"""Window features of long patterns: the route of a batch (tensor cores, the maxima formed again in the strip
kernel's order) against the strip kernel, bit for bit.

The strip kernel adds all samples in one FP32 chain.  On a cadence whose first
sample is off the others' phase every sample adds nearly the same term at an alias,
and the chain's roundings have one sign: its W is off by up to 1e-3 there, by
another amount at every alias.  The maxima of these patterns are closer than that
(a twentieth of the samples is shifted, which lowers W at the higher aliases by a
few 1e-4), so which eight of fourteen are highest depends on those roundings.  A
pattern by itself stays below a million terms and runs the strip kernel.
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


@pytest.mark.parametrize("n,nw,shift", [(32700, 30, 0.0047), (32700, 30, 0.003), (20000, 48, 0.004), (5000, 190, 0.004),
                                        (65536, 15, 0.0047)])
def test_maxima_of_long_patterns_match_the_strip_kernel(lsp, n, nw, shift):
    assert n * nw < 1e6
    ts = []
    for phase in np.linspace(0.02, 0.49, 24):
        k = np.arange(n - 1)
        ts.append(np.concatenate([[0.0], phase + k + np.where(k < n // 32, shift, 0.0)]))
    off = np.arange(len(ts) + 1, dtype=np.int64) * n
    df = np.full(len(ts), 0.5)
    nf = np.full(len(ts), nw, np.int64)
    with lsp.Context(0) as ctx:
        together = np.asarray(ctx.fap_features(off, np.concatenate(ts), df, df, nf))
        for c, t in enumerate(ts):
            alone = np.asarray(ctx.fap_features(off[:2], t, df[:1], df[:1], nf[:1]))
            assert np.array_equal(together[c].view(np.uint32), alone[0].view(np.uint32)), c
