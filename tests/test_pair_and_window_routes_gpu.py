"""Two rules of dispatch whose routes must agree bit for bit.

Pattern features: a batch with work enough takes its spectral window from the
tensor cores and re-forms the maxima in the strip kernel's order; each pattern by
itself (below a million terms) runs the strip kernel.  Equal bits, whatever the
sampling: uneven, nightly, an even cadence with dropped slots (tied maxima), and
curves of a few samples (no maxima, or all of them).

Floating-mean noise: from 304 CTAs on, four realizations share a CTA's split of
the errors; with fewer each has its own.  Same draws and order of sums, so equal
bits, with a last group of one realization and odd curve lengths.
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


def _pattern(kind, n, rng):
    if kind == "uniform":
        t = rng.uniform(0, 30.0, n)
    elif kind == "nightly":
        t = rng.integers(0, 40, n) + rng.uniform(0, 0.4, n)
    else:  # an even cadence, some slots dropped
        t = rng.permutation(n + n // 8 + 1)[:n] * 0.02
    return np.sort(t)


@pytest.mark.parametrize("kind", ["uniform", "nightly", "cadence"])
def test_window_features_of_a_batch_match_single_patterns(lsp, kind):
    rng = np.random.default_rng(len(kind))
    sizes = [4, 5, 31, 127, 128, 129, 383, 384, 385, 500] * 4
    ts = [_pattern(kind, n, rng) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    t = np.concatenate(ts)
    df = np.array([1.0 / (4.0 * (x[-1] - x[0])) for x in ts])
    f0 = df * (1 + np.arange(len(sizes)) % 3)
    nf = np.array([24 + (37 * i) % 1400 for i in range(len(sizes))], np.int64)
    assert all(n * (k + 3) < 1e6 for n, k in zip(sizes, nf)) and float(np.dot(sizes, nf)) > 2e6
    ctx = lsp.Context(0)
    together = np.asarray(ctx.fap_features(off, t, f0, df, nf))
    for c in range(len(sizes)):
        alone = np.asarray(ctx.fap_features(np.array([0, sizes[c]], np.int64), ts[c], f0[c:c + 1], df[c:c + 1],
                                            nf[c:c + 1]))
        assert np.array_equal(together[c].view(np.uint32), alone[0].view(np.uint32)), (kind, c, sizes[c], nf[c])
    ctx.close()


def test_gls_noise_by_fours_matches_one_at_a_time(lsp):
    rng = np.random.default_rng(5)
    sizes = np.array([3 + (17 * i) % 90 for i in range(80)])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    t = np.concatenate([np.sort(rng.uniform(0, 20.0, n)) for n in sizes])
    dy = np.exp(rng.uniform(np.log(0.1), np.log(10.0), t.size))
    df = np.full(80, 1.0 / 80.0)
    nf = np.array([8 + i for i in range(80)], np.int64)
    out = []
    for n_real in (17, 3):
        ctx = lsp.Context(0, batch_rhs=1, sincos_mode=lsp.SINCOS_RECUR3_X2)
        mx = np.empty(n_real * 80, np.float32)
        am = np.empty(n_real * 80, np.int32)
        ctx.batch_gls_noise(off, t, df, df, nf, dy=dy, seed=4, n_real=n_real, maxP=mx, argmax=am)
        out.append((mx.reshape(n_real, 80)[:3], am.reshape(n_real, 80)[:3]))
        ctx.close()
    assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32))
    assert np.array_equal(out[0][1], out[1][1])
