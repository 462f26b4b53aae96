"""Calls of the tensor-core sums that do not fit one launch: blocks of frequencies, chunks of curves, blocks of
realizations, at sizes that a test can check.

With a launch held to a few tiles the same call runs in many; a tile's samples are
then cut elsewhere, so P agrees to the FP32 sums' rounding: 2e-5 of max P, the bound
of the comparison with the strip kernels (both about 1e-6).  Bins that are formed
again do not depend on the cut: equal bits.  A tile is 128 coarse frequencies; the
grids end short of, at and past one and several of them.
"""
import numpy as np
import pytest

import oracle
from tests.parity import TOL_ABS

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def lsp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1007_1658_gb300 import build, lsp as L
    build.build()
    return L


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("nf", [32767, 32768, 32769, 131072, 200003])
@pytest.mark.parametrize("gls", [False, True])
def test_frequency_blocks_of_one_curve(lsp, nf, gls):
    n = 2500
    rng = np.random.default_rng(nf)
    t = np.sort(rng.uniform(0.0, 40.0, n))
    X, dy = rng.normal(size=n) + 2.0 * np.sin(2 * np.pi * 1.3 * t), rng.uniform(0.3, 3.0, n)
    df = 1.0 / (40.0 * (t[-1] - t[0]))  # the first dozen bins are ill-conditioned with the floating mean
    args = (_dev(t), _dev(X), df, df, nf)
    out = []
    with lsp.Context(0) as ctx:
        for tiles in (0, 4, 7):
            ctx.test_tensor_tiles(tiles)
            padded = torch.full((nf + 512,), -7.0, device="cuda")  # what lies around P stays as it was
            P = padded[256:256 + nf]
            ctx.periodogram_gls(*args, dy=_dev(dy), out=P) if gls else ctx.periodogram(*args, out=P)
            ctx.sync(60.0)
            assert torch.all(padded[:256] == -7.0) and torch.all(padded[256 + nf:] == -7.0)
            out.append((P.cpu().numpy().astype(np.float64), ctx.last_launch_count()))
    assert nf < 70000 or out[1][1] > out[0][1]
    for P, _ in out[1:]:
        assert np.max(np.abs(P - out[0][0])) <= 2e-5 * out[0][0].max()
        if gls:
            assert np.array_equal(P[:8], out[0][0][:8])
    ks = np.unique(np.clip(np.concatenate([np.arange(3), nf - 1 - np.arange(3)] +
                                          [np.arange(-2, 3) + s for s in range(32768, nf, 32768)]), 0, nf - 1))
    f = df + ks * df
    ref = oracle.gls_at(t, X, f, dy) if gls else oracle.periodogram_at(t, X, f)
    for P, _ in out:
        assert np.max(np.abs(P[ks] - ref)) <= TOL_ABS * P.max()


@pytest.mark.parametrize("n_real", [1, 2, 19])
@pytest.mark.parametrize("gls", [False, True])
def test_chunks_of_a_batch(lsp, n_real, gls):
    rng = np.random.default_rng(6)
    nt = np.array([700, 1500, 300, 2600, 900, 400])
    nf = np.array([3000, 40000, 0, 9000, 300, 70001], np.int64)
    off = np.concatenate([[0], np.cumsum(nt)]).astype(np.int64)
    t = np.concatenate([np.sort(rng.uniform(0.0, 60.0, n)) for n in nt])
    dy = _dev(rng.uniform(0.3, 3.0, t.size))
    df = np.array([1.0 / (20.0 * 60.0)] * nt.size)
    poff = np.concatenate([[0], np.cumsum(nf + 3)]).astype(np.int64)
    args = (_dev(off), _dev(t), _dev(df), _dev(df), _dev(nf))
    res = []
    with lsp.Context(0) as ctx:
        for tiles in (0, 4, 9):
            ctx.test_tensor_tiles(tiles)
            P = torch.full((n_real * int(poff[-1]),), -7.0, device="cuda")
            m = torch.empty(n_real * nt.size, device="cuda")
            a = torch.empty(n_real * nt.size, dtype=torch.int32, device="cuda")
            kw = dict(seed=11, n_real=n_real, P_out=P, P_off=_dev(poff), maxP=m, argmax=a)
            ctx.batch_gls_noise(*args, dy=dy, **kw) if gls else ctx.batch(*args, **kw)
            ctx.sync(60.0)
            res.append((P.cpu().numpy().reshape(n_real, -1), m.cpu().numpy().reshape(n_real, -1),
                        a.cpu().numpy().reshape(n_real, -1)))
    for P, m, a in res:
        for r in range(n_real):
            for c in range(nt.size):
                p = P[r, poff[c]:poff[c + 1]]
                want = res[0][0][r, poff[c]:poff[c + 1]]
                assert np.all(p[nf[c]:] == -7.0)
                if nf[c] == 0:
                    assert m[r, c] == 0.0 and a[r, c] == -1
                    continue
                p, want = p[:nf[c]].astype(np.float64), want[:nf[c]].astype(np.float64)
                assert np.max(np.abs(p - want)) <= 2e-5 * want.max(), (r, c)
                assert m[r, c] == np.float32(p.max()) and p[a[r, c]] == p.max()
                if gls:
                    assert np.array_equal(p[:5], want[:5])


def test_chunks_of_the_window(lsp):
    rng = np.random.default_rng(4)
    curves, m = 40, 900
    t = np.concatenate([np.sort(rng.integers(0, 30, m) + rng.uniform(0, 0.4, m)) for _ in range(curves)])
    args = (_dev(np.arange(curves + 1, dtype=np.int64) * m), _dev(t), _dev(np.full(curves, 1 / 120.0)),
            _dev(np.full(curves, 1 / 120.0)), _dev(np.full(curves, 5000, np.int64)))
    out = []
    with lsp.Context(0) as ctx:
        for tiles in (0, 4, 7):
            ctx.test_tensor_tiles(tiles)
            out.append(ctx.fap_features(*args).clone())
            ctx.sync(60.0)
    assert torch.equal(out[0], out[1]) and torch.equal(out[0], out[2])
