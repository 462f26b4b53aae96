"""The floating-mean bins that are formed again from their samples, where there are very many of them or none should be."""
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


def test_refused_errors_cost_no_more_than_valid_ones(lsp):
    """An error that is NaN makes every sum NaN; such bins are not ill-conditioned, and forming 200,000 of them again
    took 240 times the call's time.  A factor of 10 leaves room for timing on a shared machine."""
    n, nf = 100000, 200000
    rng = np.random.default_rng(8)
    t = np.sort(rng.uniform(0.0, 1000.0, n))
    X, dy = _dev(rng.normal(size=n)), rng.uniform(0.5, 2.0, n)
    bad = dy.copy()
    bad[5] = np.nan
    t, dy, bad = _dev(t), _dev(dy), _dev(bad)
    out = torch.empty(nf, device="cuda")
    with lsp.Context(0) as ctx:
        def run(e):
            best = np.inf
            for _ in range(3):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                ctx.periodogram_gls(t, X, 1 / 4000.0, 1 / 4000.0, nf, dy=e, out=out)
                b.record()
                torch.cuda.synchronize()
                best = min(best, a.elapsed_time(b))
            return best
        run(dy)
        ctx.sync(60.0)
        valid, refused = run(dy), run(bad)
        with pytest.raises(lsp.LspError) as e:
            ctx.sync(60.0)
        assert e.value.status == lsp.ERR_INVALID_ARG
        assert refused <= 10.0 * valid, (valid, refused)
        run(dy)
        ctx.sync(60.0)
        assert torch.isfinite(out).all()


def test_aliases_of_an_even_cadence_have_no_power(lsp):
    """At multiples of the sampling rate every phase is the same, and a sinusoid with an offset fits nothing: P is 0.
    1 - |C|^2, 0 but for the sums' rounding, comes out negative for about half of the weights."""
    curves, n, nf, rate, df = 120, 600, 300, 2.0, 1.0 / 64.0
    rng = np.random.default_rng(77)
    off = np.arange(curves + 1, dtype=np.int64) * n
    t = np.tile(np.arange(n) / rate, curves)
    dy, X = rng.uniform(0.3, 3.0, t.size), rng.normal(size=t.size)
    grid = _dev(np.full(curves, df))
    P_off = np.arange(curves + 1, dtype=np.int64) * nf
    P = torch.full((curves * nf,), -7.0, device="cuda")
    with lsp.Context(0) as ctx:
        ctx.batch_gls(_dev(off), _dev(t), _dev(X), grid, grid, _dev(np.full(curves, nf, np.int64)),
                      dy=_dev(dy), P_out=P, P_off=_dev(P_off), maxP=torch.empty(curves, device="cuda"),
                      argmax=torch.empty(curves, dtype=torch.int32, device="cuda"))
        ctx.sync(60.0)
    P = P.cpu().numpy().reshape(curves, nf)
    alias = np.arange(int(rate / df) - 1, nf, int(rate / df))
    assert alias.size == 2 and np.all(P[:, alias] == 0.0), P[:, alias].max(axis=0)
    for c in range(curves):  # the other bins, their peak by the oracle
        k = int(np.argmax(P[c]))
        ref = oracle.gls_at(t[:n], X[c * n:(c + 1) * n], np.array([df + k * df]), dy[c * n:(c + 1) * n])[0]
        assert abs(P[c, k] - ref) <= TOL_ABS * ref, c


def _copies(t, X, dy, df, nf, copies):
    n = t.size
    off = np.arange(copies + 1, dtype=np.int64) * n
    grid = np.full(copies, df)
    rep = lambda a: _dev(np.tile(a, copies))
    P_off = np.arange(copies + 1, dtype=np.int64) * nf
    return (_dev(off), rep(t), rep(X), _dev(grid), _dev(grid), _dev(np.full(copies, nf, np.int64))), rep(dy), _dev(P_off)


@pytest.mark.parametrize("n,nf,copies", [(600, 3000, 20), (600, 3000, 40), (300, 70001, 2)])
def test_a_bin_does_not_depend_on_how_many_others_there_are(lsp, n, nf, copies):
    """Copies of one curve on a grid whose every bin is ill-conditioned (f T < 0.3, down to 1e-4, where 1 - |C|^2 is
    lost in the sums' rounding), fewer and more of them in all than the list of such bins holds: the copies have the
    same P bit for bit, the same in every call, and with fewer the same as the curve by itself."""
    rng = np.random.default_rng(n)
    t = np.sort(rng.uniform(0.0, 40.0, n))
    X, dy = rng.normal(size=n), rng.uniform(0.3, 3.0, n)
    df = 0.3 / (t[-1] - t[0]) / nf
    out = []
    for c in (1, copies):
        args, e, P_off = _copies(t, X, dy, df, nf, c)
        with lsp.Context(0) as ctx:
            for _ in range(2):  # a second call finds the bit map as the first one did
                P = torch.full((c * nf,), -7.0, device="cuda")
                m, a = ctx.batch_gls(*args, dy=e, P_out=P, P_off=P_off, maxP=torch.empty(c, device="cuda"),
                                     argmax=torch.empty(c, dtype=torch.int32, device="cuda"))
                ctx.sync(60.0)
                out.append((P.cpu().numpy().reshape(c, nf), m.cpu().numpy(), a.cpu().numpy()))
    want, best, at = out[0]
    assert np.all(want >= 0.0) and best[0] == want.max() and want[0, at[0]] == best[0]
    if copies * nf > 1 << 16:
        want, best, at = out[2][0][:1], out[2][1][:1], out[2][2][:1]
        assert np.max(np.abs(want - out[0][0])[0, nf // 10:]) <= 1e-5 * want.max()  # both good to 2^-24 / 3e-3 there
    for P, m, a in out[1 if copies * nf <= 1 << 16 else 2:]:
        assert np.array_equal(P.view(np.uint32), np.broadcast_to(want, P.shape).view(np.uint32))
        assert np.all(m == best[0]) and np.all(a == at[0])
