"""GPU tests of the tensor-core sums (the AUTO choice on large calls) at the sizes where their tiles, units
and lists end.

Tolerances, before any run: against the FP64 oracle the library's own 1e-4 of
max P; against the packed strip kernels 2e-5 of max P (both sums carry FP32
rounding errors of about 1e-6 of max P).  Ill-conditioned floating-mean bins:
P = num / den with sums good to 2^-24, so 4 * 2^-24 / den relative, den the
smaller eigenvalue of the centred second moments (formed here in FP64).
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


@pytest.fixture(scope="module")
def ctx(lsp):
    c = lsp.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _curve(n, seed):
    rng = np.random.default_rng(seed)
    t = np.sort(rng.uniform(0.0, 40.0, n))
    X = rng.normal(size=n) + 2.0 * np.sin(2 * np.pi * 1.3 * t)
    return t, X, rng.uniform(0.3, 3.0, n)


def _both(ctx, call):
    out = []
    for mode in (0, 4):
        ctx.set_options(sincos_mode=mode)
        P = call()
        ctx.sync(60.0)
        out.append(P.cpu().numpy().astype(np.float64))
    return out


# one frequency block short of, at and past its end (64 x 256, 64 x 240 bins), one row's worth, few bins for many
# samples; units of 128 samples and running sums of 16,384 short of, at and past their ends
@pytest.mark.parametrize("n,nf", [(4097, 16384), (4096, 16385), (4096, 30721), (129, 600001), (16385, 4099),
                                  (32768, 2048), (70001, 1000), (250000, 333)])
@pytest.mark.parametrize("gls", [False, True])
def test_edges_match_oracle_and_strips(ctx, n, nf, gls):
    t, X, dy = _curve(n, n + nf)
    df = 1.0 / (4.0 * (t[-1] - t[0]))
    f0 = 1.3 - 200 * df if nf < 5000 else df
    td, Xd, dyd = _dev(t), _dev(X), _dev(dy)
    if gls:
        a, b = _both(ctx, lambda: ctx.periodogram_gls(td, Xd, f0, df, nf, dy=dyd))
    else:
        a, b = _both(ctx, lambda: ctx.periodogram(td, Xd, f0, df, nf))
    assert np.max(np.abs(a - b)) <= 2e-5 * b.max()
    rng = np.random.default_rng(1)
    ks = np.unique(np.concatenate([np.arange(min(nf, 4)), nf - 1 - np.arange(min(nf, 4)), rng.integers(0, nf, 40),
                                   np.clip(np.arange(-2, 3) + int(np.argmax(a)), 0, nf - 1)]))
    f = f0 + ks * df
    ref = oracle.gls_at(t, X, f, dy) if gls else oracle.periodogram_at(t, X, f)
    assert np.max(np.abs(a[ks] - ref)) <= TOL_ABS * ref.max()


@pytest.mark.parametrize("n_real", [1, 3])
@pytest.mark.parametrize("gls", [False, True])
def test_batch_matches_strips(ctx, n_real, gls):
    """Curves from 3 samples to several units, grids from none to several blocks, offsets of P with slack."""
    rng = np.random.default_rng(5)
    nt = np.array([3, 128, 129, 1000, 40, 5000, 257])
    nf = np.array([1, 0, 2048, 2049, 70, 40000, 511], np.int64)
    off = np.concatenate([[0], np.cumsum(nt)]).astype(np.int64)
    t = np.concatenate([np.sort(rng.uniform(0.0, 60.0, n)) for n in nt])
    dy = rng.uniform(0.3, 3.0, t.size)
    df = np.array([1.0 / (4.0 * (t[off[c + 1] - 1] - t[off[c]])) for c in range(nt.size)])
    poff = np.concatenate([[0], np.cumsum(nf + 5)]).astype(np.int64)
    args = [_dev(off), _dev(t), _dev(df), _dev(df), _dev(nf)]
    res = []
    for mode in (0, 4):
        ctx.set_options(sincos_mode=mode)
        P = torch.full((n_real * int(poff[-1]),), -7.0, device="cuda")
        maxP = torch.empty(n_real * nt.size, device="cuda")
        arg = torch.empty(n_real * nt.size, dtype=torch.int32, device="cuda")
        if gls:
            ctx.batch_gls_noise(*args, dy=_dev(dy), seed=11, n_real=n_real, P_out=P, P_off=_dev(poff), maxP=maxP, argmax=arg)
        else:
            ctx.batch(*args, seed=11, n_real=n_real, P_out=P, P_off=_dev(poff), maxP=maxP, argmax=arg)
        ctx.sync(60.0)
        res.append((P.cpu().numpy().reshape(n_real, -1), maxP.cpu().numpy().reshape(n_real, -1),
                    arg.cpu().numpy().reshape(n_real, -1)))
    for r in range(n_real):
        for c in range(nt.size):
            a, b = (x[0][r, poff[c]:poff[c + 1]] for x in res)
            assert np.all(a[nf[c]:] == -7.0)
            if nf[c] == 0:
                assert res[0][1][r, c] == 0.0 and res[0][2][r, c] == -1
                continue
            if nt[c] > 3:  # three samples leave the fit no freedom: conditioning decides
                assert np.max(np.abs(a[:nf[c]] - b[:nf[c]])) <= 2e-5 * max(1.0, b[:nf[c]].max()), (r, c)
            assert res[0][1][r, c] == a[:nf[c]].max() and a[res[0][2][r, c]] == res[0][1][r, c]


def _smaller_eigenvalue(t, f, dy):
    w = dy ** -2.0 / np.sum(dy ** -2.0)
    out = []
    for x in f:
        e = np.exp(2j * np.pi * x * (t - t[0]))
        C, W = np.sum(w * e), np.sum(w * e * e)
        out.append(0.5 * (1.0 - abs(C) ** 2 - abs(W - C * C)))
    return np.array(out)


@pytest.mark.parametrize("n,nf,span", [(20001, 4000, 40.0), (600, 150001, 0.1)])
def test_ill_conditioned_bins_are_formed_again(ctx, n, nf, span):
    """Floating-mean bins with f T below a third: a few at the low end of an oversampled grid, and a grid made of
    nothing else, with more of them than the list holds."""
    t, X, dy = _curve(n, 3)
    T = t[-1] - t[0]
    f0 = 0.1 / T
    df = span / T / nf
    ctx.set_options()
    P = ctx.periodogram_gls(_dev(t), _dev(X), f0, df, nf, dy=_dev(dy))
    ctx.sync(60.0)
    got = P.cpu().numpy().astype(np.float64)
    rng = np.random.default_rng(2)
    ks = np.unique(np.concatenate([np.arange(30), rng.integers(0, nf, 60), [nf - 1]]))
    f = f0 + ks * df
    ref = oracle.gls_at(t, X, f, dy)
    bound = np.maximum(TOL_ABS * ref.max(), 4 * 2.0 ** -24 / _smaller_eigenvalue(t, f, dy) * ref)
    assert np.all(np.abs(got[ks] - ref) <= bound)
    low = f * T < 0.3
    assert np.all(np.abs(got[ks] - ref)[low] <= 4 * 2.0 ** -24 / _smaller_eigenvalue(t, f[low], dy) * ref[low])
