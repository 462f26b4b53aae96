"""A wait of the tensor-core kernel that runs out: the call ends, its outputs are NaN, lsp_sync says so, and the
context computes the same bits as before afterwards.

The waits are made to give up at their first look, when nothing has been written
yet; no kernel waits for anything that does not come.
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


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _calls():
    rng = np.random.default_rng(12)
    n, nf, curves = 8000, 16000, 12
    t = np.sort(rng.uniform(0.0, 50.0, n))
    X, dy = rng.normal(size=n), rng.uniform(0.5, 2.0, n)
    off = np.arange(curves + 1, dtype=np.int64) * 600
    ts = np.concatenate([np.sort(rng.uniform(0.0, 50.0, 600)) for _ in range(curves)])
    df = 1.0 / 200.0
    one = (_dev(t), _dev(X), df, df, nf)
    many = (_dev(off), _dev(ts), _dev(np.full(curves, df)), _dev(np.full(curves, df)),
            _dev(np.full(curves, 1500, np.int64)))
    e, es = _dev(dy), _dev(rng.uniform(0.5, 2.0, ts.size))
    return {"periodogram": lambda c: c.periodogram(*one), "gls": lambda c: c.periodogram_gls(*one, dy=e),
            "batch": lambda c: c.batch(*many, seed=3, n_real=2)[0],
            "batch_gls_noise": lambda c: c.batch_gls_noise(*many, dy=es, seed=3, n_real=2)[0],
            "features": lambda c: c.fap_features(*many)}


@pytest.mark.parametrize("which", ["periodogram", "gls", "batch", "batch_gls_noise", "features"])
def test_a_wait_that_runs_out_is_reported(lsp, which):
    call = _calls()[which]
    with lsp.Context(0) as ctx:
        want = call(ctx).clone()
        ctx.sync(60.0)
        assert torch.isfinite(want).all()
        ctx.test_give_up_waits(True)
        got = call(ctx)
        with pytest.raises(lsp.LspError) as e:
            ctx.sync(60.0)
        assert e.value.status == lsp.ERR_CUDA and "wait" in str(e.value)
        assert torch.isnan(got).all()
        ctx.test_give_up_waits(False)
        again = call(ctx)
        ctx.sync(60.0)
        assert torch.equal(again, want)
