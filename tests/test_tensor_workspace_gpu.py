"""Calls that the tensor cores would run and whose workspace there cannot be allocated: the strip kernels run them.

lsp_test_fail_allocation makes the n-th workspace allocation of a fresh context
fail as cudaMalloc would; n covers the tensor-core path's own buffers, in the order
the call asks for them.  The results are the strips' bit for bit, and the next call
runs on the tensor cores again.
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


@pytest.fixture(scope="module")
def calls(lsp):
    rng = np.random.default_rng(21)
    n, curves, m = 8000, 12, 600
    df = 1.0 / 200.0
    one = (_dev(np.sort(rng.uniform(0.0, 50.0, n))), _dev(rng.normal(size=n)), df, df, 16000)
    e = _dev(rng.uniform(0.5, 2.0, n))
    many = (_dev(np.arange(curves + 1, dtype=np.int64) * m),
            _dev(np.concatenate([np.sort(rng.uniform(0.0, 50.0, m)) for _ in range(curves)])),
            _dev(np.full(curves, df)), _dev(np.full(curves, df)), _dev(np.full(curves, 1500, np.int64)))
    es = _dev(rng.uniform(0.5, 2.0, curves * m))
    out = {"periodogram": lambda c: c.periodogram(*one), "gls": lambda c: c.periodogram_gls(*one, dy=e),
           "batch": lambda c: c.batch(*many, seed=3, n_real=2)[0],
           "batch_gls_noise": lambda c: c.batch_gls_noise(*many, dy=es, seed=3, n_real=2)[0]}
    ref = {}
    for k, f in out.items():
        for mode in (lsp.SINCOS_AUTO, lsp.SINCOS_RECUR3_X2):
            with lsp.Context(0, sincos_mode=mode) as c:
                ref[k, mode] = f(c).clone()
                c.sync(60.0)
        assert not torch.equal(ref[k, lsp.SINCOS_AUTO], ref[k, lsp.SINCOS_RECUR3_X2]), k
    return out, ref, many


@pytest.mark.parametrize("which,first,last", [("periodogram", 1, 2), ("gls", 1, 5), ("batch", 8, 10),
                                              ("batch_gls_noise", 8, 13)])
def test_without_the_workspace_the_strips_run(lsp, calls, which, first, last):
    call, ref, _ = calls[0][which], calls[1], calls[2]
    for nth in range(first, last + 1):
        with lsp.Context(0) as ctx:
            ctx.test_fail_allocation(nth)
            got = call(ctx)
            ctx.sync(60.0)
            assert torch.equal(got, ref[which, lsp.SINCOS_RECUR3_X2]), nth
            got = call(ctx)
            ctx.sync(60.0)
            assert torch.equal(got, ref[which, lsp.SINCOS_AUTO]), nth
        # the allocation after them is one that every route needs
    with lsp.Context(0) as ctx:
        if which in ("periodogram", "gls"):
            ctx.test_fail_allocation(last + 1)
            with pytest.raises(lsp.LspError) as e:
                call(ctx)
            assert e.value.status == lsp.ERR_OOM


@pytest.mark.parametrize("nth", [8, 9, 10, 11, 12])
def test_features_without_the_workspace(lsp, calls, nth):
    many = calls[2]
    with lsp.Context(0) as ctx:
        want = ctx.fap_features(*many).clone()
        ctx.sync(60.0)
    with lsp.Context(0) as ctx:
        ctx.test_fail_allocation(nth)
        got = ctx.fap_features(*many)
        ctx.sync(60.0)
        assert torch.equal(got, want)


@pytest.mark.parametrize("other", ["features", "batch_gls"])
def test_a_cached_batch_is_planned_again_after_a_failure(lsp, calls, other):
    """The tile list and the partial tiles are shared with other calls: one that fails half way through growing them
    leaves no batch graph behind that still points there."""
    batch, ref, many = calls[0]["batch"], calls[1], calls[2]
    rng = np.random.default_rng(2)
    curves, m = 300, 700
    big = (_dev(np.arange(curves + 1, dtype=np.int64) * m),
           _dev(np.concatenate([np.sort(rng.uniform(0.0, 50.0, m)) for _ in range(curves)])),
           _dev(np.full(curves, 1 / 200.0)), _dev(np.full(curves, 1 / 200.0)), _dev(np.full(curves, 6000, np.int64)))
    with lsp.Context(0) as ctx:
        assert torch.equal(batch(ctx), ref["batch", lsp.SINCOS_AUTO])
        n = 0
        while True:  # every allocation of the larger call in turn
            n += 1
            ctx.test_fail_allocation(n)
            try:
                ctx.fap_features(*big) if other == "features" else ctx.batch_gls(big[0], big[1], big[1], *big[2:])
                failed = False
            except lsp.LspError as e:
                assert e.status == lsp.ERR_OOM
                failed = True
            ctx.sync(60.0)
            assert torch.equal(batch(ctx), ref["batch", lsp.SINCOS_AUTO]), n
            ctx.sync(60.0)
            if not failed and n > 20:
                break
        ctx.test_fail_allocation(0)
