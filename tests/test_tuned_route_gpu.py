"""What a tuned size does to the route of later AUTO calls, the tensor cores' against the strips'.

The two routes round differently, so equal bits tell which one ran: P with the
defaults of an untuned context against P of the packed strips asked for.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

N, NF = 20000, 40000  # strips 0.2 ms, tensor cores 0.08


@pytest.fixture(scope="module")
def lsp():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1007_1658_gb300 import build, lsp as L
    build.build()
    return L


@pytest.fixture(scope="module")
def data():
    rng = np.random.default_rng(31)
    t = np.sort(rng.uniform(0.0, 100.0, N))
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    return d(t), d(rng.normal(size=N) + np.sin(2 * np.pi * 1.7 * t)), d(rng.uniform(0.5, 2.0, N)), 1.0 / 400.0


def _run(ctx, data, gls):
    t, X, dy, df = data
    P = ctx.periodogram_gls(t, X, df, df, NF, dy=dy) if gls else ctx.periodogram(t, X, df, df, NF)
    ctx.sync(60.0)
    return P.cpu().numpy()


def _default(lsp, data, gls, **opts):
    with lsp.Context(0, **opts) as ctx:
        return _run(ctx, data, gls)


def _strip_file(lsp, path, **more):
    """A tuning file with one strip entry for the size (its bucket: floor of log2)."""
    with lsp.Context(0) as ctx:
        ctx.tune_save(path)
    head = path.read_text().splitlines()[0]
    extra = "".join(', "%s": %d' % kv for kv in more.items())
    path.write_text('%s\n{"kind": 1, "nt": 14, "nf": 15, "sincos": 4, "F": 24, "split": 10, "ms": 0.2%s}\n]}\n'
                    % (head, extra))


def test_floating_mean_calls_do_not_follow_a_classic_entry(lsp, data, tmp_path):
    want = _default(lsp, data, True)
    assert not np.array_equal(want, _default(lsp, data, True, sincos_mode=lsp.SINCOS_RECUR3_X2))
    path = tmp_path / "tune.json"
    _strip_file(lsp, path, beat_tensor=1)
    with lsp.Context(0) as ctx:
        assert ctx.tune_load(path) == 1
        assert np.array_equal(_run(ctx, data, True), want)


def test_an_entry_not_timed_against_the_tensor_cores_leaves_them(lsp, data, tmp_path):
    """A file of a version that timed strips only, and one whose strip won."""
    tensor, strips = _default(lsp, data, False), _default(lsp, data, False, sincos_mode=lsp.SINCOS_RECUR3_X2, split=10)
    assert not np.array_equal(tensor, strips)
    path = tmp_path / "tune.json"
    for more, want in (({}, tensor), ({"beat_tensor": 1}, strips)):
        _strip_file(lsp, path, **more)
        with lsp.Context(0) as ctx:
            assert ctx.tune_load(path) == 1
            assert np.array_equal(_run(ctx, data, False), want)


def test_tuning_a_large_size_keeps_the_tensor_cores(lsp, data, tmp_path):
    want = _default(lsp, data, False)
    path = tmp_path / "tune.json"
    _strip_file(lsp, path)
    with lsp.Context(0) as ctx:
        ctx.tune_load(path)
        chosen = ctx.autotune(N, NF)
        assert np.array_equal(_run(ctx, data, False), want)
        ctx.tune_save(path)
        # the fastest strip, for whoever asks for it
        entry = [x for x in path.read_text().splitlines() if '"kind": 1' in x]
        assert len(entry) == 1 and '"beat_tensor": 0' in entry[0] and chosen["split"] >= 1
        ctx.set_options(**chosen)
        assert not np.array_equal(_run(ctx, data, False), want)
