"""Performance cases of the periodogram engine: the calls its users make, over the sizes they make them at.

Kinds, each through the ``lsp.Context`` entry point of that name on device arrays:

* ``single``   -- ``periodogram``: one light curve on its own grid (Eq. 9-11 of the paper).
* ``gls``      -- ``periodogram_gls``: the floating-mean periodogram of one curve with errors.
* ``pr``       -- ``press_rybicki``: the fast approximation of one curve.
* ``batch``    -- ``batch`` with measured curves: a survey's light curves, whole periodograms and peaks.
* ``mc``       -- ``batch`` with noise: Monte-Carlo maxima of sampling patterns (false-alarm statistics).
* ``batch_gls``-- ``batch_gls``: a survey's curves with errors, peaks only.
* ``mc_gls``   -- ``batch_gls_noise``: the floating-mean Monte Carlo.
* ``predict``  -- ``fap_predict``: features of sampling patterns and the network's quantiles.
* ``grad``     -- ``fap_gradients``: forward and backward pass of the surrogate's network on a minibatch.

``exact`` evaluates every kind in 64 bits with plain torch, from the definitions in include/lsp.h.
"""
import math

import numpy as np
import torch

from paper_1007_1658_gb300 import lsp

HIDDEN = 256
LEVELS = (0.05, 0.10, 0.25, 0.50, 0.75, 0.90, 0.95, 0.98, 0.99)


def listed():
    return [
        # the smallest call: a short ground-based series, where launches and latency count
        {"name": "single_1k", "kind": "single", "n": 1000, "nf": 2000, "span": 100.0, "sampling": "uniform"},
        # a space mission's regular cadence with dropped slots, a ragged grid up to f t of 3e4 turns
        {"name": "single_65k", "kind": "single", "n": 65536, "nf": 318500, "span": 1300.0, "over": 10.0,
         "sampling": "cadence"},
        # the headline workload: 1000 nights of 100 samples, oversampling 4
        {"name": "single_100k", "kind": "single", "n": 100000, "nf": 200000, "span": 1000.0, "sampling": "nightly"},
        # the paper's own shape (Sec. 5.2): 382,003 samples, 1,528,064 frequencies; the largest call
        {"name": "single_382k", "kind": "single", "n": 382003, "nf": 1528064, "span": 150.0, "sampling": "cadence"},
        # the headline series with per-sample errors, the offset fitted with the sinusoid
        {"name": "gls_100k", "kind": "gls", "n": 100000, "nf": 200000, "span": 1000.0, "sampling": "nightly"},
        # the paper's shape through the approximation: a quick look before the exact evaluation
        {"name": "pr_382k", "kind": "pr", "n": 382003, "nf": 1528064, "span": 150.0, "sampling": "cadence"},
        # one noise realization of each of 4096 patterns: training targets of the surrogate
        {"name": "mc_4096", "kind": "mc", "curves": 4096, "reals": 1, "nt_min": 200, "nt_max": 20000},
        # many realizations of each pattern: the noise-peak distribution of a pattern (Sec. 6.2)
        {"name": "mc_256x64", "kind": "mc", "curves": 256, "reals": 64, "nt_min": 200, "nt_max": 20000},
        # a survey field: measured curves with errors in one call, their peaks
        {"name": "batch_gls_1024", "kind": "batch_gls", "curves": 1024, "reals": 1, "nt_min": 200, "nt_max": 20000},
        # noise-peak distributions that depend on the errors as well
        {"name": "mc_gls_256x16", "kind": "mc_gls", "curves": 256, "reals": 16, "nt_min": 200, "nt_max": 20000},
        # false-alarm levels of a field's patterns without any Monte Carlo
        {"name": "predict_256", "kind": "predict", "curves": 256, "reals": 1, "nt_min": 200, "nt_max": 20000},
        # a training minibatch of the surrogate, gradients back
        {"name": "grad_4096", "kind": "grad", "rows": 4096},
    ]


def draw(rng):
    """One more case of the same ranges, sizes log-uniform, odd ones as likely as even ones."""
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["single", "single", "gls", "pr", "batch", "mc", "mc", "batch_gls", "mc_gls", "predict", "grad"])
    if kind == "grad":
        return {"kind": kind, "rows": log_int(256, 8192)}
    if kind in ("single", "gls", "pr"):
        n = log_int(300, 200000)
        return {"kind": kind, "n": n, "nf": max(64, min(int(n * rng.uniform(0.7, 5.0)), 600000)),
                "span": round(math.exp(rng.uniform(math.log(30.0), math.log(1500.0))), 3),
                "over": rng.choice([4.0, 5.0, 10.0]), "sampling": rng.choice(["uniform", "nightly", "cadence"])}
    nt_min = log_int(100, 600)
    nt_max = log_int(1500, 20000)
    if kind == "mc":
        reals = rng.choice([1, 1, log_int(2, 100)])
    else:
        reals = log_int(2, 40) if kind == "mc_gls" else 1
    most = 2000 if kind in ("mc", "batch_gls") else 300
    return {"kind": kind, "curves": max(3, min(log_int(8, most), int(6000 / reals))), "reals": reals, "nt_min": nt_min,
            "nt_max": nt_max}


# ---------------------------------------------------------------- inputs


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(g, n, a=0.0, b=1.0):
    return a + (b - a) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _curve(case, seed):
    """Times, values (three sinusoids in noise on an offset) and errors of one curve, and its grid."""
    g = _gen(seed)
    n, nf, span = case["n"], case["nf"], case["span"]
    if case["sampling"] == "uniform":
        t = _uniform(g, n, 0.0, span)
    elif case["sampling"] == "nightly":  # half of every day, 100 samples a night where there are as many
        nights = max(1, min(int(span), n // 100))
        day = torch.arange(n, device="cuda", dtype=torch.float64).remainder(nights) * (span / nights)
        t = day + 0.5 * _uniform(g, n) * min(1.0, span / nights)
    else:  # regular slots, a tenth of them dropped, half a second of jitter
        slots = n + n // 10 + 2
        keep = torch.randperm(slots, generator=g, device="cuda")[:n].double()
        t = keep * (span / slots) + _uniform(g, n, -0.5, 0.5) / 86400.0
    t = torch.sort(t).values.contiguous()
    df = 1.0 / (case.get("over", 4.0) * float(t[-1] - t[0]))
    dy = 0.5 * torch.exp(_uniform(g, n, math.log(0.3), math.log(3.0)))
    rs = np.random.default_rng(seed)
    X = torch.full_like(t, 1.5) + torch.randn(n, generator=g, device="cuda", dtype=torch.float64) * (
        dy if case["kind"] == "gls" else 0.5)
    for a in (1.0, 0.3, 0.05):
        f = rs.uniform(0.02, 0.9) * nf * df
        X += a * torch.sin(2 * math.pi * ((f * t) % 1.0) + rs.uniform(0, 2 * math.pi))
    return {"t": t, "X": X, "dy": dy, "f0": df, "df": df, "nf": nf}


def _sizes(case):
    """Samples of every pattern: the log-uniform law's quantiles, so that the work is the same for every seed."""
    q = (np.arange(case["curves"]) + 0.5) / case["curves"]
    return np.maximum(4, np.floor(case["nt_min"] * (case["nt_max"] / case["nt_min"]) ** q)).astype(np.int64)


def _patterns(case, seed):
    """Sampling patterns with nightly windows and one seasonal gap each, in CSR form, with their grids (oversampling 4
    up to the mean Nyquist frequency)."""
    g = _gen(seed)
    rs = np.random.default_rng(seed)
    nt = rs.permutation(_sizes(case))
    n = nt.size
    T = np.exp(rs.uniform(np.log(30.0), np.log(1000.0), n))
    frac, gap = rs.uniform(0.3, 0.7, n), rs.uniform(0.05, 0.4, n)
    at = rs.uniform(0.0, 1.0, n)
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum(nt)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    c = torch.repeat_interleave(torch.arange(n, device="cuda"), d(nt))
    days = torch.floor(_uniform(g, int(off[-1])) * (d(T) * (1 - d(gap)))[c])
    days = days + torch.where(days > d(at * (1 - gap) * T)[c], torch.floor(d(gap * T))[c], 0.0)
    t = days + _uniform(g, int(off[-1])) * d(frac)[c]
    key = torch.sort(c.double() * 2048.0 + t).values  # by curve, then by time
    t = (key - c.double() * 2048.0).contiguous()
    first, last = t[d(off[:-1])], t[d(off[1:] - 1)]
    df = (1.0 / (4.0 * (last - first))).contiguous()
    nf = d(2 * nt)
    P_off = np.zeros(n + 1, np.int64)
    P_off[1:] = np.cumsum(2 * nt)
    dy = torch.exp(_uniform(g, int(off[-1]), math.log(0.3), math.log(3.0)))
    amp, fr = d(rs.uniform(0.2, 1.5, n)), d(rs.uniform(0.05, 0.95, n))
    X = 3.0 + dy * torch.randn(int(off[-1]), generator=g, device="cuda", dtype=torch.float64)
    X += amp[c] * torch.sin(2 * math.pi * ((fr * df * nf)[c] * t % 1.0))
    return {"t_off": d(off), "t": t, "X": X, "dy": dy, "f0": df, "df": df, "nf": nf, "P_off": d(P_off),
            "off": off, "poff": P_off, "nt": nt, "n": n}


def _weights(seed, out):
    """Flat network parameters: He-normal hidden layers, a small output layer, then 32 feature means and scales."""
    rs = np.random.default_rng(seed + 77)
    H = HIDDEN
    parts = []
    for fan, width, s in ((32, H, 1.0), (H, H, 1.0), (H, H, 1.0), (H, 9, out)):
        parts += [rs.normal(0.0, s * math.sqrt(2.0 / fan), fan * width), rs.normal(0.0, 0.02, width)]
    # means and scales of the features as training patterns have them
    mean = np.concatenate([[7.6, 5.1, 8.3, -1.4, 7.6, 0.7], [-4.5, -2.9, -1.7, -0.6, 0.3], [0.85, 0.4, 0.2, 0.2, 0.1],
                           np.linspace(0.8, 0.2, 8), np.full(8, 0.01)])
    return np.concatenate(parts + [mean, np.concatenate([np.full(16, 1.0), np.full(8, 0.2), np.full(8, 0.05)])]).astype(np.float32)


def _minibatch(case, seed):
    g, B = _gen(seed), case["rows"]
    nt = torch.floor(torch.exp(_uniform(g, B, math.log(200.0), math.log(20000.0))))
    mean = torch.from_numpy(_weights(0, 0.1)[-64:-32]).cuda().double()
    scale = torch.from_numpy(_weights(0, 0.1)[-32:]).cuda().double()
    feats = mean + scale * torch.randn(B, 32, generator=g, device="cuda", dtype=torch.float64)
    y = torch.log(2.0 * nt) - torch.log(-torch.log(_uniform(g, B, 1e-6, 1.0)))  # a Gumbel noise peak
    return feats.float().contiguous(), torch.stack([nt, 2.0 * nt], 1).float().contiguous(), y.float().contiguous()


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "ctx": lsp.Context(0), "seed": int(seed)}
    if kind in ("single", "gls", "pr"):
        s.update(_curve(case, seed))
        s["out"] = torch.empty(case["nf"], dtype=torch.float32, device="cuda")
    elif kind == "grad":
        s["ctx"].fap_set_params(_weights(seed, 0.1), hidden=HIDDEN)
        s["batch"] = _minibatch(case, seed)
    else:
        s.update(_patterns(case, seed))
        s["reals"] = case["reals"]
        s["maxP"] = torch.empty(case["reals"] * s["n"], dtype=torch.float32, device="cuda")
        s["argmax"] = torch.empty(s["n"], dtype=torch.int32, device="cuda")
        if kind == "batch":
            s["P"] = torch.empty(int(s["poff"][-1]), dtype=torch.float32, device="cuda")
        if kind == "predict":
            s["ctx"].fap_set_params(_weights(seed, 0.1), hidden=HIDDEN)
    return s


def run(s):
    ctx, kind = s["ctx"], s["kind"]
    if kind == "single":
        return ctx.periodogram(s["t"], s["X"], s["f0"], s["df"], s["nf"], out=s["out"])
    if kind == "gls":
        return ctx.periodogram_gls(s["t"], s["X"], s["f0"], s["df"], s["nf"], dy=s["dy"], out=s["out"])
    if kind == "pr":
        return ctx.press_rybicki(s["t"], s["X"], s["f0"], s["df"], s["nf"], out=s["out"])
    if kind == "grad":
        return ctx.fap_gradients(*s["batch"])
    grids = (s["f0"], s["df"], s["nf"])
    if kind == "batch":
        ctx.batch(s["t_off"], s["t"], *grids, X=s["X"], P_out=s["P"], P_off=s["P_off"], maxP=s["maxP"],
                  argmax=s["argmax"])
        return s["P"], s["maxP"], s["argmax"]
    if kind == "mc":
        ctx.batch(s["t_off"], s["t"], *grids, seed=s["seed"], n_real=s["reals"], maxP=s["maxP"])
        return s["maxP"]
    if kind == "batch_gls":
        ctx.batch_gls(s["t_off"], s["t"], s["X"], *grids, dy=s["dy"], maxP=s["maxP"], argmax=s["argmax"])
        return s["maxP"], s["argmax"]
    if kind == "mc_gls":
        ctx.batch_gls_noise(s["t_off"], s["t"], *grids, dy=s["dy"], seed=s["seed"], n_real=s["reals"], maxP=s["maxP"])
        return s["maxP"]
    return ctx.fap_predict(s["t_off"], s["t"], *grids)


def work(case):
    """Inputs once and outputs once; the multiply-adds of the sums over every (sample, frequency) term: four per term
    (XC, XS and the two window sums), six with weights and offset, the pattern's own sums once for all realizations; the
    spectral window two.  The approximation: an FFT of the grid; the network: its matrix products."""
    kind = case["kind"]
    if kind == "grad":
        B, H = case["rows"], HIDDEN
        macs = 32 * H + 2 * H * H + 9 * H
        p = macs + 3 * H + 9
        return {"bytes": B * 35 * 4 + p * 8, "flops": 2 * B * (3 * macs - 32 * H)}
    if kind in ("single", "gls", "pr"):
        n, nf = case["n"], case["nf"]
        arrays = 3 if kind == "gls" else 2
        if kind == "pr":
            m = 2 ** math.ceil(math.log2(8 * (nf + 1)))
            return {"bytes": 16 * n + 4 * nf, "flops": 5.0 * m * math.log2(m) + 60.0 * n}
        return {"bytes": 8 * arrays * n + 4 * nf, "flops": (12.0 if kind == "gls" else 8.0) * n * nf}
    nt = _sizes(case).astype(np.float64)
    total, terms, R = float(nt.sum()), float((2 * nt * nt).sum()), case["reals"]
    bytes_in = 8 * total * {"batch": 2, "mc": 1, "batch_gls": 3, "mc_gls": 2, "predict": 1}[kind] + 32 * nt.size
    if kind == "predict":
        return {"bytes": bytes_in + 36 * nt.size, "flops": 4 * terms}
    shared = 8.0 if kind in ("batch_gls", "mc_gls") else 4.0
    out = 8 * R * nt.size + (8 * total if kind == "batch" else 0)
    return {"bytes": bytes_in + out, "flops": terms * (shared + 4.0 * R)}


# ---------------------------------------------------------------- the same in 64 bits


def _sums(t, ys, f0, df, nf, h=1):
    """sum_j y_j exp(2 pi i h (f0 + k df) t_j) for k < nf, one row for each of ys: grid frequencies as a coarse one plus a
    fine offset, so that the sum is a complex matrix product."""
    fine = 512 if nf > 4096 else 64
    coarse = -(-nf // fine)
    fb = h * df * torch.arange(fine, device="cuda", dtype=torch.float64)
    fa = h * (f0 + df * fine * torch.arange(coarse, device="cuda", dtype=torch.float64))
    out = torch.zeros(len(ys), coarse, fine, dtype=torch.complex128, device="cuda")
    step = max(256, min(t.numel(), int(4e7) // max(coarse, fine)))
    turn = lambda p: torch.polar(torch.ones_like(p), 2 * math.pi * (p - torch.round(p)))  # noqa: E731
    for j in range(0, t.numel(), step):
        tj = t[j:j + step]
        A, B = turn(fa[:, None] * tj[None, :]), turn(tj[:, None] * fb[None, :])
        for i, y in enumerate(ys):
            out[i] += (A if y is None else A * y[j:j + step]) @ B
    return out.reshape(len(ys), -1)[:, :nf]


def _ratio(num, den, thr):
    return torch.where(den > thr, num.clamp_min(0.0) / den.clamp_min(1e-300), torch.zeros_like(num))


def _power(Z, W, n):
    """Eq. 5-6 from Z = XC + i XS and W = CC - SS + 2i CS; terms with a denominator up to n 2^-16 are left out."""
    R = W.abs()
    u = torch.where(R > 0, W / R.clamp_min(1e-300), torch.ones_like(W))
    z2, cross = Z.abs() ** 2, (u.conj() * Z * Z).real
    thr = n * 2.0 ** -16
    return 0.5 * (_ratio(0.5 * (z2 + cross), 0.5 * (n + R), thr) + _ratio(0.5 * (z2 - cross), 0.5 * (n - R), thr))


def _power_gls(Z, C, W, n):
    """(n / 2) p from Z = sum w x' e, C = sum w e, W = sum w e^2 (weights summing to 1, unit variance)."""
    M = W - C * C                          # CC - SS + 2i CS, centred
    T, R = 1.0 - C.abs() ** 2, M.abs()     # CC + SS, centred
    u = torch.where(R > 0, M / R.clamp_min(1e-300), torch.ones_like(M))
    z2, cross = Z.abs() ** 2, (u.conj() * Z * Z).real
    thr = 2.0 ** -24
    return 0.5 * n * (_ratio(0.5 * (z2 + cross), 0.5 * (T + R), thr) + _ratio(0.5 * (z2 - cross), 0.5 * (T - R), thr))


def _normal(X):
    X = X - X.mean(-1, keepdim=True)
    return X / torch.sqrt((X * X).mean(-1, keepdim=True))


def _weighted(X, w):
    X = X - (w * X).sum(-1, keepdim=True)
    return w * X / torch.sqrt((w * X * X).sum(-1, keepdim=True))


def _philox_normals(seed, curve, reals, n):
    """[reals, n] N(0,1) values: Philox-4x32-10 with counter (j/4, curve, realization, 0), then Box-Muller."""
    blocks = -(-n // 4)
    mask = 0xFFFFFFFF
    c = [torch.arange(blocks, device="cuda").repeat(reals), torch.full((blocks * reals,), curve, device="cuda"),
         torch.arange(reals, device="cuda").repeat_interleave(blocks), torch.zeros(blocks * reals, dtype=torch.int64, device="cuda")]
    k0, k1 = seed & mask, (seed >> 32) & mask
    mul = lambda a, m: (((a >> 16) * m + (((a & 0xFFFF) * m) >> 16)) >> 16, (a * m) & mask)  # noqa: E731  (hi, lo) words
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [(h1 ^ c[1] ^ k0) & mask, l1, (h0 ^ c[3] ^ k1) & mask, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u = [(2 * (w >> 9) + 1).double() * 2.0 ** -24 for w in c]
    z = []
    for a, b in ((u[0], u[1]), (u[2], u[3])):
        r = torch.sqrt(-2.0 * torch.log(a))
        z += [r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)]
    return torch.stack(z, 1).reshape(reals, 4 * blocks)[:, :n]


def _many_sums(t, Y, f0, df, nf):
    """Complex [R, nf] sums of many rows Y[R, n] over one pattern: blocks of frequencies, cos and sin times Y."""
    out = torch.empty(Y.shape[0], nf, dtype=torch.complex128, device="cuda")
    step = max(16, int(3e7) // t.numel())
    for k in range(0, nf, step):
        f = f0 + df * torch.arange(k, min(nf, k + step), device="cuda", dtype=torch.float64)
        p = t[:, None] * f[None, :]
        p = 2 * math.pi * (p - torch.round(p))
        out[:, k:k + step] = torch.complex(Y @ torch.cos(p), Y @ torch.sin(p))
    return out


def _features(t, f0, df, nf):
    n, T = t.numel(), float(t[-1] - t[0])
    gaps = t[1:] - t[:-1]
    srt = torch.sort(gaps).values
    q = [float(srt[int(math.floor(p * (n - 2)))]) for p in (0.05, 0.25, 0.5, 0.75, 0.95)]
    fmax = f0 + (nf - 1) * df
    f = [math.log(n), math.log(T), math.log(nf), math.log(1.0 / (df * T)), math.log(fmax * T / n), math.log1p(f0 / df)]
    f += [math.log(max(v, 1e-12 * T) / (T / (n - 1))) for v in q]
    r = gaps / q[2]
    f += [float(gaps[r > c * (1 + 1e-6)].sum()) / T for c in (2, 10, 100)]
    f += [float(gaps.max()) / T, float((r > 2 * (1 + 1e-6)).double().mean())]
    m = int(math.floor(fmax / df * (1 + 1e-12)))
    W = (_sums(t, [None], df, df, m)[0].abs() / n) ** 2
    i = torch.arange(1, m - 1, device="cuda")
    ok = (W[1:-1] > W[:-2]) & (W[1:-1] >= W[2:]) & ((i + 1).double() * df * T >= 1.0)
    top = torch.topk(W[i[ok]], min(8, int(ok.sum())))
    at = (i[ok][top.indices] + 1).double() * df / fmax
    pad = [0.0] * (8 - top.values.numel())
    return f + top.values.tolist() + pad + at.tolist() + pad


def _quantiles(flat, feats, counts):
    """The network and its head on Eq. 3's quantiles in 64 bits."""
    H, o, x = HIDDEN, 0, (feats - flat[-64:-32]) / flat[-32:]
    for i, (a, b) in enumerate(((32, H), (H, H), (H, H), (H, 9))):
        x = x @ flat[o:o + a * b].reshape(a, b) + flat[o + a * b:o + a * b + b]
        o += a * b + b
        if i < 3:
            x = torch.nn.functional.gelu(x)
    p = torch.tensor(LEVELS, device="cuda", dtype=torch.float64)
    N, Nf = counts[:, :1], counts[:, 1:]
    e = torch.log(0.5 * N) + torch.log(-torch.expm1(2.0 / (N - 3.0) * torch.log(-torch.expm1(torch.log(p) / Nf))))
    steps = (e[:, 1:] - e[:, :-1]) * torch.nn.functional.softplus(x[:, 1:]) / math.log(2.0)
    return torch.exp(torch.cumsum(torch.cat([e[:, :1] + x[:, :1], steps], 1), 1))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("single", "gls", "pr"):
        s = _curve(case, seed)
        t, grid = s["t"] - s["t"][0], (s["f0"], s["df"], s["nf"])
        n = t.numel()
        if kind == "single":
            return _power(_sums(t, [_normal(s["X"])], *grid)[0], _sums(t, [None], *grid, h=2)[0], n)
        if kind == "gls":
            w = s["dy"] ** -2 / (s["dy"] ** -2).sum()
            Z = _sums(t, [_weighted(s["X"], w), w], *grid)
            return _power_gls(Z[0], Z[1], _sums(t, [w], *grid, h=2)[0], n)
        m = 1  # Press & Rybicki's grid, four Lagrange nodes for each sample
        while m < 8 * (s["nf"] + 1):
            m *= 2
        z = torch.zeros(2, m, dtype=torch.float64, device="cuda")
        for i, y in enumerate((_normal(s["X"]), torch.ones_like(t))):
            p = (i + 1) * t * s["df"]
            pos = (p - torch.floor(p)) * m
            lo = torch.floor(pos) - 1
            d = pos - lo
            for a in range(4):
                wt = torch.ones_like(d)
                for b in range(4):
                    if b != a:
                        wt = wt * (d - b) / (a - b)
                z[i].index_add_(0, (lo.long() + a) % m, wt * y)
        F = torch.fft.ifft(z, dim=1, norm="forward")[:, 1:s["nf"] + 1]
        return _power(F[0], F[1], n)
    if kind == "grad":
        flat = torch.from_numpy(_weights(seed, 0.1)).cuda().double().requires_grad_(True)
        feats, counts, y = (v.double() for v in _minibatch(case, seed))
        u = y[:, None] - _quantiles(flat, feats, counts)
        p = torch.tensor(LEVELS, device="cuda", dtype=torch.float64)
        loss = torch.maximum(p * u, (p - 1.0) * u).sum(1).mean()
        return torch.autograd.grad(loss, flat)[0][:-64], float(loss.detach())
    s = _patterns(case, seed)
    f0, df, nf = (s[k].tolist() for k in ("f0", "df", "nf"))
    feats, best, full = [], [], []
    for c in range(s["n"]):
        a, b = s["off"][c], s["off"][c + 1]
        t, grid, n = s["t"][a:b] - s["t"][a], (f0[c], df[c], nf[c]), int(b - a)
        if kind == "predict":
            feats.append(_features(t, *grid))
            continue
        if kind in ("batch_gls", "mc_gls"):
            dy = s["dy"][a:b]
            w = dy ** -2 / (dy ** -2).sum()
            C, W = _sums(t, [w], *grid)[0], _sums(t, [w], *grid, h=2)[0]
            if kind == "batch_gls":
                P = _power_gls(_sums(t, [_weighted(s["X"][a:b], w)], *grid)[0], C, W, n)[None]
            else:
                X = dy * _philox_normals(int(seed), c, case["reals"], n).float().double()
                P = _power_gls(_many_sums(t, _weighted(X, w), *grid), C, W, n)
        else:
            W = _sums(t, [None], *grid, h=2)[0]
            if kind == "batch" or case["reals"] == 1:
                X = s["X"][a:b] if kind == "batch" else _philox_normals(int(seed), c, 1, n)[0]
                P = _power(_sums(t, [_normal(X)], *grid)[0], W, n)[None]
            else:
                P = _power(_many_sums(t, _normal(_philox_normals(int(seed), c, case["reals"], n)), *grid), W, n)
        best.append(P.max(dim=1).values)
        if kind == "batch":
            full.append(P[0])
    if kind == "predict":
        feats = torch.tensor(feats, dtype=torch.float64, device="cuda")
        counts = torch.from_numpy(np.column_stack([s["nt"], 2 * s["nt"]]).astype(np.float64)).cuda()
        return _quantiles(torch.from_numpy(_weights(seed, 0.1)).cuda().double(), feats, counts)
    peaks = torch.stack(best, 1).reshape(-1)
    if kind == "batch":
        return torch.cat(full), peaks, None
    return (peaks, None) if kind == "batch_gls" else peaks
