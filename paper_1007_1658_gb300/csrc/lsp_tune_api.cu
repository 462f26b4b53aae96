// lsp_tune_api.cu -- lsp_autotune: pick the sin/cos mode, strip length F
// (which is also the recurrence's re-seed length K) and N_t split for a
// problem size by timing candidates on the device, behind a precision gate; the
// tensor cores are a candidate where AUTO would take them.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>

#include "lsp_ctx.h"

using namespace lsp::host;

namespace {

int bucket(int64_t v) {
    int b = 0;
    while (v > 1) {
        v >>= 1;
        ++b;
    }
    return b;
}

}  // namespace

lsp::host::BatchBucket lsp::host::batch_bucket(int n_curves, int64_t total_samples, int64_t total_freqs, int n_real) {
    // terms per realization: sum over curves of N_t N_f, estimated from the
    // totals as (mean N_t) (total N_f) (the buckets are powers of two)
    const int64_t mean_nt = std::max<int64_t>(1, total_samples / std::max(1, n_curves));
    const double terms = (double)mean_nt * (double)std::max<int64_t>(1, total_freqs);
    BatchBucket b;
    b.terms = (int)std::floor(std::log2(std::max(1.0, terms)));
    b.mean_nt = bucket(mean_nt);
    b.real = n_real <= 1 ? 1 : (n_real < 4 ? 2 : (n_real < 8 ? 4 : 8));
    return b;
}

const lsp::host::BatchTuneEntry* lsp::host::tuned_batch(const lsp_ctx* ctx, const BatchBucket& b) {
    for (const BatchTuneEntry& e : ctx->tune_batch)
        if (e.bucket == b) return &e;
    return nullptr;
}

// Entry for (N_t, N_f) in the context's tuning table, or null.
const lsp::host::TuneEntry* lsp::host::tuned(const lsp_ctx* ctx, int64_t N, int64_t N_f) {
    const int a = bucket(N), b = bucket(N_f);
    for (const TuneEntry& e : ctx->tune)
        if (e.nt_bucket == a && e.nf_bucket == b) return &e;
    return nullptr;
}

extern "C" lsp_status lsp_autotune(lsp_ctx* ctx, int64_t N_t, int64_t N_f, lsp_options* chosen) {
    if (!ctx) return LSP_ERR_INVALID_ARG;
    ctx->err.clear();
    if (N_t < 2 || N_t > (int64_t(1) << 26) || N_f < 1 || N_f >= (int64_t(1) << 31))
        return fail(ctx, LSP_ERR_INVALID_ARG, "autotune sizes out of range");
    DeviceGuard guard(ctx->device);
    // synthetic input of the requested size: jittered even sampling, a sinusoid plus a deterministic
    // pseudo-random component (the kernels' cost does not depend on the values)
    std::vector<double> t((size_t)N_t), X((size_t)N_t);
    for (int64_t j = 0; j < N_t; ++j) {
        const double u = std::fmod((double)j * 0.6180339887498949, 1.0);
        t[(size_t)j] = (double)j + 0.45 * u;
        X[(size_t)j] = std::sin(0.37 * t[(size_t)j]) + (std::fmod((double)j * 0.7548776662466927, 1.0) - 0.5);
    }
    const double T = t.back() - t.front();
    const double df = 1.0 / (4.0 * T);
    DevBuf dt, dx, dp;
    auto release = [&]() {
        if (dt.p) cudaFree(dt.p);
        if (dx.p) cudaFree(dx.p);
        if (dp.p) cudaFree(dp.p);
    };
    lsp_status rs;
    if ((rs = ensure(ctx, dt, (size_t)N_t * 8)) != LSP_OK || (rs = ensure(ctx, dx, (size_t)N_t * 8)) != LSP_OK ||
        (rs = ensure(ctx, dp, (size_t)N_f * 4)) != LSP_OK) {
        release();
        return rs;
    }
    cudaMemcpy(dt.p, t.data(), (size_t)N_t * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dx.p, X.data(), (size_t)N_t * 8, cudaMemcpyHostToDevice);
    const lsp_options saved = ctx->opt;
    auto run = [&](int sincos, int F, int split, std::vector<float>* out, float* ms) -> lsp_status {
        lsp_options o = saved;
        o.sincos_mode = sincos;
        o.phase_mode = LSP_PHASE_FIXED64;
        o.freqs_per_thread = F;
        o.split = split;
        o.timing = 0;
        ctx->opt = o;
        cudaEvent_t e0 = ctx->ev[0], e1 = ctx->ev[3];
        lsp_status s = lsp_periodogram(ctx, (const double*)dt.p, (const double*)dx.p, N_t, df, df, N_f, (float*)dp.p);
        if (s != LSP_OK) return s;
        float best = 1e30f;
        for (int r = 0; r < 3; ++r) {
            cudaEventRecord(e0, ctx->stream);
            s = lsp_periodogram(ctx, (const double*)dt.p, (const double*)dx.p, N_t, df, df, N_f, (float*)dp.p);
            if (s != LSP_OK) return s;
            cudaEventRecord(e1, ctx->stream);
            if (cudaEventSynchronize(e1) != cudaSuccess) return fail(ctx, LSP_ERR_CUDA, "autotune timing");
            float m = 0.f;
            cudaEventElapsedTime(&m, e0, e1);
            best = std::min(best, m);
        }
        *ms = best;
        if (out) {
            out->resize((size_t)N_f);
            if (cudaMemcpy(out->data(), dp.p, (size_t)N_f * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
                return fail(ctx, LSP_ERR_CUDA, "autotune readback");
        }
        return LSP_OK;
    };
    // reference: hardware sin/cos for every term
    std::vector<float> ref, got;
    float ms = 0.f;
    if ((rs = run(LSP_SINCOS_MUFU, 8, 0, &ref, &ms)) != LSP_OK) {
        ctx->opt = saved;
        release();
        return rs;
    }
    float pmax = 0.f;
    for (float v : ref) pmax = std::max(pmax, v);
    struct Cand { int sincos, F; };
    const Cand cands[] = {{LSP_SINCOS_RECUR3_X2, 24}, {LSP_SINCOS_RECUR3_X2, 16}, {LSP_SINCOS_RECUR3_X2, 8},
                          {LSP_SINCOS_RECUR3_X2, 4},  {LSP_SINCOS_RECUR3, 24},    {LSP_SINCOS_RECUR, 16},
                          {LSP_SINCOS_RECUR, 8},      {LSP_SINCOS_MUFU, 8}};
    TuneEntry best{bucket(N_t), bucket(N_f), 0, 0, 0, 1e30f, 0};
    auto max_err = [&]() {
        float err = 0.f;
        for (size_t k = 0; k < got.size(); ++k) err = std::max(err, std::fabs(got[k] - ref[k]));
        return err;
    };
    for (const Cand& c : cands) {
        // the heuristic split of this candidate, then half and double of it
        ctx->opt = saved;
        ctx->opt.sincos_mode = c.sincos;
        ctx->opt.freqs_per_thread = c.F;
        ctx->opt.split = 0;
        const int base_split = choose_shape(ctx, N_t, N_f).split;
        const int max_split = (int)std::max<int64_t>(base_split, std::max<int64_t>(1, N_t / lsp::kMinChunk));
        const int splits[3] = {base_split, std::max(1, base_split / 2), std::min<int>(base_split * 2, max_split)};
        for (int si = 0; si < 3; ++si) {
            if (si > 0 && splits[si] == base_split) continue;
            if ((rs = run(c.sincos, c.F, splits[si], &got, &ms)) != LSP_OK) {
                ctx->opt = saved;
                release();
                return rs;
            }
            const float err = max_err();
            const bool pass = std::isfinite(err) && err <= 2e-5f * pmax;  // a fifth of the parity budget
            if (pass && ms < best.ms) best = TuneEntry{bucket(N_t), bucket(N_f), c.sincos, c.F, splits[si], ms, 0};
        }
    }
    // the tensor cores, with the table out of the way
    std::vector<TuneEntry> table;
    table.swap(ctx->tune);
    ctx->opt = saved;
    ctx->opt.sincos_mode = LSP_SINCOS_AUTO;
    ctx->opt.phase_mode = LSP_PHASE_FIXED64;
    ctx->opt.freqs_per_thread = ctx->opt.split = 0;
    if (use_tc(ctx, N_t, N_f, false)) {
        rs = run(LSP_SINCOS_AUTO, 0, 0, &got, &ms);
        const float err = rs == LSP_OK ? max_err() : 0.f;
        best.beat_tensor = !(std::isfinite(err) && err <= 2e-5f * pmax && ms < best.ms);
    }
    ctx->tune.swap(table);
    ctx->opt = saved;
    release();
    if (rs != LSP_OK) return rs;
    if (best.sincos == 0) return fail(ctx, LSP_ERR_CUDA, "autotune: no candidate passed the precision gate");
    ctx->tune.erase(std::remove_if(ctx->tune.begin(), ctx->tune.end(),
                                   [&](const TuneEntry& e) { return e.nt_bucket == best.nt_bucket && e.nf_bucket == best.nf_bucket; }),
                    ctx->tune.end());
    ctx->tune.push_back(best);
    if (chosen) {
        *chosen = saved;
        chosen->sincos_mode = best.sincos;
        chosen->freqs_per_thread = best.F;
        chosen->split = best.split;
    }
    return LSP_OK;
}

namespace {

lsp_status set_entry(lsp_ctx* ctx, const lsp::host::BatchTuneEntry& e) {
    auto& v = ctx->tune_batch;
    v.erase(std::remove_if(v.begin(), v.end(), [&](const lsp::host::BatchTuneEntry& x) { return x.bucket == e.bucket; }),
            v.end());
    v.push_back(e);
    return LSP_OK;
}

std::string device_name(int dev) {
    cudaDeviceProp p;
    if (cudaGetDeviceProperties(&p, dev) != cudaSuccess) {
        cudaGetLastError();
        return "unknown";
    }
    std::string n = p.name;
    for (char& c : n)
        if (c == '"' || c == '\\' || (unsigned char)c < 32) c = '_';
    return n;
}

// Value of "key": <number> on one line of the tuning file (NaN if absent).
double field(const char* line, const char* key) {
    char pat[64];
    snprintf(pat, sizeof pat, "\"%s\":", key);
    const char* p = strstr(line, pat);
    if (!p) return NAN;
    return strtod(p + strlen(pat), nullptr);
}

}  // namespace

extern "C" lsp_status lsp_autotune_batch(lsp_ctx* ctx, int32_t n_curves, const int64_t* t_off, const double* t,
                                         const double* f_0, const double* df, const int64_t* N_f, int32_t n_real,
                                         lsp_options* chosen) {
    if (!ctx) return LSP_ERR_INVALID_ARG;
    ctx->err.clear();
    if (n_curves < 1 || n_curves > 65535 || n_real < 1 || n_real > 65535 || !t_off || !t || !f_0 || !df || !N_f)
        return fail(ctx, LSP_ERR_INVALID_ARG, "bad batch description");
    DeviceGuard guard(ctx->device);
    lsp_status rs;
    std::vector<int64_t> off, nf;
    if ((rs = fetch(ctx, t_off, (size_t)n_curves + 1, off)) != LSP_OK) return rs;
    if ((rs = fetch(ctx, N_f, (size_t)n_curves, nf)) != LSP_OK) return rs;
    int64_t nf_total = 0;
    for (int c = 0; c < n_curves; ++c) nf_total += std::max<int64_t>(0, nf[c]);
    const BatchBucket bk = batch_bucket(n_curves, off[n_curves], nf_total, n_real);
    // per-periodogram maxima are the output that the Monte Carlo uses
    const size_t n_out = (size_t)n_real * (size_t)n_curves;
    DevBuf dmax, darg;
    auto release = [&]() {
        if (dmax.p) cudaFree(dmax.p);
        if (darg.p) cudaFree(darg.p);
    };
    if ((rs = ensure(ctx, dmax, n_out * 4)) != LSP_OK || (rs = ensure(ctx, darg, n_out * 4)) != LSP_OK) {
        release();
        return rs;
    }
    std::vector<BatchShape> cands;
    using lsp::kModeRecur3;
    if (n_real == 1) {
        // the packed strip in every tuned shape; the scalar one, bit-identical
        // and slower, at the default shape only
        for (int F : {24, 16})
            for (int tail : {8, 4, 0})
                for (int tile : {128, 256, 512}) cands.push_back({lsp::kModeRecur3x2, F, 1, tail, tile});
        cands.push_back({kModeRecur3, 24, 1, 8, lsp::kTile});
        cands.push_back({lsp::kModeRecur, 16, 1, 8, lsp::kTile});
    } else {
        for (int tile : {128, 256, 512}) {
            cands.push_back({kModeRecur3, 12, 4, 0, tile});
            cands.push_back({kModeRecur3, 8, 4, 0, tile});
        }
        cands.push_back({kModeRecur3, 16, 2, 0, lsp::kTile});
        cands.push_back({kModeRecur3, 4, 8, 0, lsp::kTile});
        cands.push_back({kModeRecur3, 8, 8, 0, lsp::kTile});
        cands.push_back({kModeRecur3, 24, 1, 8, lsp::kTile});
        // the packed strips of the same groups
        const int packed[][2] = {{12, 4}, {8, 4}, {16, 2}, {4, 8}, {8, 8}};
        for (const auto& fr : packed) cands.push_back({lsp::kModeRecur3x2, fr[0], fr[1], 0, lsp::kTile});
    }
    const lsp_options saved = ctx->opt;
    lsp_options o = saved;
    o.timing = 1;
    ctx->opt = o;
    std::vector<float> ref_max, got_max;
    BatchTuneEntry best{bk, {0, 0, 0, 0, 0}, 1e30f};
    const uint64_t seed = 0x5eed7u;
    for (const BatchShape& sh : cands) {
        if (sh.R > n_real) continue;
        const int occ = sh.R > 1 ? lsp::mrhs_occupancy(sh.mode, sh.F, sh.R, sh.tile, false)
                                 : lsp::batch_occupancy(sh.mode, sh.F, true, sh.tailF, sh.tile);
        if (occ <= 0) continue;
        float ms = 1e30f;
        for (int r = 0; r < 3 && rs == LSP_OK; ++r) {  // first call captures the graph, then two timed replays
            rs = batch_run(ctx, n_curves, t_off, t, nullptr, seed, n_real, f_0, df, N_f, nullptr, nullptr,
                           (float*)dmax.p, (int32_t*)darg.p, &sh);
            if (rs != LSP_OK) break;
            float a = 0.f, b = 0.f, c = 0.f;
            if ((rs = lsp_last_timing(ctx, &a, &b, &c)) != LSP_OK) break;
            if (r > 0) ms = std::min(ms, b);
        }
        if (rs != LSP_OK) break;
        got_max.resize(n_out);
        if (cudaMemcpy(got_max.data(), dmax.p, n_out * 4, cudaMemcpyDeviceToHost) != cudaSuccess) {
            rs = fail(ctx, LSP_ERR_CUDA, "autotune readback");
            break;
        }
        // every shape computes the same maxima up to FP32 rounding order:
        // keep only those within 2e-5 (relative) of the first candidate's
        if (ref_max.empty()) ref_max = got_max;
        float err = 0.f;
        for (size_t i = 0; i < n_out; ++i)
            err = std::max(err, std::fabs(got_max[i] - ref_max[i]) / std::max(ref_max[i], 1e-30f));
        if (std::isfinite(err) && err <= 2e-5f && ms < best.ms) best = BatchTuneEntry{bk, sh, ms};
    }
    ctx->opt = saved;
    release();
    if (rs != LSP_OK) return rs;
    if (best.shape.F == 0) return fail(ctx, LSP_ERR_CUDA, "autotune: no batch shape ran");
    set_entry(ctx, best);
    if (chosen) {
        *chosen = saved;
        chosen->sincos_mode = best.shape.mode == lsp::kModeRecur     ? LSP_SINCOS_RECUR
                              : best.shape.mode == lsp::kModeRecur3x2 ? LSP_SINCOS_RECUR3_X2
                                                                      : LSP_SINCOS_RECUR3;
        chosen->freqs_per_thread = best.shape.F;
        chosen->batch_rhs = best.shape.R;
    }
    return LSP_OK;
}

extern "C" lsp_status lsp_tune_save(lsp_ctx* ctx, const char* path) {
    if (!ctx || !path) return LSP_ERR_INVALID_ARG;
    ctx->err.clear();
    FILE* f = fopen(path, "w");
    if (!f) return fail(ctx, LSP_ERR_INVALID_ARG, "cannot write %s", path);
    fprintf(f, "{\"lsp_tune\": 1, \"device\": \"%s\", \"entries\": [\n", device_name(ctx->device).c_str());
    size_t n = 0, total = ctx->tune.size() + ctx->tune_batch.size();
    for (const TuneEntry& e : ctx->tune)
        fprintf(f,
                "{\"kind\": 1, \"nt\": %d, \"nf\": %d, \"sincos\": %d, \"F\": %d, \"split\": %d, \"ms\": %.6g, "
                "\"beat_tensor\": %d}%s\n",
                e.nt_bucket, e.nf_bucket, e.sincos, e.F, e.split, e.ms, e.beat_tensor, ++n < total ? "," : "");
    for (const BatchTuneEntry& e : ctx->tune_batch)
        fprintf(f,
                "{\"kind\": 2, \"terms\": %d, \"mean_nt\": %d, \"real\": %d, \"mode\": %d, \"F\": %d, \"R\": %d, "
                "\"tailF\": %d, \"tile\": %d, \"ms\": %.6g}%s\n",
                e.bucket.terms, e.bucket.mean_nt, e.bucket.real, e.shape.mode, e.shape.F, e.shape.R, e.shape.tailF,
                e.shape.tile, e.ms, ++n < total ? "," : "");
    fprintf(f, "]}\n");
    const bool ok = fclose(f) == 0;
    return ok ? LSP_OK : fail(ctx, LSP_ERR_INVALID_ARG, "cannot write %s", path);
}

extern "C" lsp_status lsp_tune_load(lsp_ctx* ctx, const char* path, int32_t* n_loaded) {
    if (!ctx || !path) return LSP_ERR_INVALID_ARG;
    ctx->err.clear();
    FILE* f = fopen(path, "r");
    if (!f) return fail(ctx, LSP_ERR_INVALID_ARG, "cannot read %s", path);
    char line[1024];
    int loaded = 0;
    bool header = false, same_device = false;
    const std::string want = "\"device\": \"" + device_name(ctx->device) + "\"";
    DeviceGuard guard(ctx->device);
    while (fgets(line, sizeof line, f)) {
        if (!header) {
            header = strstr(line, "\"lsp_tune\": 1") != nullptr;
            same_device = strstr(line, want.c_str()) != nullptr;
            if (!header) break;
            continue;
        }
        if (!same_device) break;
        const double kind = field(line, "kind");
        if (kind == 1) {
            TuneEntry e{(int)field(line, "nt"), (int)field(line, "nf"), (int)field(line, "sincos"), (int)field(line, "F"),
                        (int)field(line, "split"), (float)field(line, "ms"), field(line, "beat_tensor") == 1.0};
            lsp_options o = ctx->opt;
            o.sincos_mode = e.sincos;
            o.freqs_per_thread = e.F;
            o.split = e.split;
            if (e.sincos < 1 || e.sincos > 4 || e.F < 4 || e.F > 28 || e.F % 4 || e.split < 1 || e.split > 65535)
                continue;
            ctx->tune.erase(std::remove_if(ctx->tune.begin(), ctx->tune.end(),
                                           [&](const TuneEntry& x) {
                                               return x.nt_bucket == e.nt_bucket && x.nf_bucket == e.nf_bucket;
                                           }),
                            ctx->tune.end());
            ctx->tune.push_back(e);
            ++loaded;
        } else if (kind == 2) {
            BatchTuneEntry e{{(int)field(line, "terms"), (int)field(line, "mean_nt"), (int)field(line, "real")},
                             {(int)field(line, "mode"), (int)field(line, "F"), (int)field(line, "R"),
                              (int)field(line, "tailF"), (int)field(line, "tile")},
                             (float)field(line, "ms")};
            // only shapes this build has
            const int occ = e.shape.R > 1 ? lsp::mrhs_occupancy(e.shape.mode, e.shape.F, e.shape.R, e.shape.tile, false)
                                          : lsp::batch_occupancy(e.shape.mode, e.shape.F, true, e.shape.tailF,
                                                                 e.shape.tile);
            if (occ <= 0) continue;
            set_entry(ctx, e);
            ++loaded;
        }
    }
    fclose(f);
    if (!header) return fail(ctx, LSP_ERR_INVALID_ARG, "%s is not a tuning file", path);
    if (n_loaded) *n_loaded = loaded;
    return LSP_OK;
}
