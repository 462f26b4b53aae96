// features.cu -- sampling-pattern features for the learned false-alarm
// surrogate.
//
// The paper's false-alarm probability (Eq. 3) takes the N_f frequencies of a
// periodogram as independent; Sec. 6.2 notes that the exponent should really
// be an empirical number of independent frequencies, which depends on the
// sampling pattern.  The surrogate predicts the noise-peak quantiles from 32
// features of the pattern (definitions in include/lsp.h, lsp_fap_features).
// Two kernels:
//   ls_window_kernel  -- the spectral window W(f) = |sum_j e^{2 pi i f t_j}|^2 / N^2
//                        on f_m = m df, m = 1..floor(f_max / df): the same
//                        persistent tile loop as the batch periodogram, x = 1;
//   features_kernel   -- one CTA per pattern: cadence order statistics (a
//                        radix select of the five ranks over the gaps, in
//                        shared memory up to 32,768 of them), gap fractions,
//                        and the 8 highest window maxima outside the main lobe
//                        (per-thread top-8 lists merged by warp shuffles).
// With work enough the window comes from the tensor cores (tc_sums.cu), and the
// strip kernel's values are formed only at the few bins that can be among its 8
// highest maxima (window_peaks_kernel, window_exact_kernel): the features keep
// their bits; 256 patterns of up to 20,000 samples, the call 3.4 ms -> 1.1.
#include <algorithm>
#include <cfloat>

#include "ls_device.cuh"

namespace lsp {
namespace {

using namespace dev;

constexpr int kFeatThreads = 1024;
constexpr int kSortMaxGaps = 32768;  // gaps held in shared memory (128 KB); more are formed from t in every pass

// The five cadence order statistics sorted(gaps)[k[i]], without sorting: an
// MSB-first radix select on the FP32 bit patterns of the gaps (ordered as the
// values, gaps being >= 0), 8 bits per pass and the five ranks at once; key_at(i)
// is gap i's.  A warp whose gaps all fall into one bin adds to it once, so the
// equal gaps of an even cadence do not serialize on one counter; ranks whose
// leading bits a warp's gaps do not have cost it one vote.  hist holds 5 x 256 counters; out[i] receives the value of rank k[i].
template <class Key>
__device__ void select_gap_ranks(Key&& key_at, int M, const int (&k)[5], unsigned* hist, float* out) {
    __shared__ unsigned s_prefix[5], s_rank[5];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    if (tid < 5) {
        s_prefix[tid] = 0u;
        s_rank[tid] = (unsigned)k[tid];
    }
    unsigned mask = 0u;
    for (int shift = 24; shift >= 0; shift -= 8) {
        for (int i = tid; i < 5 * 256; i += nt) hist[i] = 0u;
        __syncthreads();
        unsigned prefix[5];
#pragma unroll
        for (int q = 0; q < 5; ++q) prefix[q] = s_prefix[q];
        // the whole warp steps together so that every lane takes part in the votes
        for (int base = tid - lane; base < M; base += nt) {
            const int i = base + lane;
            unsigned key = 0u;
            if (i < M) key = key_at(i);
            const int bin = (int)((key >> shift) & 255u);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                if (q && !mask) break;  // the first pass counts the same for all five
                const int mine = (i < M && (key & mask) == prefix[q]) ? bin : -1;
                const unsigned some = __ballot_sync(0xffffffffu, mine >= 0);
                if (!some) continue;
                const int lead = __ffs(some) - 1;
                const unsigned peers = __ballot_sync(0xffffffffu, mine == __shfl_sync(0xffffffffu, mine, lead));
                if (peers != some) {
                    if (mine >= 0) atomicAdd(&hist[q * 256 + mine], 1u);
                } else if (lane == lead) {
                    atomicAdd(&hist[q * 256 + mine], (unsigned)__popc(some));
                }
            }
        }
        __syncthreads();
        if (tid < 5 * 32) {
            // warp q: the bin holding rank s_rank[q], lane l counting bins 8 l .. 8 l + 7;
            // ranks below it move to the next pass's count
            const int w = tid >> 5;
            const unsigned* h = hist + (mask ? w * 256 : 0) + 8 * lane;
            const unsigned r = s_rank[w];
            unsigned cnt[8], sum = 0u;
#pragma unroll
            for (int x = 0; x < 8; ++x) sum += cnt[x] = h[x];
            unsigned acc = sum;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned v = __shfl_up_sync(0xffffffffu, acc, o);
                if (lane >= o) acc += v;
            }
            const unsigned past = __ballot_sync(0xffffffffu, acc > r);
            if (lane == (past ? __ffs(past) - 1 : 31)) {
                acc -= sum;
                int x = 0;
#pragma unroll
                for (int y = 0; y < 7; ++y)
                    if (x == y && acc + cnt[y] <= r) {
                        acc += cnt[y];
                        x = y + 1;
                    }
                s_rank[w] = r - acc;
                s_prefix[w] |= (unsigned)(8 * lane + x) << shift;
            }
        }
        mask |= 255u << shift;
        __syncthreads();
    }
    if (tid < 5) out[tid] = __uint_as_float(s_prefix[tid]);
    __syncthreads();
}

// The sums of e^{2 pi i f t} of a strip of F frequencies: Strip<F, kRecur3x2>'s
// seed, steps and order with x = 1 and without CC and CS, so its XC and XS bit
// for bit (1 y + s and y + s round alike; the network behind the features takes
// BF16 activations, where a last bit more or less shows).  U samples step through the strip
// together: a sample's recurrence is one chain of F steps, and a curve of a small
// batch has a sub-partition to itself, so only the other samples can fill the
// pipe meanwhile (256 patterns of 200 .. 20,000 samples, 8 CTAs an SM: U = 2, 4, 6
// 3.61, 3.39, 3.27 ms; 48 patterns 1.73, 1.37, 1.33).
template <int F>
struct UnitStrip {
    float2 s[F];  // g_i (C, S) of frequency i, the signs folded as there

    template <int U>
    __device__ __forceinline__ void add(const uint4* a, const float4* b, uint32_t k0) {
        float2 y0[U], y1[U], c2[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint4 Bu = lds128(b + u);
            const float C = __uint_as_float(Bu.y), S = __uint_as_float(Bu.z);
            float sn, cs;
            __sincosf(phase_to_angle(top_phase(lds128(a + u), k0)), &sn, &cs);
            y0[u] = make_float2(cs, sn);
            y1[u] = make_float2(fmaf(cs, C, -sn * S), fmaf(sn, C, cs * S));
            c2[u] = make_float2(__uint_as_float(Bu.w), -__uint_as_float(Bu.w));
        }
#pragma unroll
        for (int u = 0; u < U; ++u) s[0] = __fadd2_rn(s[0], y0[u]);
#pragma unroll
        for (int u = 0; u < U; ++u) s[1] = __fadd2_rn(s[1], y1[u]);
#pragma unroll
        for (int i = 2; i < F; ++i) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float c = ((i - 1) & 1) ? c2[u].y : c2[u].x;
                const float2 y2 = __ffma2_rn(make_float2(c, c), y1[u], y0[u]);
                s[i] = __fadd2_rn(s[i], y2);
                y0[u] = y1[u];
                y1[u] = y2;
            }
        }
    }
};

template <int F>
__global__ void __launch_bounds__(kMainThreads)
ls_window_kernel(const BatchItem* __restrict__ items, int n_items, unsigned* __restrict__ head,
                 const int64_t* __restrict__ off, const int64_t* __restrict__ nw, const uint4* __restrict__ recA,
                 const float4* __restrict__ recB, float* __restrict__ W, const int64_t* __restrict__ W_off,
                 const int* __restrict__ peaks) {
    __shared__ __align__(16) TileSmem<false> sm;
    __shared__ int s_item;
    for (;;) {
        if (threadIdx.x == 0) s_item = (int)atomicAdd(head, 1u);
        __syncthreads();
        const int it = s_item;
        __syncthreads();
        if (it >= n_items) break;
        const BatchItem w = items[it];
        if (peaks && peaks[(size_t)w.curve * (kWindowPeaks + 1)] >= 0) continue;  // its bins are formed one by one
        const int64_t b = off[w.curve], e = off[w.curve + 1];
        const int64_t M = nw[w.curve];
        const uint32_t k0 = (uint32_t)w.fblock * (kMainThreads * F) + (uint32_t)threadIdx.x * F;
        UnitStrip<F> st;
#pragma unroll
        for (int i = 0; i < F; ++i) st.s[i] = make_float2(0.f, 0.f);
        constexpr int U = 6;
        const bool live = k0 < (uint32_t)M;  // padding strips only help stage the tiles
        for_each_tile<false>(sm, recA, recB, nullptr, b, e, [&](const uint4* a, const float4* bb, const float*, int n) {
            if (!live) return;
            int j = 0;
#pragma unroll 1
            for (; j + U <= n; j += U) st.template add<U>(a + j, bb + j, k0);
#pragma unroll 1
            for (; j < n; ++j) st.template add<1>(a + j, bb + j, k0);
        });
        const float inv = 1.f / ((float)(e - b) * (float)(e - b));
        float* out = W + W_off[w.curve];
#pragma unroll
        for (int i = 0; i < F; ++i)
            if (k0 + i < (uint32_t)M) {
                const float2 z = st.s[i];  // the sign falls out of the squares
                out[k0 + i] = (z.x * z.x + z.y * z.y) * inv;
            }
    }
}

// W of single bins as ls_window_kernel forms it, bit for bit.  There a thread
// adds a strip's samples in order, one long chain; but only the additions are a
// chain.  Here a CTA takes a bin and its two neighbours: three warps form the
// terms of the next 384 samples (the strip's seed and the steps up to the last of
// the bins, four samples abreast; a second strip's where the three straddle one's
// end) while three lanes of the first warp add this chunk's, a bin each, in order.
// Bound by that chain, 20,000 additions for the largest patterns; with one warp
// forming and adding in turn 256 patterns took 463 us here, now 154; 48 362, now 79.
constexpr int kExactThreads = 128, kExactU = 4, kExactSamples = (kExactThreads - 32) * kExactU;
template <int F>
__global__ void __launch_bounds__(kExactThreads)
window_exact_kernel(const int64_t* __restrict__ off, const uint4* __restrict__ recA, const float4* __restrict__ recB,
                    const int* __restrict__ peaks, float* __restrict__ peak_w) {
    __shared__ __align__(16) float2 terms[2][3][kExactSamples + 2];
    const int c = blockIdx.x, tid = threadIdx.x, i = blockIdx.y;
    const int* p = peaks + (size_t)c * (kWindowPeaks + 1);
    if (i >= p[0]) return;
    const uint32_t kf = (uint32_t)(p[1 + i] - 1);  // the first of the three bins
    const int64_t b = off[c], e = off[c + 1];
    constexpr int U = kExactU;
    float2 s = make_float2(0.f, 0.f);
    const int chunks = (int)((e - b + kExactSamples - 1) / kExactSamples);
    for (int x0 = 0; x0 <= chunks; ++x0) {
        if (tid >= 32 && x0 < chunks) {
            const int64_t j0 = b + (int64_t)x0 * kExactSamples;
            const int at = tid - 32;
            float2(&out)[3][kExactSamples + 2] = terms[x0 & 1];
            uint4 A[U];
            float4 B[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int64_t j = min(j0 + at + (kExactThreads - 32) * u, e - 1);
                A[u] = recA[j];
                B[u] = recB[j];
            }
            // strips of the three bins: k0 = F (kf / F), and the next one where they reach into it
            for (uint32_t k0 = kf / F * F; k0 <= kf + 2; k0 += F) {
                const int first = (int)kf - (int)k0, last = min(first + 2, F - 1);  // the bins' steps in this strip
                float2 y0[U], y1[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    float sn, cs;
                    __sincosf(phase_to_angle(top_phase(A[u], k0)), &sn, &cs);
                    y0[u] = make_float2(cs, sn);
                    y1[u] = make_float2(fmaf(cs, B[u].y, -sn * B[u].z), fmaf(sn, B[u].y, cs * B[u].z));
                }
                auto put = [&](int step, const float2 (&y)[U]) {
                    if (step < first || step > last) return;
#pragma unroll
                    for (int u = 0; u < U; ++u) out[step - first][at + (kExactThreads - 32) * u] = y[u];
                };
                put(0, y0);
                put(1, y1);
#pragma unroll 1
                for (int x = 2; x <= last; ++x) {
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        const float cx = ((x - 1) & 1) ? -B[u].w : B[u].w;
                        const float2 y2 = __ffma2_rn(make_float2(cx, cx), y1[u], y0[u]);
                        y0[u] = y1[u];
                        y1[u] = y2;
                    }
                    put(x, y1);
                }
            }
        }
        if (tid < 3 && x0) {
            const int64_t j0 = b + (int64_t)(x0 - 1) * kExactSamples;
            const int n = (int)min((int64_t)kExactSamples, e - j0);
            const float2* y = terms[(x0 - 1) & 1][tid];
            int j = 0;
            for (; j + 16 <= n; j += 16) {
                float4 v[8];
#pragma unroll
                for (int x = 0; x < 8; ++x) v[x] = *reinterpret_cast<const float4*>(&y[j + 2 * x]);
#pragma unroll
                for (int x = 0; x < 8; ++x) {
                    s = __fadd2_rn(s, make_float2(v[x].x, v[x].y));
                    s = __fadd2_rn(s, make_float2(v[x].z, v[x].w));
                }
            }
            for (; j < n; ++j) s = __fadd2_rn(s, y[j]);
        }
        __syncthreads();
    }
    if (tid < 3) {
        const float inv = 1.f / ((float)(e - b) * (float)(e - b));
        const float2 z = s;
        peak_w[(size_t)c * (3 * kWindowPeaks) + 3 * i + tid] = (z.x * z.x + z.y * z.y) * inv;
    }
}

// (value, bin) ordered by value, then by lower bin.
__device__ __forceinline__ bool better(float v, int m, float v2, int m2) { return v > v2 || (v == v2 && m < m2); }

__device__ __forceinline__ void top8_insert(float (&v)[8], int (&m)[8], float x, int mi) {
    if (!better(x, mi, v[7], m[7])) return;
    int p = 7;
    while (p > 0 && better(x, mi, v[p - 1], m[p - 1])) {
        v[p] = v[p - 1];
        m[p] = m[p - 1];
        --p;
    }
    v[p] = x;
    m[p] = mi;
}

// The 8 best (value, bin) of a warp's lanes' lists, best first, through put(r,
// value, bin) on lane 0: eight rounds of "best head in the warp wins".
template <class Put>
__device__ __forceinline__ void warp_top8(const float (&tv)[8], const int (&tm)[8], Put&& put) {
    const int lane = threadIdx.x & 31;
    int headp = 0;
    for (int r = 0; r < 8; ++r) {
        float bv = -1.f;
        int bm = 0x7fffffff, bl = lane;
#pragma unroll
        for (int x = 0; x < 8; ++x)
            if (x == headp) {
                bv = tv[x];
                bm = tm[x];
            }
        for (int o = 16; o > 0; o >>= 1) {
            const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
            const int om = __shfl_xor_sync(0xffffffffu, bm, o);
            const int ol = __shfl_xor_sync(0xffffffffu, bl, o);
            if (better(ov, om, bv, bm)) {
                bv = ov;
                bm = om;
                bl = ol;
            }
        }
        if (lane == bl) ++headp;
        if (lane == 0) put(r, bv, bm);
    }
}

// How far the strip kernel's W and an accurate one can be apart, for n samples: its
// recurrence is off by at most F^2 ulp a term (3.4e-5) and its hardware sin/cos by
// less, 1e-4 of |sum| / n <= sqrt(W) together; and each of its FP32 additions by
// half an ulp of the running sum, 2^-24 j after j samples, n 2^-25 of the whole
// (where the terms repeat, on a cadence at its aliases, those roundings have one
// sign: up to 1.3e-4 and 3.7e-4 of n at 20,000 and 32,700 samples).  e bounds
// ||sum| - |sum'|| / n, so |W - W'| <= e (2 sqrt(W) + e).
__device__ __forceinline__ float window_error(int64_t n) { return 1e-4f + (float)n * 0x1p-25f; }
__device__ __forceinline__ float window_gap(float w, float e) { return e * (2.f * sqrtf(w) + e); }

// A pattern's bins that can hold one of the 8 highest local maxima (outside the
// main lobe) of the strip kernel's W: with g the gap above, maxima of the accurate
// W by more than the gaps of both bins are maxima of the other too; the eighth of
// those bounds the eighth of all from below; and a bin qualifies when it is a
// maximum up to the gaps and not below that bound.
constexpr int kPeakMaxSamples = 65536;
__global__ void __launch_bounds__(kFeatThreads)
window_peaks_kernel(const double* __restrict__ t, const int64_t* __restrict__ off, const double* __restrict__ dfa,
                    const float* __restrict__ W, const int64_t* __restrict__ W_off, const int64_t* __restrict__ nw,
                    int* __restrict__ peaks) {
    __shared__ float wv[32 * 8];
    __shared__ float s_eighth;
    __shared__ int s_n;
    const int c = blockIdx.x, tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5;
    const int64_t b = off[c], e = off[c + 1], mw = nw[c];
    const double df = dfa[c], T = t[e - 1] - t[b];
    const float* Wc = W + W_off[c];
    int* p = peaks + (size_t)c * (kWindowPeaks + 1);
    if (e - b > kPeakMaxSamples) {
        if (tid == 0) p[0] = -1;
        return;
    }
    const float err = window_error(e - b);
    float tv[8];
    int tm[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        tv[r] = -1.f;
        tm[r] = 0x7fffffff;
    }
    if (tid == 0) s_n = 0;
    for (int64_t i = 1 + tid; i + 1 < mw; i += nt) {
        const float w = Wc[i], l = Wc[i - 1], h = Wc[i + 1], g = window_gap(w, err);
        if (w - g > l + window_gap(l, err) && w - g > h + window_gap(h, err) && (double)(i + 1) * df * T >= 1.0)
            top8_insert(tv, tm, w - g, (int)i);
    }
    warp_top8(tv, tm, [&](int r, float v, int) { wv[warp * 8 + r] = v; });
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            tv[r] = wv[tid * 8 + r];
            tm[r] = tid * 8 + r;
        }
        warp_top8(tv, tm, [&](int r, float v, int) {
            if (r == 7) s_eighth = v;
        });
    }
    __syncthreads();
    const float least = s_eighth;  // -1 where there are fewer than eight
    for (int64_t i = 1 + tid; i + 1 < mw; i += nt) {
        const float w = Wc[i], g = window_gap(w, err);
        if (!(w + g >= least)) continue;
        const float l = Wc[i - 1], h = Wc[i + 1];
        if (w + g >= l - window_gap(l, err) && w + g >= h - window_gap(h, err) && (double)(i + 1) * df * T >= 1.0) {
            const int at = atomicAdd(&s_n, 1);
            if (at < kWindowPeaks) p[1 + at] = (int)i;
        }
    }
    __syncthreads();
    if (tid == 0) p[0] = s_n <= kWindowPeaks ? s_n : -1;
}

// One CTA per pattern.  Dynamic shared memory: the gaps of patterns of up to
// kSortMaxGaps of them, behind the select's histograms.
__global__ void __launch_bounds__(kFeatThreads)
features_kernel(const double* __restrict__ t, const int64_t* __restrict__ off, const double* __restrict__ f0a,
                const double* __restrict__ dfa, const int64_t* __restrict__ nfa, const float* __restrict__ W,
                const int64_t* __restrict__ W_off, const int64_t* __restrict__ nw, float* __restrict__ feat,
                int* __restrict__ status, const int* __restrict__ peaks, const float* __restrict__ peak_w) {
    extern __shared__ unsigned hist[];
    float* const gaps = reinterpret_cast<float*>(hist + 5 * 256);
    __shared__ double red[33];
    __shared__ float wv[32 * 8];
    __shared__ int wm[32 * 8];
    __shared__ int unsorted;
    __shared__ float qsel[5];
    const int c = blockIdx.x;
    const int tid = threadIdx.x, nt = blockDim.x;
    const int64_t b = off[c], e = off[c + 1];
    const int n = (int)(e - b), M = n - 1;
    const double ps[5] = {0.05, 0.25, 0.5, 0.75, 0.95};
    const bool in_smem = M <= kSortMaxGaps;
    if (tid == 0) unsorted = 0;
    __syncthreads();
    const double T = t[e - 1] - t[b];
    for (int i = tid; i < M; i += nt) {
        const double d = t[b + i + 1] - t[b + i];
        if (d < 0.0) unsorted = 1;
        if (in_smem) gaps[i] = (float)d;
    }
    __syncthreads();
    // q(ps[i]) = sorted(gaps)[floor(ps[i] (M - 1))]; the median is q(1/2)
    int rank[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) rank[i] = (int)floor(ps[i] * (double)(M - 1));
    if (in_smem) select_gap_ranks([&](int i) { return __float_as_uint(gaps[i]); }, M, rank, hist, qsel);
    else select_gap_ranks([&](int i) { return __float_as_uint((float)(t[b + i + 1] - t[b + i])); }, M, rank, hist, qsel);
    auto q = [&](int i) { return qsel[i]; };
    const double med = (double)q(2);
    // gap sums over dt > c med (1 + 1e-6): the margin keeps exact multiples of
    // the cadence (one dropped sample on an even grid) out of the gaps
    double s2 = 0.0, s10 = 0.0, s100 = 0.0, cnt2 = 0.0, mx = 0.0;
    // (FP64 divisions are slow on this part: a gap that FP32 puts clearly below
    // every bound and below the largest so far is done with)
    const float low = 1.999f * (float)med;
    float mx32 = 0.f;
    for (int i = tid; i < M; i += nt) {
        if (in_smem && gaps[i] < low && gaps[i] < mx32) continue;
        const double d = t[b + i + 1] - t[b + i];
        mx32 = fmaxf(mx32, (float)d);
        const double r = d / med;
        if (r > 2.0 * (1.0 + 1e-6)) {
            s2 += d;
            cnt2 += 1.0;
        }
        if (r > 10.0 * (1.0 + 1e-6)) s10 += d;
        if (r > 100.0 * (1.0 + 1e-6)) s100 += d;
        mx = fmax(mx, d);
    }
    auto bsum = [&](double v) {
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        __syncthreads();
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        double r = tid < (nt >> 5) ? red[tid] : 0.0;
        if (tid < 32)
            for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
        if (tid == 0) red[32] = r;
        __syncthreads();
        return red[32];
    };
    auto bmax = [&](double v) {
        for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
        __syncthreads();
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        double r = tid < (nt >> 5) ? red[tid] : 0.0;
        if (tid < 32)
            for (int o = 16; o > 0; o >>= 1) r = fmax(r, __shfl_down_sync(0xffffffffu, r, o));
        if (tid == 0) red[32] = r;
        __syncthreads();
        return red[32];
    };
    s2 = bsum(s2);
    s10 = bsum(s10);
    s100 = bsum(s100);
    cnt2 = bsum(cnt2);
    mx = bmax(mx);

    // window maxima outside the main lobe: interior m with W[m] > W[m-1], W[m] >= W[m+1], f_m T >= 1
    const double df = dfa[c], f0 = f0a[c];
    const int64_t nf = nfa[c];
    const double f_max = f0 + (double)(nf - 1) * df;
    const int64_t mw = nw[c];
    const float* Wc = W + W_off[c];
    float tv[8];
    int tm[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        tv[r] = -1.f;
        tm[r] = 0x7fffffff;
    }
    const int* pk = peaks ? peaks + (size_t)c * (kWindowPeaks + 1) : nullptr;
    if (pk && pk[0] >= 0) {
        if (tid < pk[0]) {
            const float* x = peak_w + (size_t)c * (3 * kWindowPeaks) + 3 * tid;
            if (x[1] > x[0] && x[1] >= x[2]) top8_insert(tv, tm, x[1], pk[1 + tid]);
        }
    } else {
        for (int64_t i = 1 + tid; i + 1 < mw; i += nt) {
            const float w = Wc[i];
            if (w > Wc[i - 1] && w >= Wc[i + 1] && (double)(i + 1) * df * T >= 1.0) top8_insert(tv, tm, w, (int)i);
        }
    }
    const int warp = tid >> 5;
    warp_top8(tv, tm, [&](int r, float v, int m) {
        wv[warp * 8 + r] = v;
        wm[warp * 8 + r] = m;
    });
    __syncthreads();
    if (tid < 32) {
        // the warps' lists, then one output a lane: 11 logarithms and as many
        // divisions in FP64 take one thread longer than a pass over the gaps
        __shared__ float fv[8];
        __shared__ int fm[8];
        const bool has = tid < (nt >> 5);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            tv[r] = has ? wv[tid * 8 + r] : -1.f;
            tm[r] = has ? wm[tid * 8 + r] : 0x7fffffff;
        }
        warp_top8(tv, tm, [&](int r, float v, int m) {
            fv[r] = v;
            fm[r] = m;
        });
        __syncwarp();
        float* o = feat + (size_t)c * 32;
        const bool lost = pk && (__ldcg(status) & kStatusWait);  // a window of a wait that ran out
        if (unsorted || !(T > 0.0) || M < 1 || lost) {
            o[tid] = __int_as_float(0x7fc00000);
            if (tid == 0 && !lost) atomicOr(status, kStatusNonFinite);
            return;
        }
        // lane 0 .. 5: log n, log T, log N_f, log 1/(df T), log f_max T / n, log(1 + f0 / df);
        // 6 .. 10: log gap quantile / mean gap; 11 .. 15: shares; 16 .. 23: heights; 24 .. 31: places
        const int r = tid & 7;
        const bool ok = fv[r] >= 0.f;
        double num = 1.0, den = 1.0;
        if (tid == 0) num = (double)n;
        else if (tid == 1) num = T;
        else if (tid == 2) num = (double)nf;
        else if (tid == 3) den = df * T;
        else if (tid == 4) num = f_max * T, den = (double)n;
        else if (tid == 5) num = f0, den = df;
        else if (tid <= 10) num = fmax((double)qsel[tid - 6], 1e-12 * T), den = T / (double)M;
        else if (tid <= 14) num = tid == 11 ? s2 : tid == 12 ? s10 : tid == 13 ? s100 : mx, den = T;
        else if (tid == 15) num = cnt2, den = (double)M;
        else if (tid >= 24) num = ok ? (double)(fm[r] + 1) * df : 0.0, den = f_max;
        const double x = num / den;
        o[tid] = tid == 5 ? (float)log1p(x) : tid <= 10 ? (float)log(x) : tid <= 15 || (tid >= 24 && ok) ? (float)x
                 : ok && tid < 24 ? fv[r] : 0.f;
    }
}

}  // namespace

cudaError_t launch_window(int F, int grid, const BatchItem* items, int n_items, unsigned* head, const int64_t* off,
                          const int64_t* nw, const uint4* recA, const float4* recB, float* W, const int64_t* W_off,
                          cudaStream_t st, const int* peaks) {
    switch (F) {
        case 8: ls_window_kernel<8><<<grid, kMainThreads, 0, st>>>(items, n_items, head, off, nw, recA, recB, W, W_off, peaks); break;
        case 16: ls_window_kernel<16><<<grid, kMainThreads, 0, st>>>(items, n_items, head, off, nw, recA, recB, W, W_off, peaks); break;
        case 24: ls_window_kernel<24><<<grid, kMainThreads, 0, st>>>(items, n_items, head, off, nw, recA, recB, W, W_off, peaks); break;
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// CTAs per SM of the window pass: two one-warp CTAs a sub-partition.  All that
// fit (24) would take every item of a few hundred patterns at once, in whatever
// order they start, and one SM's share of the longest ones decides; with 8, the
// ticket deals the shorter ones out as the long ones go on (256 patterns: 4, 6, 8,
// 10, 12, 16, 24 CTAs 3.51, 3.48, 3.27, 3.94, 3.60, 4.04, 4.82 ms).
constexpr int kWindowCtas = 8;

int window_occupancy(int F) {
    const void* fn = F == 8 ? (const void*)ls_window_kernel<8> : F == 16 ? (const void*)ls_window_kernel<16>
                                                                           : (const void*)ls_window_kernel<24>;
    int nb = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, kMainThreads, 0) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return nb > kWindowCtas ? kWindowCtas : nb > 0 ? nb : 1;
}

size_t features_smem_bytes(int64_t max_n) {
    const int64_t gaps = max_n - 1 <= kSortMaxGaps ? max_n - 1 : kSortMaxGaps;
    return (size_t)5 * 256 * sizeof(unsigned) + (size_t)gaps * sizeof(float);
}

cudaError_t launch_window_peaks(int n_patterns, const double* t, const int64_t* off, const double* df, const float* W,
                                const int64_t* W_off, const int64_t* nw, int* peaks, cudaStream_t st) {
    window_peaks_kernel<<<n_patterns, kFeatThreads, 0, st>>>(t, off, df, W, W_off, nw, peaks);
    return cudaGetLastError();
}

cudaError_t launch_window_exact(int F, int n_patterns, const int64_t* off, const uint4* recA, const float4* recB,
                                const int* peaks, float* peak_w, cudaStream_t st) {
    if (F != 24) return cudaErrorInvalidValue;
    dim3 grid((unsigned)n_patterns, kWindowPeaks);
    window_exact_kernel<24><<<grid, kExactThreads, 0, st>>>(off, recA, recB, peaks, peak_w);
    return cudaGetLastError();
}

cudaError_t launch_features(int n_patterns, int64_t max_n, const double* t, const int64_t* off, const double* f0,
                            const double* df, const int64_t* nf, const float* W, const int64_t* W_off,
                            const int64_t* nw, float* feat, int* status, cudaStream_t st, const int* peaks,
                            const float* peak_w) {
    const size_t smem = features_smem_bytes(max_n);
    cudaError_t e = cudaFuncSetAttribute(features_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    features_kernel<<<n_patterns, kFeatThreads, smem, st>>>(t, off, f0, df, nf, W, W_off, nw, feat, status, peaks,
                                                           peak_w);
    return cudaGetLastError();
}

}  // namespace lsp
