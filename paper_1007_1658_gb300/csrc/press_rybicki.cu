// press_rybicki.cu -- the fast approximate periodogram of Press & Rybicki
// (1989), the O(N log N) alternative the paper's introduction cites: the data
// are "extirpolated" onto a uniform periodic grid and one FFT gives the sums
// of Eq. 5-8 at every grid frequency.
//
// Grid: n_fft nodes (a power of two) spanning one period 1/df, so FFT bin K
// is the frequency K df.  Sample j sits at g = frac(t'_j df) n_fft for the
// sums over x and at g2 = frac(2 t'_j df) n_fft for the sums over the doubled
// angle; each is spread onto the macc nodes around it with the Lagrange
// weights that would interpolate a function from those nodes to g.  The two
// real grids travel as one complex array z = grid_x + i grid_1; one FFT with
// the e^{+2 pi i K m / n} sign gives Z, and the transforms of the two real
// grids are (Z[K] + conj Z[n-K]) / 2 and (Z[K] - conj Z[n-K]) / 2i.  With
// XC + i XS = sum x e^{i w t'} and CC - SS + 2i CS = sum e^{2 i w t'}, Eq. 5-6
// follow in the closed form of periodogram_value.
//
// Kernels: spread (FP64 positions, FP32 Lagrange weights, FP64 atomics into a
// double2 grid), then Stockham passes of radix 16 to 256, each through shared
// memory; the first reads the FP64 grid and rounds it to FP32, and the last forms
// the periodogram of the requested bins from its own outputs and writes nothing
// else.  A pass moves the grid once each way and is bound by that, so the radix is
// as large as shared memory holds 16 adjacent columns (whole 128-byte lines) of
// with several CTAs an SM.  2^24 nodes (382,003 samples, 1,528,064 bins): three
// passes of 69, 50 and 54 us, 5.8 and 5.1 TB/s for the first two, where six
// radix-16 passes through global memory and a separate finalize took the call
// 475 us; now 281, with the grid's memset and the spread's atomics 70 of it.
#include <type_traits>
#include <utility>

#include "ls_device.cuh"

namespace lsp {
namespace {

constexpr int kPrThreads = 256;

constexpr int kMaxMacc = 16;

// Lagrange weights of the macc nodes lo .. lo+macc-1 for a position d = g - lo
// in [macc/2 - 1, macc/2): w_i = prod_{l != i} (d - l) / prod_{l != i} (i - l),
// numerators from prefix and suffix products, denominators 1 / (i! (macc-1-i)!)
// with the sign (-1)^(macc-1-i).  FP32 (d is small; the FFT is FP32 too).  MACC: macc
// where it is known when compiling, which keeps w in registers; else 0.
template <int MACC>
__device__ __forceinline__ void lagrange_weights(float d, int macc_, float* w) {
    const int macc = MACC ? MACC : macc_;
    float pre = 1.f;
#pragma unroll
    for (int i = 0; i < macc; ++i) {
        w[i] = pre;
        pre *= d - (float)i;
    }
    float suf = 1.f;
#pragma unroll
    for (int i = macc - 1; i >= 0; --i) {
        float den = 1.f;
#pragma unroll
        for (int l = 0; l < macc; ++l)
            if (l != i) den *= (float)(i - l);
        w[i] *= suf / den;
        suf *= d - (float)i;
    }
}

template <int MACC>
__global__ void __launch_bounds__(kPrThreads)
pr_spread_kernel(const double* __restrict__ t, const double* __restrict__ X, int64_t n,
                 const CurveStats* __restrict__ stats, double df, int64_t n_fft, int macc_,
                 double2* __restrict__ acc) {
    const int macc = MACC ? MACC : macc_;
    const CurveStats st = stats[0];
    const double nd = (double)n_fft;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const double tt = t[j] - st.t_ref;
        const double x = (X[j] - st.mean) * st.inv_sd;
#pragma unroll 1
        for (int which = 0; which < 2; ++which) {
            // position in FP64 (node choice exact), offset from the first node in FP32
            const double p = (which ? 2.0 * tt : tt) * df;
            const double g = (p - floor(p)) * nd;
            const int64_t lo = (int64_t)floor(g) - (macc / 2 - 1);
            float w[MACC ? MACC : kMaxMacc];
            lagrange_weights<MACC>((float)(g - (double)lo), macc, w);
#pragma unroll
            for (int i = 0; i < macc; ++i) {
                const int64_t m = (lo + i) & (n_fft - 1);  // periodic grid, n_fft a power of two
                if (which == 0)
                    atomicAdd(&acc[m].x, (double)w[i] * x);
                else
                    atomicAdd(&acc[m].y, (double)w[i]);
            }
        }
    }
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// e^{+2 pi i f / 2^bits} for integer f (reduced exactly to half a turn either way
// first, so the FP32 argument of sincospif is small).
__device__ __forceinline__ float2 twiddle(uint32_t f, int bits) {
    const int g = (int)(f << (32 - bits)) >> (32 - bits);
    float s, c;
    sincospif((float)g * __int_as_float((128 - bits) << 23), &s, &c);  // 2 g / 2^bits
    return make_float2(c, s);
}

template <class T>
__device__ __forceinline__ float2 load_c(const T* p, int64_t i);
template <>
__device__ __forceinline__ float2 load_c<float2>(const float2* p, int64_t i) {
    return p[i];
}
template <>
__device__ __forceinline__ float2 load_c<double2>(const double2* p, int64_t i) {
    const double2 v = p[i];
    return make_float2((float)v.x, (float)v.y);
}

// In-place 4-point DFT with the e^{+2 pi i / 4} = i kernel.
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3) {
    const float2 a0 = make_float2(x0.x + x2.x, x0.y + x2.y);
    const float2 a1 = make_float2(x0.x - x2.x, x0.y - x2.y);
    const float2 a2 = make_float2(x1.x + x3.x, x1.y + x3.y);
    const float2 a3 = make_float2(-(x1.y - x3.y), x1.x - x3.x);
    x0 = make_float2(a0.x + a2.x, a0.y + a2.y);
    x1 = make_float2(a1.x + a3.x, a1.y + a3.y);
    x2 = make_float2(a0.x - a2.x, a0.y - a2.y);
    x3 = make_float2(a1.x - a3.x, a1.y - a3.y);
}

// In-place N-point DFT of v[0], v[1], ..., natural order in and out.  16 = 4 x 4:
// with q = 4a + b and k = c + 4d, X[c + 4d] = sum_b i^{bd} w^{bc} sum_a
// v[4a + b] i^{ac}, w = e^{+2 pi i / 16}; 8 = 2 x 4 likewise.
template <int N>
__device__ __forceinline__ void dft(float2 (&v)[N]) {
    constexpr float c1 = 0.92387953251128674f, s1 = 0.38268343236508978f, h = 0.70710678118654752f;
    if constexpr (N == 4) {
        dft4(v[0], v[1], v[2], v[3]);
    } else if constexpr (N == 8) {
        float2 y[8];
#pragma unroll
        for (int b = 0; b < 4; ++b) {  // y[4c + b]
            y[b] = make_float2(v[b].x + v[4 + b].x, v[b].y + v[4 + b].y);
            y[4 + b] = make_float2(v[b].x - v[4 + b].x, v[b].y - v[4 + b].y);
        }
        y[5] = cmul(y[5], make_float2(h, h));
        y[6] = make_float2(-y[6].y, y[6].x);
        y[7] = cmul(y[7], make_float2(-h, h));
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            dft4(y[4 * c], y[4 * c + 1], y[4 * c + 2], y[4 * c + 3]);
#pragma unroll
            for (int d = 0; d < 4; ++d) v[c + 2 * d] = y[4 * c + d];
        }
    } else {
        static_assert(N == 16, "");
#pragma unroll
        for (int b = 0; b < 4; ++b) dft4(v[b], v[4 + b], v[8 + b], v[12 + b]);  // v[4c + b] = Y_b[c]
        // inner twiddles w^{bc}
        v[5] = cmul(v[5], make_float2(c1, s1));    // b = 1, c = 1
        v[6] = cmul(v[6], make_float2(h, h));      // b = 2, c = 1
        v[7] = cmul(v[7], make_float2(s1, c1));    // b = 3, c = 1
        v[9] = cmul(v[9], make_float2(h, h));      // b = 1, c = 2
        v[10] = make_float2(-v[10].y, v[10].x);    // b = 2, c = 2: w^4 = i
        v[11] = cmul(v[11], make_float2(-h, h));   // b = 3, c = 2
        v[13] = cmul(v[13], make_float2(s1, c1));  // b = 1, c = 3
        v[14] = cmul(v[14], make_float2(-h, h));   // b = 2, c = 3
        v[15] = cmul(v[15], make_float2(-c1, -s1));  // b = 3, c = 3: w^9
        float2 x[16];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            dft4(v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
#pragma unroll
            for (int d = 0; d < 4; ++d) x[c + 4 * d] = v[4 * c + d];
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) v[k] = x[k];
    }
}

// P of bin K from Z[K] = a and Z[n_fft - K] = b: the transform of the x grid is
// (a + conj b) / 2, of the unit grid (a - conj b) / 2i.
__device__ __forceinline__ float pr_value(float2 a, float2 b, float n) {
    const float XC = 0.5f * (a.x + b.x), XS = 0.5f * (a.y - b.y);
    const float A2 = 0.5f * (a.y + b.y), B2 = -0.5f * (a.x - b.x);
    return dev::periodogram_value(XC, XS, 0.5f * (n + A2), 0.5f * B2, n);
}

// A pass takes sub-transforms of length Ns to length R Ns, R = 2^LR: column j of
// n / R reads in[j + q n / R], q < R, twiddles by e^{+2 pi i r q / (R Ns)} with
// r = j mod Ns, and its R-point DFT goes to out[(j - r) R + r + k Ns].  R = A B,
// q = a B + b, k = c + A d: thread b of a column sums over a, thread c then over
// b, with shared memory between.  A CTA holds kCols adjacent columns, 128 bytes
// of a row of FP32 nodes, and kLanes threads for each.
constexpr int kCols = 16, kLanes = 16;
static_assert(kCols * kLanes == kPrThreads, "");
constexpr int kMinBits = 4, kMaxBits = 8;

template <int LR>
struct Radix {
    static constexpr int A = 1 << (LR / 2), B = 1 << (LR - LR / 2), R = A * B;
    float2 tile[kCols * (R + 1)];  // [c B + b][column]; the first pass's outputs as [column][R + 1]
    float2 ta[A * kCols];          // e^{+2 pi i r a B / (R Ns)}

    // This thread's B outputs k = c + A d of column j, in v[d]; c = lane, or
    // A - 1 - lane for the mirrored columns of the last pass.  Nothing where lane >= A.
    // The twiddles of b, e^{+2 pi i b (r + c Ns) / (R Ns)}, are each formed for its
    // one use: as products of two tables they cost a rounding more.
    template <class T>
    __device__ __forceinline__ void run(const T* in, int64_t m, int64_t j, int lNs, bool mirrored, float2 (&v)[B]) {
        const int col = threadIdx.x % kCols, lane = threadIdx.x / kCols;
        const uint32_t r = (uint32_t)j & ((1u << lNs) - 1u);
        float2 u[A];
        if (lane < B) {
#pragma unroll
            for (int a = 0; a < A; ++a) u[a] = load_c(in, j + (int64_t)(a * B + lane) * m);
        }
        if (lNs && lane < A) ta[lane * kCols + col] = twiddle(r * (uint32_t)(lane * B), LR + lNs);
        __syncthreads();  // the table; the tile's last readers
        if (lane < B) {
            if (lNs) {
#pragma unroll
                for (int a = 1; a < A; ++a) u[a] = cmul(u[a], ta[a * kCols + col]);
            }
            dft(u);
#pragma unroll
            for (int c = 0; c < A; ++c)
                tile[(c * B + lane) * kCols + col] =
                    cmul(u[c], twiddle((r + ((uint32_t)c << lNs)) * (uint32_t)lane, LR + lNs));
        }
        __syncthreads();
        if (lane < A) {
            const int c = mirrored ? A - 1 - lane : lane;
#pragma unroll
            for (int b = 0; b < B; ++b) v[b] = tile[(c * B + b) * kCols + col];
            dft(v);
        }
    }
};

template <int LR, class T>
__global__ void __launch_bounds__(kPrThreads)
fft_pass(const T* __restrict__ in, float2* __restrict__ out, int64_t n, int lNs) {
    using S = Radix<LR>;
    __shared__ S s;
    const int col = threadIdx.x % kCols, lane = threadIdx.x / kCols;
    const int64_t m = n / S::R, j0 = (int64_t)blockIdx.x * kCols, j = j0 + col;
    float2 v[S::B];
    s.run(in, m, j, lNs, false, v);
    if (lNs) {
        const int64_t Ns = int64_t(1) << lNs;
        const int64_t r = j & (Ns - 1), d0 = (j - r) * S::R + r;
        if (lane < S::A)
#pragma unroll
            for (int d = 0; d < S::B; ++d) out[d0 + (lane + S::A * d) * Ns] = v[d];
        return;
    }
    // Ns = 1: a column's outputs are adjacent; through shared memory to whole lines
    __syncthreads();
    if (lane < S::A)
#pragma unroll
        for (int d = 0; d < S::B; ++d) s.tile[col * (S::R + 1) + lane + S::A * d] = v[d];
    __syncthreads();
    for (int i = threadIdx.x; i < kCols * S::R; i += kPrThreads)
        out[j0 * S::R + i] = s.tile[i / S::R * (S::R + 1) + i % S::R];
}

// The last pass (R Ns = n) and P.  Bin K = r + k Ns pairs with n - K, which is
// output R - 1 - k of column Ns - r: a CTA takes columns r <= Ns / 2 and their
// mirror images, and a thread both outputs of a pair.  Column 0 is its own image
// with output (R - k) mod R.  Bins are below n / 4 (the grid is oversampled by
// 2 macc >= 4).
template <int LR>
__global__ void __launch_bounds__(kPrThreads, 3)
fft_last_pass(const float2* __restrict__ in, int lNs, int64_t j0, int64_t N_f, float samples,
              float* __restrict__ P_out) {
    using S = Radix<LR>;
    constexpr int A = S::A, B = S::B, R = S::R;
    __shared__ S s;
    __shared__ float2 zero[R];  // column 0
    const int col = threadIdx.x % kCols, lane = threadIdx.x / kCols;
    const int64_t Ns = int64_t(1) << lNs, r = (int64_t)blockIdx.x * kCols + col;
    const int64_t c1 = r < Ns / 2 ? r : Ns / 2;
    float2 v[B], u[B];
    s.run(in, Ns, c1, lNs, false, v);
    s.run(in, Ns, (Ns - c1) & (Ns - 1), lNs, true, u);
    if (blockIdx.x == 0) {
        if (r == 0 && lane < A)
#pragma unroll
            for (int d = 0; d < B; ++d) zero[lane + A * d] = v[d];
        __syncthreads();
    }
    if (lane >= A || r > Ns / 2) return;
#pragma unroll
    for (int d = 0; d < B / 4; ++d) {
        const int k = lane + A * d;
        const int64_t at = r + k * Ns - j0;
        if (at >= 0 && at < N_f) P_out[at] = pr_value(v[d], r ? u[B - 1 - d] : zero[(R - k) & (R - 1)], samples);
        // the mirrored column's bin A - 1 - lane + A d, with output lane + A (B - 1 - d) here
        const int64_t at2 = Ns - r + (A - 1 - lane + A * d) * Ns - j0;
        if (r > 0 && r < Ns / 2 && at2 >= 0 && at2 < N_f) P_out[at2] = pr_value(u[d], v[B - 1 - d], samples);
    }
}

// Grids too small for two passes: a warp a bin, by the definition.
__global__ void __launch_bounds__(kPrThreads)
pr_direct_kernel(const double2* __restrict__ acc, int bits, int64_t j0, int64_t N_f, float n,
                 float* __restrict__ P_out) {
    const int lane = threadIdx.x & 31;
    const int64_t k = (int64_t)blockIdx.x * (kPrThreads / 32) + (threadIdx.x >> 5), K = j0 + k;
    if (k >= N_f) return;
    float2 a = make_float2(0.f, 0.f), b = a;  // Z[K], Z[n - K]
    for (int64_t m = lane; m < int64_t(1) << bits; m += 32) {
        const float2 z = load_c(acc, m), w = twiddle((uint32_t)(K * m), bits);
        const float2 p = cmul(z, w), q = cmul(z, make_float2(w.x, -w.y));
        a = make_float2(a.x + p.x, a.y + p.y);
        b = make_float2(b.x + q.x, b.y + q.y);
    }
    for (int o = 16; o; o >>= 1) {
        a.x += __shfl_xor_sync(0xffffffffu, a.x, o);
        a.y += __shfl_xor_sync(0xffffffffu, a.y, o);
        b.x += __shfl_xor_sync(0xffffffffu, b.x, o);
        b.y += __shfl_xor_sync(0xffffffffu, b.y, o);
    }
    if (lane == 0) P_out[k] = pr_value(a, b, n);
}

// f(std::integral_constant<int, bits>{})
template <class F>
void with_bits(int bits, F&& f) {
    switch (bits) {
        case 4: f(std::integral_constant<int, 4>{}); break;
        case 5: f(std::integral_constant<int, 5>{}); break;
        case 6: f(std::integral_constant<int, 6>{}); break;
        case 7: f(std::integral_constant<int, 7>{}); break;
        default: f(std::integral_constant<int, 8>{}); break;
    }
}

unsigned blocks_for(int64_t work) {
    int64_t b = (work + kPrThreads - 1) / kPrThreads;
    if (b > 152 * 64) b = 152 * 64;
    return (unsigned)(b < 1 ? 1 : b);
}

}  // namespace

int64_t pr_fft_size(int64_t k_hi, int macc) {
    const int64_t need = 2 * (int64_t)macc * (k_hi + 1);
    int64_t n = 1;
    while (n < need) n <<= 1;
    return n;
}

cudaError_t launch_pr(const double* t, const double* X, int64_t N, const CurveStats* stats, double df, int64_t j0,
                      int64_t N_f, int macc, int64_t n_fft, double2* acc, float2* z0, float2* z1, float* P_out,
                      int* launches, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(acc, 0, (size_t)n_fft * sizeof(double2), st);
    if (e != cudaSuccess) return e;
    if (macc == 4) pr_spread_kernel<4><<<blocks_for(N), kPrThreads, 0, st>>>(t, X, N, stats, df, n_fft, macc, acc);
    else pr_spread_kernel<0><<<blocks_for(N), kPrThreads, 0, st>>>(t, X, N, stats, df, n_fft, macc, acc);
    int L = 0;
    while ((int64_t(1) << L) < n_fft) ++L;
    int nl = 2;
    if (L < 2 * kMinBits + 1) {
        constexpr int kWarps = kPrThreads / 32;
        pr_direct_kernel<<<(unsigned)((N_f + kWarps - 1) / kWarps), kPrThreads, 0, st>>>(acc, L, j0, N_f, (float)N,
                                                                                         P_out);
    } else {
        // the bits spread evenly over as few passes as hold them, the fewer first
        // (the first pass's nodes are twice as wide)
        const int passes = (L + kMaxBits - 1) / kMaxBits;
        int lNs = 0;
        float2 *cur = z0, *nxt = z1;
        for (int p = 0; p < passes; ++p, ++nl) {
            const int bits = (L + p) / passes;
            with_bits(bits, [&](auto lr) {
                constexpr int LR = decltype(lr)::value;
                const unsigned grid = (unsigned)((n_fft >> LR) / kCols);
                if (p == 0)
                    fft_pass<LR><<<grid, kPrThreads, 0, st>>>(acc, cur, n_fft, lNs);
                else if (p < passes - 1)
                    fft_pass<LR><<<grid, kPrThreads, 0, st>>>((const float2*)cur, nxt, n_fft, lNs);
                else if constexpr (LR > kMinBits)
                    fft_last_pass<LR><<<grid / 2 + 1, kPrThreads, 0, st>>>(cur, lNs, j0, N_f, (float)N, P_out);
            });
            if (p) std::swap(cur, nxt);
            lNs += bits;
        }
        --nl;
    }
    if (launches) *launches = nl;
    return cudaGetLastError();
}

}  // namespace lsp
