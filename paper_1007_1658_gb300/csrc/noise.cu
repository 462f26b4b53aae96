// noise.cu -- Gaussian noise for Monte-Carlo periodograms (Sec. 6.2: the
// statistics of peak heights under pure noise, e.g. the number of independent
// frequencies behind Eq. 3, are estimated from many noise periodograms).
//
// Sample j of realization r of curve c is drawn from Philox-4x32-10 (Salmon,
// Moraes, Dror & Shaw 2011) with counter (j/4, c, r, 0) and key (seed low,
// seed high): every value is a pure function of (seed, c, r, j), so runs are
// reproducible and resumable.  Each 32-bit word w becomes the uniform
// u = (2 (w >> 9) + 1) 2^-24 in (0, 1) (exact in FP32), and the Box-Muller
// transform (Box & Muller 1958) turns (u0, u1), (u2, u3) into four N(0, 1)
// values: sqrt(-2 ln u_a) (cos, sin)(2 pi u_b).
#include <cfloat>

#include "lsp_kernels.cuh"
#include "pair.cuh"
#include "philox.cuh"

namespace lsp {
namespace {

constexpr int kNoiseThreads = 256;

using dev::Pair;
using dev::pair_of;
using dev::philox4x32_10;

__device__ __forceinline__ float unit_uniform(uint32_t w) { return (float)(2u * (w >> 9) + 1u) * 0x1p-24f; }

// Four N(0,1) values of Philox block `blk` of (curve, real).
__device__ __forceinline__ float4 normals4(uint64_t seed, uint32_t blk, uint32_t curve, uint32_t real) {
    const uint4 w = philox4x32_10(blk, curve, real, 0u, (uint32_t)seed, (uint32_t)(seed >> 32));
    const float r0 = sqrtf(-2.f * logf(unit_uniform(w.x)));
    const float r1 = sqrtf(-2.f * logf(unit_uniform(w.z)));
    float s0, c0, s1, c1;
    sincospif(2.f * unit_uniform(w.y), &s0, &c0);
    sincospif(2.f * unit_uniform(w.w), &s1, &c1);
    return make_float4(r0 * c0, r0 * s0, r1 * c1, r1 * s1);
}

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ double block_sum(double v, double* sh) {
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    double r = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
    if (w == 0) r = warp_sum(r);
    if (threadIdx.x == 0) sh[32] = r;
    __syncthreads();
    return sh[32];
}

// Raw N(0,1) values of one (curve, realization), samples [0, n).
__global__ void __launch_bounds__(kNoiseThreads)
noise_raw_kernel(uint64_t seed, uint32_t curve, uint32_t real, int64_t n, float* __restrict__ out) {
    const int64_t nb = (n + 3) / 4;
    for (int64_t blk = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; blk < nb;
         blk += (int64_t)gridDim.x * blockDim.x) {
        const float4 z = normals4(seed, (uint32_t)blk, curve, real);
        const int64_t j = blk * 4;
        out[j] = z.x;
        if (j + 1 < n) out[j + 1] = z.y;
        if (j + 2 < n) out[j + 2] = z.z;
        if (j + 3 < n) out[j + 3] = z.w;
    }
}

// One CTA per (curve, realization): draw the noise into xr, then normalize it
// in place to zero mean and unit population variance (Sec. 3), over two passes.
// The threads' sums are FP32 pairs, the block's FP64.  Bound by the instructions
// of the generator; with FP64 sums and differences it was nine FP64 operations a
// sample, and a Monte Carlo of 256 patterns of 200 .. 20,000 samples by 64
// realizations took 13.94 ms, now 12.99 (with errors, by 16: 7.04 -> 6.54).
__global__ void __launch_bounds__(kNoiseThreads)
noise_prep_kernel(const int64_t* __restrict__ off, const uint64_t* __restrict__ seed_p, int64_t total,
                  float* __restrict__ xr, float4* __restrict__ recB) {
    __shared__ double sh[33];
    const int c = blockIdx.x, r = blockIdx.y;
    const int64_t b = off[c], n = off[c + 1] - off[c];
    float* x = xr + (size_t)r * (size_t)total + b;
    const uint64_t seed = *seed_p;
    Pair s = {0.f, 0.f};
    for (int64_t blk = threadIdx.x; blk * 4 < n; blk += blockDim.x) {
        const float4 z = normals4(seed, (uint32_t)blk, (uint32_t)c, (uint32_t)r);
        const int64_t j = blk * 4;
        const float zz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (j + u < n) {
                x[j + u] = zz[u];
                s = s + Pair{zz[u], 0.f};
            }
    }
    __syncthreads();
    const Pair minus_mean = pair_of(-(block_sum(s.value(), sh) / (double)n));
    Pair v = {0.f, 0.f};
#pragma unroll 4
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        const Pair d = Pair{x[j], 0.f} + minus_mean;
        v = v + d * d;
    }
    const double var = block_sum(v.value(), sh) / (double)n;
    const Pair inv_sd = pair_of(var > 0.0 ? 1.0 / sqrt(var) : 0.0);
#pragma unroll 4
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        const float xh = rounded_product(Pair{x[j], 0.f} + minus_mean, inv_sd);
        x[j] = xh;
        if (recB) recB[b + j].x = xh;  // single realization: straight into the sample records
    }
}

// One CTA per curve and RR realizations of the floating-mean Monte Carlo: the
// same N(0,1) draws z_j as noise_prep_kernel, X_j = dy_j z_j (z_j without dy),
// then the weighted normalization of prep_records_kernel's floating-mean form,
// x_j = q_j (X_j - mean_w) / sd_w, with v_j = 1/dy_j^2 formed in FP32 as the
// prep kernels form it, mean_w = sum v X / sum v and the population variance
// sum v (X - mean_w)^2 / sum v, the threads' sums FP32 pairs but for sum v: errors
// around 1e-19 (fluxes in cgs units) have weights of 1e38, which only FP64 can add
// up; every other sum is of the size of dy, of 1/dy or of 1.  X_j is re-formed
// from the stored z_j in every pass.  The four FP64 operations that split dy_j and
// the one that adds v_j serve the RR realizations.
template <int RR>
__global__ void __launch_bounds__(kNoiseThreads)
gls_noise_prep_kernel(const int64_t* __restrict__ off, uint64_t seed, int64_t total, int n_real,
                      const double* __restrict__ dy, const float* __restrict__ q, float* __restrict__ xr) {
    __shared__ double sh[33];
    const int c = blockIdx.x, r0 = blockIdx.y * RR, nr = min(RR, n_real - r0);
    const int64_t b = off[c], n = off[c + 1] - off[c];
    float* const x = xr + (size_t)r0 * (size_t)total + b;
    // dy_j and v_j
    auto error = [&](int64_t j, Pair& e, float& v) {
        e = dy ? pair_of(dy[b + j]) : Pair{1.f, 0.f};
        v = dy ? dev::error_weight(e.h) : 1.f;
    };
    double sv = 0.0;
    Pair acc[RR], minus_mean[RR], inv_sd[RR];
#pragma unroll
    for (int i = 0; i < RR; ++i) acc[i] = {0.f, 0.f};
    for (int64_t blk = threadIdx.x; blk * 4 < n; blk += blockDim.x) {
        const int64_t j = blk * 4;
        Pair e[4];
        float v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (j + u >= n) break;
            error(j + u, e[u], v[u]);
            sv += (double)v[u];
        }
#pragma unroll
        for (int i = 0; i < RR; ++i) {
            if (i >= nr) break;
            const float4 z = normals4(seed, (uint32_t)blk, (uint32_t)c, (uint32_t)(r0 + i));
            const float zz[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (j + u >= n) break;
                x[(size_t)i * (size_t)total + j + u] = zz[u];
                acc[i] = acc[i] + e[u] * zz[u] * v[u];
            }
        }
    }
    __syncthreads();
    const double svd = block_sum(sv, sh);
#pragma unroll
    for (int i = 0; i < RR; ++i) {
        minus_mean[i] = pair_of(-(block_sum(acc[i].value(), sh) / svd));
        acc[i] = {0.f, 0.f};
    }
#pragma unroll 2
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        Pair e;
        float v;
        error(j, e, v);
#pragma unroll
        for (int i = 0; i < RR; ++i)
            if (i < nr) {
                const Pair d = e * x[(size_t)i * (size_t)total + j] + minus_mean[i];
                acc[i] = acc[i] + d * v * d;
            }
    }
#pragma unroll
    for (int i = 0; i < RR; ++i) {
        const double var = block_sum(acc[i].value(), sh) / svd;
        inv_sd[i] = pair_of(var > 0.0 ? 1.0 / sqrt(var) : 0.0);
    }
#pragma unroll 2
    for (int64_t j = threadIdx.x; j < n; j += blockDim.x) {
        Pair e;
        float v;
        error(j, e, v);
        const float qj = q[b + j];
#pragma unroll
        for (int i = 0; i < RR; ++i)
            if (i < nr) {
                float& xj = x[(size_t)i * (size_t)total + j];
                xj = rounded_product(e * xj + minus_mean[i], inv_sd[i]) * qj;
            }
    }
}

}  // namespace

cudaError_t launch_gls_noise_prep(const int64_t* off, int n_curves, int n_real, uint64_t seed, int64_t total,
                                  const double* dy, const float* q, float* xr, cudaStream_t st) {
    // four realizations a CTA where that leaves two CTAs an SM and more
    constexpr int RR = 4;
    if ((int64_t)n_curves * (n_real / RR) >= 2 * 152)
        gls_noise_prep_kernel<RR><<<dim3((unsigned)n_curves, (unsigned)((n_real + RR - 1) / RR)), kNoiseThreads, 0, st>>>(
            off, seed, total, n_real, dy, q, xr);
    else
        gls_noise_prep_kernel<1><<<dim3((unsigned)n_curves, (unsigned)n_real), kNoiseThreads, 0, st>>>(
            off, seed, total, n_real, dy, q, xr);
    return cudaGetLastError();
}

cudaError_t launch_noise_raw(uint64_t seed, uint32_t curve, uint32_t real, int64_t n, float* out, cudaStream_t st) {
    const int64_t nb = (n + 3) / 4;
    int64_t blocks = (nb + kNoiseThreads - 1) / kNoiseThreads;
    if (blocks > 4096) blocks = 4096;
    if (blocks < 1) blocks = 1;
    noise_raw_kernel<<<(unsigned)blocks, kNoiseThreads, 0, st>>>(seed, curve, real, n, out);
    return cudaGetLastError();
}

cudaError_t launch_noise_prep(const int64_t* off, int n_curves, int n_real, const uint64_t* seed_dev,
                              int64_t total, float* xr, float4* recB, cudaStream_t st) {
    dim3 grid((unsigned)n_curves, (unsigned)n_real);
    noise_prep_kernel<<<grid, kNoiseThreads, 0, st>>>(off, seed_dev, total, xr, n_real == 1 ? recB : nullptr);
    return cudaGetLastError();
}

}  // namespace lsp
