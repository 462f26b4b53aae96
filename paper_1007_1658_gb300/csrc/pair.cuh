// pair.cuh -- values as unevaluated sums of two FP32 numbers, about 48 bits, for
// sums, moments and centred differences that FP32 alone would round too soon.
// FP64 runs at two operations per clock and SM on this part, FP32 at 128: a pair's
// addition takes 10 of those, its product 4.
#pragma once

#include <cuda_runtime.h>

namespace lsp {
namespace dev {

struct Pair {
    float h, l;
    __device__ __forceinline__ double value() const { return (double)h + (double)l; }
};

__device__ __forceinline__ Pair pair_of(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
}

__device__ __forceinline__ Pair operator-(Pair a) { return {-a.h, -a.l}; }

// a + b; the low part takes the rounding of the high one (Knuth's exact two-sum).
// Products are formed by __fmul_rn so that none is contracted into the sum here,
// which would count its rounding twice.
__device__ __forceinline__ Pair operator+(Pair a, Pair b) {
    const float s = __fadd_rn(a.h, b.h), t = s - a.h;
    return {s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l)};
}

// The product of two FP32 values (exact), of a pair and one, and of two pairs.
__device__ __forceinline__ Pair product(float a, float b) {
    const float p = __fmul_rn(a, b);
    return {p, fmaf(a, b, -p)};
}
__device__ __forceinline__ Pair operator*(Pair a, float b) {
    const float p = __fmul_rn(a.h, b);
    return {p, fmaf(a.l, b, fmaf(a.h, b, -p))};
}
__device__ __forceinline__ Pair operator*(Pair a, Pair b) {
    const float p = __fmul_rn(a.h, b.h);
    return {p, fmaf(a.h, b.l, fmaf(a.l, b.h, fmaf(a.h, b.h, -p)))};
}

// 1 / e^2, a sample's weight from its error, in FP32 (FP64 division is slow on this
// part).  Below 2^-60 e is scaled first: its square would be subnormal and short
// of digits, the weight itself stays below 2^128 down to e = 2^-64.
__device__ __forceinline__ float error_weight(float e) {
    const bool tiny = fabsf(e) < 0x1p-60f;
    const float m = tiny ? e * 0x1p62f : e, v = 1.f / (m * m);
    return tiny ? v * 0x1p62f * 0x1p62f : v;
}

// a b to FP32.
__device__ __forceinline__ float rounded_product(Pair a, Pair b) { return fmaf(a.h, b.h, fmaf(a.h, b.l, a.l * b.h)); }

}  // namespace dev
}  // namespace lsp
