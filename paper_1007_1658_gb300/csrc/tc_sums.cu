// tc_sums.cu -- the periodogram's sums on the tensor cores.
//
// Every frequency of a uniform grid is a coarse frequency plus or minus a fine
// offset, f = f_a +- f_b, and exp(2 pi i f t) = exp(2 pi i f_a t)
// exp(+- 2 pi i f_b t): the sums of Eq. 8 over the samples j,
//     sum_j y_j e^{2 pi i f_a t_j} cos 2 pi f_b t_j,  ... sin 2 pi f_b t_j,
// are a real matrix product A^T B with A[j][2a, 2a+1] = y_j (cos, sin)(2 pi f_a
// t_j) and B[j][2b, 2b+1] = (cos, sin)(2 pi f_b t_j); its four entries for
// (a, b) give the complex sums at f_a + f_b and f_a - f_b, so a term still
// costs two multiply-adds per sum, and the operands cost 128 + cols/2 complex
// values per sample for 128 cols terms.  With y = x_hat this is XC + i XS; the
// tau sums CC - SS + 2i CS are the same product with y = 1 at doubled phases.
// Phases are the exact 64-bit fixed-point turns of the strip kernels.
//
// FP32 accuracy from FP16 operands: a value v is split into hi = fp16(v) and
// lo = fp16(v - hi) (22 bits, error at most 2^-24 for |v| <= 1), and the
// product runs as hi hi + hi lo + lo hi, each exact, accumulated in FP32 by
// the tensor core.  That accumulation truncates: every product is cut at a
// quarter ulp of the accumulator and every step rounds toward zero, which
// shrinks a coherent sum by ~1.5e-7 per 64 samples.  So an accumulator takes
// only kTcUnit samples; then its values are added in FP32 (round to nearest)
// to running sums in registers while the next unit accumulates in the other
// half of tensor memory.
//
// The product runs on CTA pairs (256 x cols x 16 an instruction): a CTA makes and
// holds half of the rows of A and half of the columns of B, so its operands per
// term are two thirds of a single CTA's, in the making and in shared memory.
//
// What bounds it: with cols = 256 the three MMAs of 16 samples take 390 cycles (24
// a sample for 32,768 terms), the operands 128 complex values a sample and CTA.  A
// unit of 128 samples takes a pair 3750 cycles, its MMAs alone 3120.  100,000
// samples by 200,000 frequencies: this kernel 285 us, the FP32 strips 3605.
#include "ls_device.cuh"
#include "pair.cuh"
#include "tc_device.cuh"
#include "tc_sums.cuh"

#include <cooperative_groups.h>
#include <cuda_fp16.h>

namespace lsp {
namespace {

constexpr int kStage = 32;                        // samples of one operand stage
constexpr int kSets = kTcUnit / kStage;           // sets of warps, each filling every kSets-th stage
constexpr int kBufs = 6;                          // stage buffers
constexpr int kAbytes = 128 * kStage * 2;         // one half (hi or lo) of A: 128 rows
constexpr int kBbytes = kTcMaxCols / 2 * kStage * 2;  // one half of a CTA's columns of B
constexpr int kStageBytes = 2 * kAbytes + 2 * kBbytes;
constexpr int kSbo = kStage * 16;                 // bytes of one 8-row group of an operand
constexpr int kGenWarps = 16;
constexpr int kSetWarps = kGenWarps / kSets;
constexpr size_t kSmem = kBufs * (size_t)kStageBytes + sizeof(float) * 12 * kGenWarps * 32;

// (cos, sin) of a 64-bit fixed-point turn: quadrant and 30-bit remainder of the
// top word, then the Taylor series on [-pi/4, pi/4] (truncation below 2e-9).
__device__ __forceinline__ float2 turn_cos_sin(uint64_t ph) {
    const uint32_t top = (uint32_t)(ph >> 32);
    const uint32_t qd = (top + 0x20000000u) >> 30;
    const float x = (float)(int32_t)(top - (qd << 30)) * 1.4629180792671596e-9f;  // 2 pi / 2^32
    const float w = x * x;
    float s = fmaf(w, 2.7557319223985893e-6f, -1.9841269841269841e-4f);
    s = fmaf(w, s, 8.3333333333333333e-3f);
    s = fmaf(w, s, -1.6666666666666667e-1f);
    s = fmaf(x * w, s, x);
    float c = fmaf(w, -2.7557319223985888e-7f, 2.4801587301587302e-5f);
    c = fmaf(w, c, -1.3888888888888889e-3f);
    c = fmaf(w, c, 4.1666666666666664e-2f);
    c = fmaf(w, c, -0.5f);
    c = fmaf(w, c, 1.f);
    const float cc = (qd & 1) ? s : c, ss = (qd & 1) ? c : s;
    return make_float2(__uint_as_float(__float_as_uint(cc) ^ (((qd + 1) & 2) << 30)),
                       __uint_as_float(__float_as_uint(ss) ^ ((qd & 2) << 30)));
}

// A rotation and its products, scalar.
__device__ __forceinline__ float2 cmul(float2 z, float2 e) {
    return make_float2(fmaf(-z.y, e.y, z.x * e.x), fmaf(z.y, e.x, z.x * e.y));
}
__device__ __forceinline__ float2 csquare(float2 e) {
    return make_float2(fmaf(-e.y, e.y, e.x * e.x), (e.x + e.x) * e.y);
}

// Two neighbouring complex values in the lanes of packed FP32: a product with
// one rotation is four packed operations, and (re, re') and (im, im') are the
// pairs that an FP16 word of an operand row holds.
struct Pair {
    float2 re, im;
};
__device__ __forceinline__ Pair mul_pair(const Pair& z, float2 e) {
    const float2 c = make_float2(e.x, e.x), s = make_float2(e.y, e.y), n = make_float2(-e.y, -e.y);
    Pair r;
    r.re = __ffma2_rn(z.im, n, __fmul2_rn(z.re, c));
    r.im = __ffma2_rn(z.im, c, __fmul2_rn(z.re, s));
    return r;
}

// Eight consecutive values of an operand row group, split into their FP16
// halves, 16 bytes each.
__device__ __forceinline__ void split_pair(float2 v, uint32_t& hi, uint32_t& lo) {
    const __half2 a = __floats2half2_rn(v.x, v.y);
    float2 d;  // v - a, exact, by FP32 additions that take an FP16 operand
    asm("{\n .reg .b16 p, q, m;\n mov.b32 {p, q}, %4;\n mov.b16 m, 0xBC00;\n"
        " fma.rn.f32.f16 %0, p, m, %2;\n fma.rn.f32.f16 %1, q, m, %3;\n}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(v.x), "f"(v.y), "r"(*reinterpret_cast<const uint32_t*>(&a)));
    const __half2 b = __floats2half2_rn(d.x, d.y);
    hi = *reinterpret_cast<const uint32_t*>(&a);
    lo = *reinterpret_cast<const uint32_t*>(&b);
}

__device__ __forceinline__ void store_group(const Pair (&z)[4], unsigned char* re_hi, unsigned char* re_lo,
                                            unsigned char* im_hi, unsigned char* im_lo) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) split_pair(z[i].re, h[i], l[i]);
    *reinterpret_cast<uint4*>(re_hi) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(re_lo) = make_uint4(l[0], l[1], l[2], l[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) split_pair(z[i].im, h[i], l[i]);
    *reinterpret_cast<uint4*>(im_hi) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4*>(im_lo) = make_uint4(l[0], l[1], l[2], l[3]);
}

// z, z e, ... z e^7 from e, e^2, e^4.
__device__ __forceinline__ void powers8(float2 z, float2 e, float2 e2, float2 e4, Pair (&p)[4]) {
    const float2 z1 = cmul(z, e);
    p[0].re = make_float2(z.x, z1.x);
    p[0].im = make_float2(z.y, z1.y);
    p[1] = mul_pair(p[0], e2);
    p[2] = mul_pair(p[0], e4);
    p[3] = mul_pair(p[1], e4);
}

// Records of every thread's next sample, filled with cp.async a stage ahead: a
// thread reads what it copied itself, so no barrier is needed.
struct Ahead {
    uint4 uv[kGenWarps * 32];
    float4 B[kGenWarps * 32];
    float2 E[kGenWarps * 32];
    float q[kGenWarps * 32], x[kGenWarps * 32];
};

// The tile of a launch, and the samples of its curve.
struct TileInfo {
    TcTile w;
    int64_t b, n;
};

__device__ __forceinline__ TcTile tile_of(const TcArgs& a, int t) {
    if (a.tiles) return a.tiles[t];
    TcTile w = a.one;
    if (t < a.h1) {
        w.g0 = kTcGroups * t;
    } else {
        w.g0 = kTcGroups * (t - a.h1);
        w.kind = a.win_kind;
        w.twice = 1;
    }
    return w;
}

__device__ __forceinline__ TileInfo tile_info(const TcArgs& a, int t) {
    TileInfo f;
    f.w = tile_of(a, t);
    f.b = a.off ? a.off[f.w.curve] : 0;
    f.n = a.off ? a.off[f.w.curve + 1] - f.b : a.n0;
    return f;
}

// A group of a tile: what its rows sum (y = 0 beyond the last set), the grid's
// group, the realization, and the power of two on y that keeps the bits of its
// FP16 halves.
struct Group {
    int kind, kg, real;
    bool live;
    float scale;
};

__device__ __forceinline__ Group group_of(const TcArgs& a, const TileInfo& f, int g) {
    Group r;
    const int G = f.w.g0 + g, set = G / f.w.gpr;
    r.kg = f.w.kg0 + (G - set * f.w.gpr);
    r.kind = f.w.kind;
    r.real = f.w.r0 + set;
    if (f.w.twice) {
        r.live = set == 0;
    } else {
        r.live = set < f.w.reals + f.w.gls;
        if (f.w.gls && set >= f.w.reals) r.kind = kTcW1;
    }
    // |x_hat| <= sqrt(n); |q x_hat| <= qmax; q^2 <= qmax^2: scaled to at most 2^14
    int ex = 0;
    if (r.kind == kTcRec || r.kind == kTcRow) {
        ex = 14 - (33 - __clz((int)min(f.n, (int64_t)0x7fffffff))) / 2;
    } else if (r.kind >= kTcW1 && a.qmax) {
        int eq;
        frexpf(a.qmax[f.w.curve], &eq);  // qmax < 2^eq
        ex = 14 - (r.kind >= kTcRecQ ? eq : 2 * eq);
    }
    r.scale = ldexpf(1.f, min(max(ex, -100), 100));
    return r;
}

// The factor that undoes the mean shrinking of a unit's accumulation (see
// above): 1 + 4 ulp.  How much a sum shrinks depends on where its growth lies
// between two powers of two, by a third either way; so four units in turn are
// scaled by (about) 1, 2^1/4, 2^1/2, 2^3/4, which makes the mean the same for every
// sum.  The scales are FP32 values whose product with their gains is 1 + 4 ulp to
// 2e-9.
__device__ __forceinline__ float unit_scale(int u) {
    return u & 2 ? (u & 1 ? 0x1.ae7ee8p+0f : 0x1.6a09ecp+0f) : (u & 1 ? 0x1.30840ep+0f : 1.f);
}
__device__ __forceinline__ float unit_gain(int u) {
    return u & 2 ? (u & 1 ? 0x1.3077bep-1f : 0x1.6a09ecp-1f) : (u & 1 ? 0x1.ae6d8p-1f : 0x1.000008p+0f);
}

// A running sum covers at most this many units (16,384 samples); then it is
// added to the piece's slot, so that its rounding error does not grow with the
// length of the curve (382,003 samples in runs of any length: 8e-7 of the
// result's norm from the 64-bit one, against 4e-7 with the strip kernels).
constexpr int kRunUnits = 128;

// In each CTA of the pair, sixteen warps form the operands (its 64 coarse
// frequencies, its half of the fine offsets) and drain its accumulators, in
// four sets of four: a set fills every fourth stage of 32 samples, a thread 16
// coarse rows and up to 16 fine offsets of one sample, so that the four warps
// of an SM sub-partition are at different points of their work and hide each
// other's waits; six stage buffers leave a set two stages ahead of the MMAs.
// Warp 16 of the first CTA issues the MMAs of both (issuing blocks while the
// queue is full, so in a warp that also forms operands the two would take
// turns), all its lanes together but for the instruction itself.  The register split comes from setmaxnreg: 640 threads at 96
// registers launch, 512 x 112 + 128 x 32 are those 61,440.  Barriers:
// filled (a stage, counted at the first CTA) and empty, full (an accumulator, a
// unit's MMAs done), drained (counted at the first CTA) and finished.  No pair
// waits for another pair, and every wait has a limit.  Where one runs out, its warp
// stops waiting, the issuing one issues no more, and the status word makes the
// finalize pass write NaN; the tensor memory is given back and the CTAs end only
// after `finished`, which every MMA issued so far completes.
// GIVE_UP, for a test: every wait gives up at its first look.
template <bool GIVE_UP>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1) tc_sums_kernel(const TcArgs a) {
    extern __shared__ __align__(128) unsigned char stages[];
    Ahead& ahead = *reinterpret_cast<Ahead*>(stages + kBufs * kStageBytes);
    __shared__ uint64_t filled[kBufs], empty[kBufs], full[2], drained[2], finished;
    __shared__ uint32_t tbase;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int rank = (int)tc::pair_rank(), pair = blockIdx.x >> 1;
    if (tid == 0) {
#pragma unroll
        for (int i = 0; i < kBufs; ++i) {
            tc::mbar_init(&filled[i], 2 * kSetWarps);
            tc::mbar_init(&empty[i], 1);
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&full[i], 1);
            tc::mbar_init(&drained[i], 2 * kGenWarps);
        }
        tc::mbar_init(&finished, 1);
        tc::mbar_init_done();
    }
    if (warp == 0) tc::tmem_alloc(&tbase, 512);
    tc::fence_operands();
    tc::fence_before_sync();
    __syncthreads();
    tc::pair_sync();
    tc::fence_after_sync();
    const uint32_t tb = tbase;

    const int64_t lo = tc_bound(a.work, a.pairs, pair), hi = tc_bound(a.work, a.pairs, pair + 1);
    const int64_t cost0 = a.tiles ? 0 : (a.n0 + kTcUnit - 1) / kTcUnit * tc_unit_cost(a.one.cols);
    // first tile that reaches beyond lo
    int t = 0;
    if (a.tiles) {
        int h = a.n_tiles;
        while (t < h) {
            const int m = (t + h) >> 1;
            if (a.pre[m + 1] > lo) h = m;
            else t = m + 1;
        }
    } else {
        t = (int)(lo / cost0);
    }
    bool ok = true;
    auto wait = [](uint64_t* b, uint32_t parity) {
        return GIVE_UP ? tc::mbar_test(b, parity) : tc::mbar_wait(b, parity);
    };
    uint32_t group = 0, it = 0;  // units and stages so far
    // the next piece of a tile in this pair's range: its tile, first sample and length
    TileInfo f;
    int64_t j0 = 0;
    int left = 0;
    auto next_piece = [&]() {
        for (; t < a.n_tiles; ++t) {
            const int64_t p = a.tiles ? a.pre[t] : (int64_t)t * cost0;
            if (p >= hi) return false;
            f = tile_info(a, t);
            int64_t u0, u1;
            tc_units(p, (f.n + kTcUnit - 1) / kTcUnit, tc_unit_cost(f.w.cols), lo, hi, &u0, &u1);
            if (u0 >= u1) continue;
            j0 = f.b + u0 * kTcUnit;
            left = (int)(min(f.n, u1 * kTcUnit) - u0 * kTcUnit);
            return true;
        }
        return false;
    };

    if (warp >= kGenWarps) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
        if (warp == kGenWarps && rank == 0) {
            uint32_t buf = 0, phase = 0;
            for (; next_piece(); ++t) {
                const uint32_t id = tc::instr_desc(f.w.cols);
                for (int m = 0; m < left; m += kTcUnit, ++group) {
                    const uint32_t d = tb + (group & 1) * 256u;
                    if (group >= 2) ok = ok && wait(&drained[group & 1], ((group >> 1) - 1) & 1);
                    for (int q = m; q < min(left, m + kTcUnit); q += kStage) {
                        ok = ok && wait(&filled[buf], phase);
                        __syncwarp();
                        tc::fence_after_sync();
                        const uint64_t da = tc::operand_desc(tc::smem_addr(stages) + buf * kStageBytes, 128, kSbo);
                        const uint64_t db = da + (2 * kAbytes >> 4);
                        constexpr uint64_t al = kAbytes >> 4, bl = kBbytes >> 4, k1 = 256 >> 4;
                        const bool two = left - q > 16;  // the second 16 samples of the stage
                        if (tc::elect_one() && ok) {
                            tc::mma_f16(d, da, db + bl, id, q > m);  // hi lo
                            if (two) tc::mma_f16(d, da + k1, db + bl + k1, id, 1);
                            tc::mma_f16(d, da + al, db, id, 1);      // lo hi
                            if (two) tc::mma_f16(d, da + al + k1, db + k1, id, 1);
                            tc::mma_f16(d, da, db, id, 1);           // hi hi
                            if (two) tc::mma_f16(d, da + k1, db + k1, id, 1);
                            tc::mma_commit(&empty[buf]);
                            if (q + kStage >= min(left, m + kTcUnit)) tc::mma_commit(&full[group & 1]);
                        }
                        __syncwarp();
                        if (++buf == kBufs) {
                            buf = 0;
                            phase ^= 1;
                        }
                    }
                }
            }
            if (tc::elect_one()) tc::mma_commit(&finished);
        }
        __syncwarp();
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
        // this warp's set, its group of rows and offsets, its lanes and columns of the accumulators
        const int set = warp >> 2, grp = warp & 3, quad = grp, cg = set;
        for (; next_piece(); ++t) {
            const bool twice = f.w.twice;
            const int cols = f.w.cols, hb = cols >> 2;  // fine offsets (of one sign) of this CTA: hb
            const Group r = group_of(a, f, 4 * rank + grp);
            const float yscale = r.live ? r.scale : 0.f;
            const float* xrow = a.xr ? a.xr + (size_t)r.real * (size_t)a.total : nullptr;
            auto fetch = [&](int j) {    // sample j of the piece
                if (j < left) {
                    dev::cp_async16(&ahead.uv[tid], a.recA + j0 + j);
                    dev::cp_async16(&ahead.B[tid], a.recB + j0 + j);
                    dev::cp_async8(&ahead.E[tid], a.recE + j0 + j);
                    if (r.kind >= kTcW1) dev::cp_async4(&ahead.q[tid], a.q + j0 + j);
                    if (r.live && (r.kind == kTcRow || r.kind == kTcRowQ)) dev::cp_async4(&ahead.x[tid], xrow + j0 + j);
                } else {  // beyond the piece: zeros, and y = 0 below
                    ahead.uv[tid] = make_uint4(0, 0, 0, 0);
                    ahead.B[tid] = make_float4(0.f, 0.f, 0.f, 0.f);
                    ahead.E[tid] = make_float2(0.f, 0.f);
                    ahead.q[tid] = ahead.x[tid] = 0.f;
                }
                dev::cp_async_commit();
            };
            float run[64];
#pragma unroll
            for (int i = 0; i < 64; ++i) run[i] = 0.f;
            // adds a finished unit's accumulators to the running sums
            auto drain = [&](uint32_t g, int unit) {
                const float gain = unit_gain(unit);
                ok = ok && wait(&full[g & 1], (g >> 1) & 1);
                __syncwarp();
                tc::fence_after_sync();
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    if (cg * 64 + c * 32 < cols) {
                        uint32_t r[32];
                        tc::tmem_ld32(r, tb + (g & 1) * 256u + ((uint32_t)quad << 21) + (uint32_t)(cg * 64 + c * 32));
#pragma unroll
                        for (int i = 0; i < 32; ++i)
                            run[c * 32 + i] = fmaf(__uint_as_float(r[i]), gain, run[c * 32 + i]);
                    }
                }
                tc::fence_before_sync();
                __syncwarp();
                if (lane == 0) tc::mbar_arrive_first(&drained[g & 1]);
            };
            // the running sums into this piece's slot: columns of the tile, rows contiguous
            auto flush = [&](bool add) {
                float* const out = a.part + (size_t)(t + pair) * (size_t)a.slot_floats +
                                   (size_t)rank * (size_t)(a.slot_floats / 2) + (size_t)(cg * 64) * 128 + quad * 32 + lane;
                // rows of a CTA: real parts of its four groups, then imaginary parts
                const float inv = 1.f / group_of(a, f, 4 * rank + (2 * quad + (lane >> 4) & 3)).scale;
#pragma unroll
                for (int i = 0; i < 64; ++i)
                    if (cg * 64 + i < cols) out[i * 128] = fmaf(run[i], inv, add ? out[i * 128] : 0.f);
            };
            fetch(set * kStage + lane);
            for (int m = 0; m < left; m += kTcUnit, ++group) {
                const int jm = m + set * kStage;  // this set's stage of the unit
                if (jm < left) {
                    asm volatile("cp.async.wait_group 0;" ::: "memory");
                    const uint4 uv = ahead.uv[tid];
                    const float4 B = ahead.B[tid];
                    float2 e1 = make_float2(B.y, B.z), E = ahead.E[tid];
                    float y = jm + lane < left ? yscale * unit_scale(m / kTcUnit) : 0.f;
                    if (r.live) {
                        if (r.kind >= kTcW1) {
                            const float q = ahead.q[tid];
                            y *= q;
                            if (r.kind <= kTcW2) y *= q;
                        }
                        if ((r.kind & 3) > 1) y *= (r.kind & 1) ? ahead.x[tid] : B.x;
                    }
                    fetch(jm + kTcUnit + lane);
                    const uint64_t u = ((uint64_t)uv.y << 32) | uv.x;
                    const uint64_t v = (((uint64_t)uv.w << 32) | uv.z) - kPhaseOffset;
                    const uint64_t uh = u >> 1;
                    // the middle of the first of 16 coarse blocks of cols bins, and the first of 16 fine offsets
                    uint64_t pa = v + (uint64_t)((uint32_t)r.kg * (uint32_t)(kTcGroup * cols) + (uint32_t)(2 * hb)) * u - uh;
                    uint64_t pb = (uint64_t)(rank * hb + 16 * grp) * u + uh;
                    if (twice) {
                        pa <<= 1;
                        pb <<= 1;
                        e1 = csquare(e1);
                        E = csquare(E);
                    }
                    const uint32_t si = it + set, buf = si % kBufs, use = si / kBufs;
                    if (use > 0) ok = ok && wait(&empty[buf], (use - 1) & 1);
                    unsigned char* const Ah = stages + buf * kStageBytes + lane * 16;
                    {
                        float2 z = turn_cos_sin(pa);
                        z.x *= y;
                        z.y *= y;
                        const float2 E2 = csquare(E), E4 = csquare(E2), E8 = csquare(E4);
                        Pair p[4];
                        powers8(z, E, E2, E4, p);
                        unsigned char* re = Ah + 2 * grp * kSbo;
                        unsigned char* im = re + 8 * kSbo;
                        store_group(p, re, re + kAbytes, im, im + kAbytes);
#pragma unroll
                        for (int i = 0; i < 4; ++i) p[i] = mul_pair(p[i], E8);
                        store_group(p, re + kSbo, re + kSbo + kAbytes, im + kSbo, im + kSbo + kAbytes);
                    }
                    if (16 * grp < hb) {
                        const float2 e2 = csquare(e1), e4 = csquare(e2), e8 = csquare(e4);
                        Pair p[4];
                        powers8(turn_cos_sin(pb), e1, e2, e4, p);
                        unsigned char* co = Ah + 2 * kAbytes + 2 * grp * kSbo;
                        unsigned char* sn = co + (hb >> 3) * kSbo;
                        store_group(p, co, co + kBbytes, sn, sn + kBbytes);
                        if (16 * grp + 8 < hb) {
#pragma unroll
                            for (int i = 0; i < 4; ++i) p[i] = mul_pair(p[i], e8);
                            store_group(p, co + kSbo, co + kSbo + kBbytes, sn + kSbo, sn + kSbo + kBbytes);
                        }
                    }
                    tc::fence_operands();
                    __syncwarp();
                    if (lane == 0) tc::mbar_arrive_first(&filled[buf]);
                }
                it += (uint32_t)((min(left - m, kTcUnit) + kStage - 1) / kStage);
                if (m > 0) drain(group - 1, m / kTcUnit - 1);
                if (m > 0 && (m / kTcUnit) % kRunUnits == 0) {
                    flush(m / kTcUnit > kRunUnits);
#pragma unroll
                    for (int i = 0; i < 64; ++i) run[i] = 0.f;
                }
            }
            drain(group - 1, (left - 1) / kTcUnit);
            flush(left > kRunUnits * kTcUnit);
            asm volatile("cp.async.wait_group 0;" ::: "memory");
        }
    }
    if (warp == 0) ok = tc::mbar_wait(&finished, 0) && ok;
    if (!ok && a.status) atomicOr(a.status, kStatusWait);
    tc::fence_before_sync();
    __syncthreads();
    tc::pair_sync();
    if (warp == 0) tc::tmem_free(tb, 512);
}

// The slots of a tile's pieces, in order (the pairs that got at least one unit
// of it), and their number; one warp calls it.
struct Pieces {
    int n;
    int slot[kTcMaxPairs];
};

__device__ void find_pieces(const TcArgs& a, int tile, int64_t n, int cols, Pieces& out) {
    const int lane = threadIdx.x & 31;
    const int64_t units = (n + kTcUnit - 1) / kTcUnit, c = tc_unit_cost(cols);
    const int64_t p = a.tiles ? a.pre[tile] : (int64_t)tile * units * c;
    const int i0 = tc_pair_of(a.work, a.pairs, p), i1 = tc_pair_of(a.work, a.pairs, p + (units - 1) * c);
    int at = 0;
    if (i0 == i1) {
        if (lane == 0) out.slot[0] = tile + i0;
        at = 1;
    } else {
        for (int i = i0; i <= i1; i += 32) {
            const int me = i + lane;
            int64_t u0 = 0, u1 = 0;
            if (me <= i1) tc_units(p, units, c, tc_bound(a.work, a.pairs, me), tc_bound(a.work, a.pairs, me + 1), &u0, &u1);
            const unsigned has = __ballot_sync(0xffffffffu, u0 < u1);
            if (u0 < u1) out.slot[at + __popc(has & ((1u << lane) - 1u))] = tile + me;
            at += __popc(has);
        }
    }
    if (lane == 0) out.n = at;
}

// The complex sums at f_a + f_b and f_a - f_b of S tiles, from a tile's four
// entries each (at[x], cos, real part; the others 64 and hb columns on), the
// pieces added in order with compensated FP32 sums; four pieces of every tile
// are loaded before any of them is added.
template <int S>
__device__ __forceinline__ void tile_sums(const TcArgs& a, const Pieces* const (&q)[S], const size_t (&at)[S], int hb,
                                          float2 (&plus)[S], float2 (&minus)[S]) {
    float s[S][4] = {}, c[S][4] = {};
    const size_t step[4] = {0, 64, (size_t)hb * 128, (size_t)hb * 128 + 64};
    int most = q[0]->n;
#pragma unroll
    for (int x = 1; x < S; ++x) most = max(most, q[x]->n);
    if (most == 1) {  // a tile of one pair: nothing to add
#pragma unroll
        for (int x = 0; x < S; ++x)
#pragma unroll
            for (int i = 0; i < 4; ++i)
                s[x][i] = a.part[(size_t)q[x]->slot[0] * (size_t)a.slot_floats + at[x] + step[i]];
    } else {
        for (int i0 = 0; i0 < most; i0 += 4) {
            float v[S][4][4];
#pragma unroll
            for (int x = 0; x < S; ++x)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float* d = a.part + (size_t)q[x]->slot[min(i0 + u, q[x]->n - 1)] * (size_t)a.slot_floats + at[x];
#pragma unroll
                    for (int i = 0; i < 4; ++i) v[x][u][i] = i0 + u < q[x]->n ? d[step[i]] : 0.f;
                }
#pragma unroll
            for (int x = 0; x < S; ++x)
#pragma unroll
                for (int u = 0; u < 4; ++u)
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float y = v[x][u][i], t = s[x][i] + y;
                        c[x][i] += fabsf(s[x][i]) >= fabsf(y) ? (s[x][i] - t) + y : (y - t) + s[x][i];
                        s[x][i] = t;
                    }
        }
    }
#pragma unroll
    for (int x = 0; x < S; ++x) {
#pragma unroll
        for (int i = 0; i < 4; ++i) s[x][i] += c[x][i];
        plus[x] = make_float2(s[x][0] - s[x][3], s[x][1] + s[x][2]);
        minus[x] = make_float2(s[x][0] + s[x][3], s[x][1] - s[x][2]);
    }
}

// P from Z = sum x e and W = sum e^2: dev::periodogram_value2's two terms over
// their common denominator, where its square root and four of its five divisions
// cancel,
//     P = (n |Z|^2 - Re(conj(W) Z^2)) / (n^2 - |W|^2),
// while the two denominators n +- |W| are of a size; that form (with the rule on a
// vanishing term) where they are not.  This pass is bound by its instructions
// (65 % of the issue slots at 24 warps an SM before): 256 patterns by 64
// realizations, the call 12.90 -> 12.73 ms, one realization of 4096 9.47 -> 9.37.
__device__ __forceinline__ float classic_power(float2 Z, float2 W, float n) {
    const float nn = n * n, D = fmaf(-W.y, W.y, fmaf(-W.x, W.x, nn));
    if (!(D >= 0.125f * nn)) return dev::periodogram_value2(Z.x, Z.y, W.x, W.y, n);
    const float x2 = Z.x * Z.x, y2 = Z.y * Z.y;
    return fmaf(-W.y, 2.f * Z.x * Z.y, fmaf(-W.x, x2 - y2, n * (x2 + y2))) / D;
}

// Where the smaller eigenvalue of the floating-mean form's second moments is
// below this (f T under about a third, or an alias of it), P divides by a
// difference that separately rounded sums leave with too few digits (1.7e-3 of P
// at f T = 0.1; the strip kernels' sums, formed together, keep 1.9e-4): such bins
// are formed again, sample by sample and from moments that do not cancel.
constexpr float kGlsRefine = 0x1p-5f;

// P of the floating-mean form from Z = sum w x' e, C = sum w e, W = sum w e^2:
// dev::gls_value's two terms over their common denominator, where the square
// root and three of its four divisions cancel.  With M = W - C^2 (= A + iB, the
// centred CC - SS + 2i CS) and T = 1 - |C|^2 (CC + SS),
//     p = 2 (|Z|^2 T - Re(conj(M) Z^2)) / (T^2 - |M|^2).
// In FP32 pairs, whose 2^-48 the differences leave enough of: D >= T / 8 >= 1/64
// where the result is used.  The quotient is corrected once by its remainder.
// *ill: the smaller eigenvalue, between (T^2 - |M|^2) / 4T and / 2T, may lie
// below kGlsRefine; so it does where T does, whose sign is then lost in the sums'
// rounding.  (Not where the sums are NaN, of errors that the statistics refuse: P
// is 0 then, whichever way.)  n: the sample count.
__device__ __forceinline__ float gls_power(float2 Zf, float2 Cf, float2 Wf, dev::Pair n, bool* ill) {
    using dev::Pair;
    using dev::product;
    const Pair cx2 = product(Cf.x, Cf.x), cy2 = product(Cf.y, Cf.y);
    const Pair A = Pair{Wf.x, 0.f} + (cy2 + -cx2), B = Pair{Wf.y, 0.f} + product(-2.f * Cf.x, Cf.y);
    const Pair T = Pair{1.f, 0.f} + -(cx2 + cy2);
    const Pair D = T * T + -(A * A + B * B);
    const Pair sx = product(Zf.x, Zf.x), sy = product(Zf.y, Zf.y);
    const Pair num = T * (sx + sy) + -(A * (sx + -sy) + B * product(2.f * Zf.x, Zf.y));
    *ill = T.h < kGlsRefine || D.h + D.l < (float)(4.0 * kGlsRefine) * (T.h + T.l);
    const float r = 1.f / D.h, q = num.h * r;
    const float rest = (fmaf(-q, D.h, num.h) + num.l) - q * D.l;
    return fmaxf(rounded_product(Pair{q, rest * r}, n), 0.f);
}

// Sums over samples b + i0, b + i0 + step, ... < b + n at frequency k from which
// the centred moments of such a bin can be had without cancellation, with s =
// sin and v = 1 - cos of the phase (small where the phases are, and formed as
// such): w s, w v, w s^2, w v^2, w s v, w x' s, w x' v, w x'.  Compensated FP32
// (s + c).
constexpr int kMoments = 8;
__device__ __forceinline__ void direct_gls(const TcArgs& a, int64_t b, int64_t n, const float* x, uint32_t k, int i0,
                                           int step, float (&s)[kMoments], float (&c)[kMoments]) {
#pragma unroll 4
    for (int64_t j = b + i0; j < b + n; j += step) {
        const uint4 A = a.recA[j];
        const uint64_t u = ((uint64_t)A.y << 32) | A.x;
        const uint64_t ph = (((uint64_t)A.w << 32) | A.z) - kPhaseOffset + (uint64_t)k * u;
        const float2 e = turn_cos_sin(ph);
        // within an eighth of a turn 1 - cos by its series, from the signed turn
        const float h = (float)(int32_t)(uint32_t)(ph >> 32) * 1.4629180792671596e-9f, h2 = h * h;  // 2 pi / 2^32
        float v = fmaf(h2, 2.7557319223985888e-7f, -2.4801587301587302e-5f);
        v = fmaf(h2, v, 1.3888888888888889e-3f);
        v = fmaf(h2, v, -4.1666666666666664e-2f);
        v = h2 * fmaf(h2, v, 0.5f);
        if (fabsf(h) > 0.78f) v = 1.f - e.x;
        const float q = a.q[j], xj = x ? x[j] : a.recB[j].x;
        const float si = q * e.y, vi = q * v;
        const float f[kMoments] = {q, q, si, vi, si, xj, xj, xj}, g[kMoments] = {si, vi, si, vi, vi, si, vi, q};
#pragma unroll
        for (int i = 0; i < kMoments; ++i) {
            const float y = fmaf(f[i], g[i], c[i]), t = s[i] + y;
            c[i] = y - (t - s[i]);
            s[i] = t;
        }
    }
}

// P from those sums: dev::gls_value with the moments centred in FP64.  The
// smaller eigenvalue comes from the determinant, so that it keeps its digits; a
// direction whose eigenvalue is at most 2^-24 adds nothing, as there.
__device__ float moments_value(const float (&s)[kMoments], const float (&c)[kMoments], double n) {
    double m[kMoments];
#pragma unroll
    for (int i = 0; i < kMoments; ++i) m[i] = (double)s[i] + (double)c[i];
    const double ss = m[2] - m[0] * m[0], vv = m[3] - m[1] * m[1], sv = m[4] - m[0] * m[1];
    const double ys = m[5] - m[7] * m[0], yv = m[6] - m[7] * m[1];
    // cos = 1 - v: CC = vv, SS = ss, CS = -sv, YC = -yv, YS = ys
    const double T = vv + ss, A = vv - ss, B = -2.0 * sv, R = sqrt(A * A + B * B);
    const double big = 0.5 * (T + R), det = vv * ss - sv * sv, thr = 0x1p-24;
    if (!(big > thr)) return 0.f;
    if (det > thr * big) {
        const double p = (yv * yv * ss + ys * ys * vv - 2.0 * sv * yv * ys) / det;
        return (float)(0.5 * n * fmax(p, 0.0));
    }
    // the projection on the larger direction
    const double z2 = yv * yv + ys * ys, cross = R > 0.0 ? (A * (yv * yv - ys * ys) - 2.0 * B * yv * ys) / R : z2;
    return (float)(0.5 * n * fmax(0.5 * (z2 + cross), 0.0) / big);
}

constexpr int kFinB = 4;  // fine offsets a CTA takes at a time
constexpr int kFinRows = kTcGroups / 2 * kTcGroup;
constexpr int kFinThreads = kFinRows * kFinB;

// One CTA: the 64 coarse frequencies of half a tile (four groups) and every
// gridDim.y-th run of 4 fine offsets, both signs, a pair of frequencies a thread.
// Reads run along the coarse frequencies (contiguous in a slot).  P, where it is
// asked for, is gathered in shared memory and written in runs of 4 bins; the
// maxima need no exchange until the end.
template <int FORM>
__global__ void __launch_bounds__(kFinThreads, FORM == kTcGls ? 2 : 4) tc_final_kernel(const TcArgs a, const TcFinal f) {
    __shared__ float sp[kFinRows][2 * kFinB + 1];
    constexpr int S = FORM == kTcWindow ? 1 : FORM == kTcClassic ? 2 : 3;
    __shared__ Pieces pd, pw[4], pc[FORM == kTcGls ? 4 : 1];
    __shared__ unsigned long long s_red[kFinB][4];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int td = a.tiles ? f.data_tiles[blockIdx.x >> 1] : (int)blockIdx.x >> 1;
    const int half = (int)blockIdx.x & 1;
    const TileInfo t = tile_info(a, td);
    const TcTile& w = t.w;
    const int cols = w.cols, hb = cols >> 2, nb = cols >> 1;
    const int64_t n = t.n, nf = a.tiles ? f.nf[w.curve] : f.nf0;
    // this thread's row, its group's set and place in the grid, and the same
    // frequencies' rows in the h = 2 tile and in the set y = q^2
    const int ra = tid & (kFinRows - 1), bi = tid / kFinRows, grp = ra >> 4;
    const int G = w.g0 + 4 * half + grp, set = G / w.gpr, kl = G - set * w.gpr, Gc = w.reals * w.gpr + kl;
    const int64_t k0 = ((int64_t)(w.kg0 + kl) * kTcGroup + (ra & 15)) * cols;
    const bool live = set < w.reals && k0 < nf;
    const int real = w.r0 + set;
    const bool lost = a.status && (__ldcg(a.status) & kStatusWait);  // sums of a wait that ran out
    if (!__syncthreads_or(live)) return;
    {
        // warps 0 .. 3 find the h = 2 pieces of group `warp`, 4 .. 7 the y = q^2 ones, 0 the data tile's
        const int g = warp & 3, Gg = w.g0 + 4 * half + g, sg = Gg / w.gpr, lg = Gg - sg * w.gpr;
        if (FORM == kTcWindow) {
        } else if (warp < 4) find_pieces(a, w.wt0 + lg / kTcGroups, n, cols, pw[g]);
        else if (FORM == kTcGls) find_pieces(a, w.ht0 + (w.reals * w.gpr + lg) / kTcGroups, n, cols, pc[FORM == kTcGls ? g : 0]);
        if (warp == 0) find_pieces(a, td, n, cols, pd);
    }
    __syncthreads();
    const size_t half_slot = (size_t)(a.slot_floats / 2);
    auto row_at = [&](int g) { return (size_t)((g & 7) >> 2) * half_slot + (size_t)((g & 3) << 4 | (ra & 15)); };
    const size_t at_d = row_at(G - w.g0), at_w = row_at(kl), at_c = row_at(Gc);
    float* P = f.P;
    if (P && f.P_off) P += (size_t)real * (size_t)f.P_total + f.P_off[w.curve];
    unsigned long long best = 0ull;
    auto keep = [&](float p, int64_t k) {
        const unsigned long long key = ((unsigned long long)__float_as_uint(p) << 32) | (unsigned long long)(~(uint32_t)k);
        if (k < nf && !(FORM == kTcGls && p < 0.f)) best = key > best ? key : best;
    };
    for (int b0 = (int)blockIdx.y * kFinB; b0 < nb; b0 += (int)gridDim.y * kFinB) {
        const int rb = b0 + bi;
        if (live) {
            // columns: cos, sin of the first CTA's hb offsets, then of the second's
            const size_t col = (size_t)(rb < hb ? rb : hb + rb) * 128;
            const int64_t km = k0 + nb - 1 - rb, kp = k0 + nb + rb;
            float2 zp[S], zm[S];
            float vp, vm;
            if constexpr (FORM == kTcWindow) {
                const Pieces* const q[1] = {&pd};
                const size_t at[1] = {at_d + col};
                tile_sums<1>(a, q, at, hb, zp, zm);
                const float inv = 1.f / ((float)n * (float)n);
                vp = (zp[0].x * zp[0].x + zp[0].y * zp[0].y) * inv;
                vm = (zm[0].x * zm[0].x + zm[0].y * zm[0].y) * inv;
            } else if constexpr (FORM == kTcClassic) {
                const Pieces* const q[2] = {&pd, &pw[grp]};
                const size_t at[2] = {at_d + col, at_w + col};
                tile_sums<2>(a, q, at, hb, zp, zm);
                vp = classic_power(zp[0], zp[1], (float)n);
                vm = classic_power(zm[0], zm[1], (float)n);
            } else {
                const Pieces* const q[3] = {&pd, &pw[grp], &pc[grp]};
                const size_t at[3] = {at_d + col, at_w + col, at_c + col};
                tile_sums<3>(a, q, at, hb, zp, zm);
                bool lp, lm;
                vp = gls_power(zp[0], zp[2], zp[1], dev::pair_of((double)n), &lp);
                vm = gls_power(zm[0], zm[2], zm[1], dev::pair_of((double)n), &lm);
#pragma unroll 1
                for (int s = 0; s < 2; ++s) {
                    const int64_t k = s ? kp : km;
                    if (lost || !(s ? lp : lm) || k >= nf) continue;
                    const unsigned at = atomicAdd(f.n_bins, 1u);
                    if (at < (unsigned)kTcBins) {
                        f.bins[at] = TcBin{w.curve, real, (uint32_t)k, 0u};
                    } else {  // the list is full
                        const int fine = s ? nb + rb : nb - 1 - rb;
                        const int64_t row = (int64_t)blockIdx.x * kFinRows + ra;  // of the launch's h = 1 tiles
                        atomicOr(&f.mask[row * (a.slot_floats / tc_slot_floats(32)) + (fine >> 5)], 1u << (fine & 31));
                    }
                    (s ? vp : vm) = -1.f;  // left to launch_tc_refine
                }
            }
            if (lost) vm = vp = __int_as_float(0x7fc00000);
            keep(vm, km);
            keep(vp, kp);
            sp[ra][kFinB - 1 - bi] = vm;
            sp[ra][kFinB + bi] = vp;
        }
        if (!f.P) continue;
        __syncthreads();
        // bin i of a row: the minus run ends below the middle, the plus run starts above it; 8 threads a row
        for (int x = tid; x < kFinRows * 2 * kFinB; x += kFinThreads) {
            const int r = x / (2 * kFinB), i = x % (2 * kFinB);
            const int Gr = w.g0 + 4 * half + (r >> 4), sr = Gr / w.gpr;
            const int fine = i < kFinB ? nb - b0 - kFinB + i : nb + b0 + (i - kFinB);
            const int64_t k = ((int64_t)(w.kg0 + Gr - sr * w.gpr) * kTcGroup + (r & 15)) * cols + fine;
            if (sr < w.reals && k < nf) {
                const float p = sp[r][i];
                if (!(FORM == kTcGls && p < 0.f))
                    f.P[(f.P_off ? (size_t)(w.r0 + sr) * (size_t)f.P_total + f.P_off[w.curve] : 0) + k] = p;
            }
        }
        __syncthreads();
    }
    if (!f.maxkey) return;
    // the largest of each group: 16 lanes, then the four offsets
    for (int o = 8; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_down_sync(0xffffffffu, best, o, 16);
        best = y > best ? y : best;
    }
    if ((tid & 15) == 0) s_red[bi][grp] = best;
    __syncthreads();
    if (bi == 0 && (ra & 15) == 0 && set < w.reals) {
        for (int x = 1; x < kFinB; ++x) best = s_red[x][grp] > best ? s_red[x][grp] : best;
        if (best) atomicMax(&f.maxkey[(size_t)real * (size_t)f.n_curves + w.curve], best);
    }
}

constexpr int64_t kRefineAlone = 4096;

// s + c += t + d, s and t the leading parts (FP64 adds are slow on this part).
__device__ __forceinline__ void add_pair(float& s, float& c, float t, float d) {
    const float y = s + t, z = y - s;
    c += ((s - (y - z)) + (t - z)) + d;
    s = y;
}

// Joins the sums of the first `width` lanes in lane 0.
__device__ __forceinline__ void join_lanes(float (&s)[kMoments], float (&c)[kMoments], int width) {
    for (int o = width / 2; o > 0; o >>= 1)
#pragma unroll
        for (int x = 0; x < kMoments; ++x)
            add_pair(s[x], c[x], __shfl_down_sync(0xffffffffu, s[x], o), __shfl_down_sync(0xffffffffu, c[x], o));
}

// One cluster of CL CTAs per bin: its sums over all samples, then P.  A single long
// curve lists a few bins of many samples (CL = 8: 100,000 samples in
// one CTA are 40 us of arithmetic), a batch many bins of shorter curves (CL = 1),
// and a single short curve far beyond its mean Nyquist frequency thousands of bins
// with a sample or a few for each of 128 threads (500 samples, 100,000 frequencies
// on a nightly cadence, the finalize stage: CL = 8 78 us, 128 threads 20; 20,000
// samples, 2000 frequencies 31 and 68, 6000 by 12,000 31 and 39).
// With more bins than the list holds (a grid below 1 / 3T, one sample whose weight
// exceeds all others') a warp takes a bin, those listed and then those in the bit
// map: 100,000 samples by 200,000 such bins 72 ms, by clusters 135; 2000 patterns of
// 200 .. 1000 samples by 64 realizations, about one such bin each, the call 11.8 ms,
// by CTAs 14.3.  So how a bin is summed depends on the number of them, not on the
// order in which they came.
template <int CL, int kThreads>
__global__ void __launch_bounds__(kThreads) tc_refine_kernel(const TcArgs a, const TcFinal f) {
    __shared__ float2 sh[kThreads / 32][kMoments];
    __shared__ float2 part[CL][kMoments];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rank = CL > 1 ? (int)(blockIdx.x % CL) : 0;
    const unsigned found = *f.n_bins;
    auto sums = [&](const TcBin& w, int i0, int step, float (&s)[kMoments], float (&c)[kMoments]) {
        const int64_t b = a.off ? a.off[w.curve] : 0, n = a.off ? a.off[w.curve + 1] - b : a.n0;
#pragma unroll
        for (int x = 0; x < kMoments; ++x) s[x] = c[x] = 0.f;
        direct_gls(a, b, n, a.xr ? a.xr + (size_t)w.real * (size_t)a.total : nullptr, w.k, i0, step, s, c);
    };
    auto put = [&](const TcBin& w, const float (&s)[kMoments], const float (&c)[kMoments]) {
        const int64_t n = a.off ? a.off[w.curve + 1] - a.off[w.curve] : a.n0;
        const float p = moments_value(s, c, (double)n);
        if (f.P) f.P[(size_t)w.real * (size_t)f.P_total + (f.P_off ? f.P_off[w.curve] : 0) + w.k] = p;
        if (f.maxkey)
            atomicMax(&f.maxkey[(size_t)w.real * (size_t)f.n_curves + w.curve],
                      ((unsigned long long)__float_as_uint(p) << 32) | (unsigned long long)(~w.k));
    };
    float s[kMoments], c[kMoments];
    if (found > (unsigned)kTcBins) {
        auto form = [&](const TcBin& w) {
            sums(w, lane, 32, s, c);
            join_lanes(s, c, 32);
            if (lane == 0) put(w, s, c);
        };
        const int me = blockIdx.x * (kThreads / 32) + warp, all = gridDim.x * (kThreads / 32);
        for (int i = me; i < kTcBins; i += all) form(f.bins[i]);
        const int per_row = (int)(a.slot_floats / tc_slot_floats(32));  // words
        const int64_t words = tc_mask_words(a.tiles ? f.n_data : a.h1, 32 * per_row);
        // an odd number of warps: such bins are often the first of every row, a fixed number of words apart
        for (int64_t word = me; word < words && me < all - 1; word += all - 1) {
            unsigned bits = f.mask[word];
            if (!bits) continue;
            __syncwarp();
            if (lane == 0) f.mask[word] = 0u;
            const int64_t row = word / per_row;
            const int tile = (int)(row / (2 * kFinRows)), r = (int)(row % (2 * kFinRows));
            const TcTile w = tile_of(a, a.tiles ? f.data_tiles[tile] : tile);
            const int G = w.g0 + r / kTcGroup, set = G / w.gpr;
            const int64_t k0 = ((int64_t)(w.kg0 + G - set * w.gpr) * kTcGroup + r % kTcGroup) * w.cols + word % per_row * 32;
            // (a bit left by a call whose refine pass was never launched may lie beyond this grid)
            const int64_t bins = set < w.reals ? (a.tiles ? f.nf[w.curve] : f.nf0) - k0 : 0;
            if (bins < 32) bits &= bins > 0 ? (1u << (int)bins) - 1u : 0u;
            for (; bits; bits &= bits - 1) form(TcBin{w.curve, w.r0 + set, (uint32_t)k0 + (uint32_t)__ffs(bits) - 1u, 0u});
        }
        return;
    }
    for (unsigned i = blockIdx.x / CL; i < found; i += gridDim.x / CL) {
        const TcBin w = f.bins[i];
        sums(w, rank * kThreads + (int)threadIdx.x, CL * kThreads, s, c);
        join_lanes(s, c, 32);
        if (lane == 0)
#pragma unroll
            for (int x = 0; x < kMoments; ++x) sh[warp][x] = make_float2(s[x], c[x]);
        __syncthreads();
        if (warp == 0) {
#pragma unroll
            for (int x = 0; x < kMoments; ++x) {
                const float2 v = lane < kThreads / 32 ? sh[lane][x] : make_float2(0.f, 0.f);
                s[x] = v.x;
                c[x] = v.y;
            }
            join_lanes(s, c, kThreads / 32);
        }
        if constexpr (CL > 1) {
            if (threadIdx.x == 0) {
                float2* first = cooperative_groups::this_cluster().map_shared_rank(&part[0][0], 0);
#pragma unroll
                for (int x = 0; x < kMoments; ++x) first[rank * kMoments + x] = make_float2(s[x], c[x]);
            }
            cooperative_groups::this_cluster().sync();
            if (threadIdx.x == 0 && rank == 0) {
                for (int r = 1; r < CL; ++r)
#pragma unroll
                    for (int x = 0; x < kMoments; ++x) add_pair(s[x], c[x], part[r][x].x, part[r][x].y);
            }
        }
        if (threadIdx.x == 0 && rank == 0) put(w, s, c);
        if constexpr (CL > 1) cooperative_groups::this_cluster().sync();
        else __syncthreads();
    }
}

}  // namespace

cudaError_t launch_tc_refine(const TcArgs& a, const TcFinal& f, cudaStream_t st) {
    if (a.off || a.n0 <= kRefineAlone) {
        if (a.off) tc_refine_kernel<1, 512><<<304, 512, 0, st>>>(a, f);
        else tc_refine_kernel<1, 128><<<152 * 8, 128, 0, st>>>(a, f);
        return cudaGetLastError();
    }
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 8;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(304);
    cfg.blockDim = dim3(512);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, tc_refine_kernel<8, 512>, a, f);
}

cudaError_t launch_tc_sums(const TcArgs& a, cudaStream_t st) {
    auto* const kernel = a.give_up ? tc_sums_kernel<true> : tc_sums_kernel<false>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    kernel<<<2 * a.pairs, kTcThreads, kSmem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_tc_final(int form, const TcArgs& a, const TcFinal& f, cudaStream_t st) {
    const int n_data = a.tiles ? f.n_data : a.h1;
    if (n_data < 1) return cudaSuccess;
    const int max_cols = (int)(a.slot_floats / tc_slot_floats(1));
    // all runs of offsets in CTAs of their own, until there are some thousands of CTAs
    int y = (max_cols / 2 + kFinB - 1) / kFinB;
    const int most = 8192 / (2 * n_data);
    y = y > most ? (most < 1 ? 1 : most) : y;
    dim3 grid((unsigned)n_data * 2u, (unsigned)y);
    if (form == kTcClassic) tc_final_kernel<kTcClassic><<<grid, kFinThreads, 0, st>>>(a, f);
    else if (form == kTcGls) tc_final_kernel<kTcGls><<<grid, kFinThreads, 0, st>>>(a, f);
    else tc_final_kernel<kTcWindow><<<grid, kFinThreads, 0, st>>>(a, f);
    return cudaGetLastError();
}

}  // namespace lsp
