// tc_sums.cuh -- the tensor-core evaluation of the periodogram's sums: work
// list, launch interface and the closed-form split of the work over the CTAs
// (shared by the kernels of tc_sums.cu and their callers).
#pragma once

#include "lsp_kernels.cuh"

namespace lsp {

// What a tile sums over its curve's samples j, for a block of frequencies:
// sum_j y_j exp(2 pi i h phase_j(k)).
enum : int {
    kTcOne1 = 0,  // y = 1, h = 1: the spectral window
    kTcOne2 = 1,  // y = 1, h = 2: CC - SS + 2i CS
    kTcRec = 2,   // y = x_hat of the records, h = 1: XC + i XS
    kTcRow = 3,   // y = x_hat of a realization's row, h = 1
    kTcW1 = 4,    // y = q^2, h = 1: the floating-mean form's C + i S
    kTcW2 = 5,    // y = q^2, h = 2
    kTcRecQ = 6,  // y = q x_hat of the records, h = 1
    kTcRowQ = 7   // y = q x_hat of a realization's row, h = 1
};

// Work on a curve's sums is cut into groups of 16 coarse frequencies of cols bins
// each, gpr of them for a grid; tiles are eight groups that share the fine
// offsets.  Groups of the h = 1 sums run through the realizations in order and,
// in the floating-mean form, end with the group set of y = q^2: group G is
// coarse frequencies 16 (G mod gpr) .. of set G / gpr.  So a short grid's
// realizations share tiles, whose cost hardly depends on how full they are.
struct TcTile {
    int32_t curve, kind;    // kind of the data sets (h = 1) or of the tile (twice)
    int32_t twice;          // an h = 2 tile: one set
    int32_t g0;             // first group
    int32_t r0, reals;      // data sets: realizations r0 .. r0 + reals
    int32_t gls;            // an h = 1 tile's sets end with y = q^2
    int32_t gpr, kg0, cols; // groups of a set, the grid's group that is its first, bins of a coarse frequency
    int32_t wt0, ht0;       // first h = 2 and first h = 1 tile of these groups
};

constexpr int kTcGroup = 16;       // coarse frequencies of a group
constexpr int kTcGroups = 8;       // groups of a tile (four a CTA: 128 operand rows, real and imaginary parts)
constexpr int kTcMaxCols = 256;    // fine offsets of a tile, at most
constexpr int kTcUnit = 128;       // samples of one unit of work
constexpr int kTcThreads = 640;
constexpr int kTcMaxPairs = 256;  // CTA pairs that a launch is split over, at most

// Cost of a unit of a tile: the operands (64 complex values a sample for a CTA's
// coarse frequencies and cols / 4 for its fine offsets) take longer than the MMAs
// (proportional to cols) below 256 columns.
__host__ __device__ inline int tc_unit_cost(int cols) { return 8 + cols / 32; }

// Bins per coarse frequency (a multiple of 32 up to 256) for a grid of N_f bins
// and `sets` sets of its h = 1 sums: the one whose tiles cost least.
inline int tc_cols(int64_t N_f, int64_t sets) {
    int best = kTcMaxCols;
    int64_t best_cost = INT64_MAX;
    for (int c = kTcMaxCols; c >= 32; c -= 32) {
        const int64_t gpr = (N_f + kTcGroup * c - 1) / (kTcGroup * c);
        const int64_t cost =
            ((sets * gpr + kTcGroups - 1) / kTcGroups + (gpr + kTcGroups - 1) / kTcGroups) * tc_unit_cost(c);
        if (cost < best_cost) {
            best_cost = cost;
            best = c;
        }
    }
    return best;
}

struct TcArgs {
    // tiles: a list with the prefix sums of their costs (pre[0..n_tiles]), or,
    // for a single curve (tiles == nullptr), `one` with g0 = 8 t for tile
    // t < h1 and, twice and of kind win_kind, g0 = 8 (t - h1) from there on
    const TcTile* tiles;
    const int64_t* pre;
    int n_tiles, h1, win_kind;
    TcTile one;
    int64_t n0;                 // samples of the single curve
    int64_t work;               // total cost
    int pairs;                  // CTA pairs the work is split over
    const int64_t* off;         // curves' sample offsets (list form)
    const uint4* recA;
    const float4* recB;
    const float2* recE;         // (cos, sin)(2 pi cols u)
    const float* q;             // sqrt weights (floating mean)
    const float* qmax;          // largest q of each curve
    const float* xr;            // realization rows
    int64_t total;              // row stride of xr
    float* part;                // slots of slot_floats: tile t's piece by pair i is slot t + i, the halves of its
    int64_t slot_floats;        // two CTAs one after the other, each [cols][128 rows]
    int* status;
    bool give_up;               // a test: every wait on a barrier gives up at its first look
};

// Where the work coordinate of pair i starts.
__host__ __device__ inline int64_t tc_bound(int64_t work, int pairs, int i) { return work * i / pairs; }
// The pair whose range holds coordinate x.
__host__ __device__ inline int tc_pair_of(int64_t work, int pairs, int64_t x) {
    return (int)(((x + 1) * pairs - 1) / work);
}
// Floats of a slot for tiles of up to cols columns.
__host__ __device__ inline int64_t tc_slot_floats(int cols) { return 256 * (int64_t)cols; }
// Pairs on a GPU of `sms` SMs.
inline int tc_pairs(int sms) { return sms < 2 ? 1 : sms / 2 < kTcMaxPairs ? sms / 2 : kTcMaxPairs; }
// Units [u0, u1) of a tile that starts at coordinate p (n units of cost c each)
// whose starts lie in [lo, hi).
__host__ __device__ inline void tc_units(int64_t p, int64_t n, int64_t c, int64_t lo, int64_t hi, int64_t* u0,
                                         int64_t* u1) {
    const int64_t a = lo <= p ? 0 : (lo - p + c - 1) / c, b = hi <= p ? 0 : (hi - p + c - 1) / c;
    *u0 = a < n ? a : n;
    *u1 = b < n ? b : n;
}

// The finalize pass over the h = 1 tiles: P (kTcWindow: |sum|^2 / n^2) of every
// frequency of their data sets.
// A bin of the floating-mean form whose sums are formed again by
// launch_tc_refine: realization `real` of `curve`, frequency k.
struct TcBin {
    int32_t curve, real;
    uint32_t k, pad;
};
constexpr int kTcBins = 1 << 16;  // bins the list holds; the others of a launch are marked in a bit map of its h = 1 tiles
// Words of the bit map of n h = 1 tiles of up to cols columns: 128 rows (coarse frequencies) of cols bits each.
__host__ __device__ inline int64_t tc_mask_words(int64_t n, int cols) { return n * 128 * (cols / 32); }

struct TcFinal {
    const int* data_tiles;      // list form: indices of the h = 1 tiles
    int n_data;
    const int64_t* nf;          // list form
    int64_t nf0;                // single curve
    float* P;                   // may be null
    const int64_t* P_off;
    int64_t P_total;
    unsigned long long* maxkey; // may be null
    int n_curves;
    TcBin* bins;                // floating mean: list of ill-conditioned bins and
    unsigned* n_bins;           // its counter (zeroed by launch_prep_stats, after qmax)
    unsigned* mask;             // bit map of the others (zero before and after)
};

enum : int { kTcClassic = 0, kTcGls = 1, kTcWindow = 2 };

cudaError_t launch_tc_sums(const TcArgs& a, cudaStream_t st);
cudaError_t launch_tc_final(int form, const TcArgs& a, const TcFinal& f, cudaStream_t st);
// Floating mean: the bins that the launch_tc_final before it, with the same
// arguments, listed and marked.  n_bins is to be zero before the next one.
cudaError_t launch_tc_refine(const TcArgs& a, const TcFinal& f, cudaStream_t st);

}  // namespace lsp
