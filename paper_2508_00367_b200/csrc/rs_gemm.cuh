// What the two tensor-core GEMM kernels share: the epilogues' names, arguments and arithmetic (Eq. att, Eq. MLP, Sec. 3.2).
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "rs.h"

namespace rs {
namespace gemm {

// EPI_SCORE_STATS: EPI_SCORE that also leaves, per row and 64 columns, the sum and the sum of
// squares of the (rounded) output values -- the row statistics of the next block's LayerNorm.
// EPI_BIAS_LN: the LayerNorm of the A operand folded into the product: with W' = W * gamma (column-wise),
// c_n = sum_k W'_nk and b'_n = b_n + sum_k W_nk beta_k,  LN(x) W^T + b = rstd (x W'^T - mu c) + b';  mu and
// rstd of a row come from the statistics above, acc = x W'^T from the tensor cores.
enum { EPI_BIAS = 0, EPI_BIAS_GELU = 1, EPI_RESID = 2, EPI_SCORE = 3, EPI_SCORE_STATS = 4, EPI_BIAS_LN = 5 };

struct GemmArgs {
    int M, N, K;
    const float* bias;        // [N] or null
    const void* residual;     // EPI_RESID: bf16 [M, N];  EPI_SCORE: fp32 [M, N]
    const void* residual2;    // EPI_SCORE, score_kind 2: bf16 [M, N] block input x
    const int* row_map;       // optional [M]: row t of the block input (EPI_RESID's residual, EPI_SCORE's residual2)
                              // is row row_map[t] of that matrix (the previous block's un-pruned output, read in place)
    float* partials;          // EPI_SCORE (and EPI_RESID when non-null): [M, N / 64] sums, one per 64 columns
    int score_kind;           // EPI_SCORE: scored pair (u, v) = 0: (m, x'), 1: (x^, x'), 2: (x^, x)
    int dist;                 // rs_dist of the score: L2 / L1 sums of (u - v)^2 / |u - v|, cosine sums of u.v, u.u, v.v
    float* stats_out;         // EPI_SCORE_STATS: [M, N / 64][2] = (sum, sum of squares) of the row's outputs in those 64 columns
    const float* stats_in;    // EPI_BIAS_LN: such statistics of the A operand's rows, stats_parts pairs per row over ln_dim = K values
    const float* colsum;      // EPI_BIAS_LN: c [N]
    int stats_parts;
    float ln_eps;
    const int* lens;          // optional [M / seq_n]: rows come as samples of seq_n, sample b's first lens[b] are in use;
    int seq_n;                // rows past them (and past kPadRows more) need not be computed
    int* status;
};
// Rows behind a sample's own that are computed all the same: attention multiplies values of up to 15 of them by zero
// weights, so they have to be finite.
constexpr int kPadRows = 16;
// Rows of sample b (of seq_n) that have to be computed.  A count is whatever the caller's array holds: it is clamped before
// kPadRows is added (INT_MAX for "the whole sample" would wrap around).
__device__ __forceinline__ int rows_needed(const int* __restrict__ lens, int b, int seq_n) {
    return min(min(max(__ldg(lens + b), 1), seq_n) + kPadRows, seq_n);
}

// Batches with a count per sample: row tiles that hold padding alone are left out.  Up to this many row tiles of 256.
constexpr int kMaskWords = 32, kMaskTiles = 32 * kMaskWords;
// The k-th row tile in use, for a caller whose k never decreases.
struct RowTiles {
    const uint32_t* mask;    // null: all
    int word = 0, before = 0;
    __device__ __forceinline__ int at(int k) {
        if (!mask) return k;
        while (word < kMaskWords - 1 && before + __popc(mask[word]) <= k) before += __popc(mask[word++]);
        uint32_t m = mask[word];
        for (int i = before; i < k; ++i) m &= m - 1;
        return word * 32 + __ffs(m) - 1;
    }
};

// Which row tiles of 256 rows hold rows in use (at most kMaskTiles), written to shared memory by the whole CTA of `threads`;
// returns how many do.
__device__ __forceinline__ int mark_row_tiles(uint32_t* mask, const int* __restrict__ lens, int seq_n, int M, int warp, int lane, int threads) {
    for (int t0 = warp * 32; t0 < kMaskTiles; t0 += threads) {
        const int r0 = (t0 + lane) * 256, r1 = min(r0 + 256, M);
        bool used = false;
        for (int b = r0 / seq_n; r0 < M && b * seq_n < r1 && !used; ++b) used = b * seq_n + rows_needed(lens, b, seq_n) > r0;
        const uint32_t w = __ballot_sync(0xffffffffu, used);
        if (lane == 0) mask[t0 / 32] = w;
    }
    __syncthreads();
    int tiles = 0;
    for (int w = 0; w < kMaskWords; ++w) tiles += __popc(mask[w]);
    return tiles;
}

// Adds one element of the scored pair (u, v) to the running sums of the chosen distance (Sec. 3.3).  Called with a
// constant distance in the pair-tile kernel (with_dist): the choice is made once per 32 columns there.
__device__ __forceinline__ void score_acc(int dist, float u, float v, float& s0, float& s1, float& s2) {
    if (dist == RS_DIST_L2) { const float d = u - v; s0 = fmaf(d, d, s0); }
    else if (dist == RS_DIST_L1) { s0 += fabsf(u - v); }
    else { s0 = fmaf(u, v, s0); s1 = fmaf(u, u, s1); s2 = fmaf(v, v, s2); }
}

template <typename F> __device__ __forceinline__ void with_dist(int dist, F f) {
    if (dist == RS_DIST_L2) f(std::integral_constant<int, RS_DIST_L2>{});
    else if (dist == RS_DIST_L1) f(std::integral_constant<int, RS_DIST_L1>{});
    else f(std::integral_constant<int, RS_DIST_COS>{});
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

}  // namespace gemm

}  // namespace rs
