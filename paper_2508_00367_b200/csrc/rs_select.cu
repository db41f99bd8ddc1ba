// Per-sample selection of the K = N - r highest-score tokens and compaction of
// the kept rows (Sec. 3.1: the reduced token set; Sec. 3.2: the r lowest-score
// tokens are removed).
//
// Selection is exact and order-stable: fp32 scores are mapped to uint32 keys that sort like the
// floats (NaN lowest); the key of the K-th best token is found by a search over the key bits, ties at
// that key go to the lower indices by a prefix count, and a prefix count of the kept tokens yields the
// ascending index list directly, with no sort.  Integer work only once the keys are formed, hence
// bit-exact.
#include "rs_internal.h"
#include "rs_device.cuh"
#include <type_traits>

namespace rs {

namespace {

// Score of one token from the partial sums the GEMM epilogues leave (fixed summation
// order: run-to-run identical).  `enc` = number of partial sums | distance << 16.  L2: sqrt of the sum of
// squares; L1: the sum; cosine: three sums per part (u.v, u.u, v.v) -> 1 - u.v / (|u||v|).
// The number of parts is even (two column halves per tile) and the rows start on 8-byte boundaries; sixteen
// parts are loaded before the first is added, so a token costs one round trip to L2 (adding as they came
// left two to four loads in flight and made the scores half of the selection's time).
__device__ __forceinline__ float finish_score(const float* __restrict__ p, int enc) {
    const int nparts = enc & 0xffff, dist = enc >> 16;
    if (dist == RS_DIST_COS) {
        float uv = 0.f, uu = 0.f, vv = 0.f;
        for (int j = 0; j < nparts; ++j) { uv += p[3 * j]; uu += p[3 * j + 1]; vv += p[3 * j + 2]; }
        return 1.f - uv / fmaxf(sqrtf(uu) * sqrtf(vv), 1e-12f);
    }
    const float2* p2 = reinterpret_cast<const float2*>(p);
    float acc = 0.f;
    for (int j0 = 0; j0 < nparts; j0 += 16) {
        float2 v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j0 + 2 * j < nparts) v[j] = __ldg(p2 + j0 / 2 + j);
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (j0 + 2 * j < nparts) { acc += v[j].x; acc += v[j].y; }
    }
    return dist == RS_DIST_L1 ? acc : sqrtf(acc);
}
__device__ __forceinline__ int partial_stride(int enc) { return (enc & 0xffff) * ((enc >> 16) == RS_DIST_COS ? 3 : 1); }

__device__ __forceinline__ uint32_t score_key(float s) {
    if (s != s) return 0u;                 // NaN ranks below every number
    if (s == 0.f) s = 0.f;                 // -0 and +0 tie
    const uint32_t b = __float_as_uint(s);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Per-sample lengths (lens, drops non-null): sample b has n_b = lens[b] tokens (clamped to 1 .. N) at
// the front of its N rows and drops r_b = drops[b] of them (clamped to 0 .. n_b - 1); the rows past
// n_b are never kept.
struct Ragged { const int32_t* lens; const int32_t* drops; int32_t* lens_out; };
__device__ __forceinline__ void sample_counts(const Ragged& rg, int b, int N, int K, int* n_b, int* k_b) {
    if (!rg.lens) { *n_b = N; *k_b = K; return; }
    const int n = min(max(__ldg(rg.lens + b), 1), N);
    const int r = min(max(__ldg(rg.drops + b), 0), n - 1);
    *n_b = n; *k_b = min(n - r, K);          // K: the row stride of the outputs, an upper bound of every count
}

constexpr int kSelMaxThreads = 1024;

// Block-wide sums of two packed counts (each below 2^16 in all), one barrier per call: every warp leaves its
// sum in a slot of the parity's row and adds up all slots itself.
struct Counts { uint32_t a, b; };
__device__ __forceinline__ Counts block_counts(uint32_t a, uint32_t b, uint2 (*slots)[32], int parity, int nw) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    a = __reduce_add_sync(0xffffffffu, a);
    b = __reduce_add_sync(0xffffffffu, b);
    if (lane == 0) slots[parity][warp] = make_uint2(a, b);
    __syncthreads();
    const uint2 v = lane < nw ? slots[parity][lane] : make_uint2(0u, 0u);
    return {__reduce_add_sync(0xffffffffu, v.x), __reduce_add_sync(0xffffffffu, v.y)};
}

// Prefix counts of flags in token order (the block's threads take consecutive tokens, slot e after slot e - 1):
// mask[e] holds this warp's flags of slot e; afterwards before(e, ...) is the number of set flags in the groups
// of 32 tokens before this warp's group of slot e.  Warp c scans the c-th 32 groups (KPT <= 32, so there are
// never more of those than warps); two barriers.
template <int KPT> struct GroupScan {
    int in_chunk[32 * KPT];                // exclusive prefix inside the group's 32
    int chunk_total[32];
    __device__ __forceinline__ int run(const unsigned (&mask)[KPT], int nw) {   // returns this lane's share of the chunk prefix
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
        for (int e = 0; e < KPT; ++e)
            if (lane == 0) in_chunk[e * nw + warp] = __popc(mask[e]);
        __syncthreads();
        const int groups = KPT * nw, idx = warp * 32 + lane;
        if (warp * 32 < groups) {
            const int v = idx < groups ? in_chunk[idx] : 0;
            int inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (lane >= o) inc += t;
            }
            if (idx < groups) in_chunk[idx] = inc - v;
            if (lane == 31) chunk_total[warp] = inc;
        }
        __syncthreads();
        const int v = lane * 32 < groups ? chunk_total[lane] : 0;
        int inc = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        return inc - v;                    // lane c: flags before the c-th 32 groups
    }
    __device__ __forceinline__ int before(int e, int nw, int chunk_prefix) const {
        const int g = e * nw + (threadIdx.x >> 5);
        return __shfl_sync(0xffffffffu, chunk_prefix, g >> 5) + in_chunk[g];
    }
};

// Selection of one sample by one CTA, every key in a register (KPT per thread, token e * blockDim + tid in
// slot e).  The key t of the last token that makes the cut is the largest t with at least `want` keys >= t:
// a search over the key bits below the candidates' common prefix, two bits (three candidate keys, counted
// together) per step and one barrier per step, ended early when some candidate key leaves exactly `want` --
// about log2(N) bits after the common prefix.  A few hundred cycles per step, so the kernel is bound by
// latency: launch, one read of the scores, about eight steps and two prefix sums.
// Measured on B200 (graph of 50 calls, scores given), against what it replaced: 32 x 577 tokens 3.8 us (17.8:
// every token ranked against every other by N / 64 CTAs per sample), 512 x 197 5.8 us (38.5), 4 x 4097 6.8 us
// (15.7: radix passes over shared memory by one CTA per sample), 10 x 14466 19 us (40.5).
template <int KPT>
__global__ void __launch_bounds__(kSelMaxThreads)
select_kernel(const float* __restrict__ scores, int nparts, float* __restrict__ scores_out, int N, int K, int has_cls,
              int32_t* __restrict__ keep_idx, int32_t* __restrict__ row_map, const Ragged rg) {
    __shared__ uint2 slots[2][32];
    __shared__ GroupScan<KPT> scan_eq, scan_kept;
    grid_dep_launch();
    grid_dep_wait();
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, nt = blockDim.x, nw = nt >> 5;
    int n_b, k_b;
    sample_counts(rg, b, N, K, &n_b, &k_b);
    const int first = has_cls ? 1 : 0;     // token 0 is kept unconditionally when has_cls
    const int want = k_b - first;          // tokens to choose among the candidates [first, n_b)
    if (tid == 0 && rg.lens_out) rg.lens_out[b] = k_b;

    uint32_t key[KPT];                     // 0 for tokens that are no candidates: no candidate key of the search counts them
    uint32_t all_and = 0xffffffffu, all_or = 0u;
#pragma unroll
    for (int e = 0; e < KPT; ++e) {
        const int i = e * nt + tid;
        key[e] = 0u;
        if (i < N) {
            float s;
            if (nparts > 0) {              // partial sums from the GEMM epilogue
                s = finish_score(scores + ((long long)b * N + i) * partial_stride(nparts), nparts);
                if (scores_out) scores_out[(long long)b * N + i] = s;
            } else {
                s = __ldg(scores + (long long)b * N + i);
            }
            if (i >= first && i < n_b) { key[e] = score_key(s); all_and &= key[e]; all_or |= key[e]; }
        }
    }

    uint32_t t = 0;                        // keep every candidate with key > t, and need_eq of those with key == t
    int need_eq = 0;
    bool cut_ties = false;                 // more candidates at t than are kept: the lowest indices win
    if (want > 0 && want < n_b - first) {
        all_and = __reduce_and_sync(0xffffffffu, all_and);
        all_or = __reduce_or_sync(0xffffffffu, all_or);
        if (lane == 0) slots[1][tid >> 5] = make_uint2(all_and, all_or);
        __syncthreads();
        {
            const uint2 v = lane < nw ? slots[1][lane] : make_uint2(0xffffffffu, 0u);
            all_and = __reduce_and_sync(0xffffffffu, v.x);
            all_or = __reduce_or_sync(0xffffffffu, v.y);
        }
        const uint32_t diff = all_and ^ all_or;
        int bits = diff ? 32 - __clz(diff) : 0;          // bits still open
        t = bits == 32 ? 0u : all_and & ~((1u << bits) - 1u);
        uint32_t n_t = (uint32_t)(n_b - first), n_above = 0;   // candidates >= t, and >= the smallest key known to leave too few
        bool exact = false;
        for (int step = 0; bits > 0 && !exact; ++step) {
            // candidate keys t + d * 2^(bits - 2), d = 1, 2, 3 (a single open bit: d = 2 only)
            const int sh = bits >= 2 ? bits - 2 : 0;
            const uint32_t c1 = bits >= 2 ? t | (1u << sh) : 0xffffffffu, c2 = bits >= 2 ? t | (2u << sh) : t | 1u,
                           c3 = bits >= 2 ? t | (3u << sh) : 0xffffffffu;
            uint32_t m12 = 0, m3 = 0;
#pragma unroll
            for (int e = 0; e < KPT; ++e) {
                m12 += (key[e] >= c1 ? 1u : 0u) + (key[e] >= c2 ? 0x10000u : 0u);
                m3 += key[e] >= c3 ? 1u : 0u;
            }
            const Counts n = block_counts(m12, m3, slots, step & 1, nw);
            const uint32_t n1 = n.a & 0xffffu, n2 = n.a >> 16, n3 = n.b, w = (uint32_t)want;
            // the largest candidate key with enough tokens; the next larger one bounds it from above
            if (n3 >= w) { t = c3; n_t = n3; }
            else if (n2 >= w) { t = c2; n_t = n2; n_above = bits >= 2 ? n3 : n_above; }
            else if (n1 >= w) { t = c1; n_t = n1; n_above = n2; }
            else n_above = bits >= 2 ? n1 : n2;
            exact = n_t == w;
            bits -= 2;
        }
        // exact: all candidates >= t are kept.  Otherwise t is the key of the last kept token itself and
        // n_above counts the candidates beyond it (with a single key in the sample: none, all tie).
        need_eq = exact ? (int)n_t : want - (int)n_above;
        cut_ties = !exact && (int)(n_t - n_above) > need_eq;
        if (exact && t > 0) { t -= 1; need_eq = 0; }     // key > t - 1 is key >= t (t == 0: ties at 0 are kept below)
    } else if (want >= n_b - first) {
        need_eq = n_b;                                   // every candidate: key > 0, or NaN (key 0)
    }

    // keep flags; then each kept token's position from the prefix counts
    unsigned mask[KPT];
    if (cut_ties) {
        unsigned eq[KPT];
#pragma unroll
        for (int e = 0; e < KPT; ++e) {
            const int i = e * nt + tid;
            eq[e] = __ballot_sync(0xffffffffu, i >= first && i < n_b && key[e] == t);
        }
        const int cp = scan_eq.run(eq, nw);
#pragma unroll
        for (int e = 0; e < KPT; ++e) {
            const int i = e * nt + tid, rank = scan_eq.before(e, nw, cp) + __popc(eq[e] & ((1u << lane) - 1u));
            const bool keep = i < first || (want > 0 && i < n_b && (key[e] > t || (key[e] == t && rank < need_eq)));
            mask[e] = __ballot_sync(0xffffffffu, keep);
        }
    } else {
#pragma unroll
        for (int e = 0; e < KPT; ++e) {
            const int i = e * nt + tid;
            const bool keep = i < first || (want > 0 && i < n_b && (key[e] > t || (key[e] == t && need_eq > 0)));
            mask[e] = __ballot_sync(0xffffffffu, keep);
        }
    }
    const int cp = scan_kept.run(mask, nw);
    int32_t* out = keep_idx + (long long)b * K;
#pragma unroll
    for (int e = 0; e < KPT; ++e) {
        const int i = e * nt + tid;
        const int base = scan_kept.before(e, nw, cp);
        if ((mask[e] >> lane) & 1u) {
            const int pos = base + __popc(mask[e] & ((1u << lane) - 1u));
            out[pos] = i;
            if (row_map) row_map[(long long)b * K + pos] = b * N + i;
        }
    }
    if (rg.lens)                           // rows of the padded output past this sample's count
        for (int j = k_b + tid; j < K; j += nt) out[j] = -1;
}

// One warp moves one kept row (16-byte pieces, all loads of a pass issued before its first store):
// to row `orow` of x_out when x_out is given, and, with LT given, LN of the row to the same row of
// ln.out.
template <int MAXV, typename LT>
__device__ __forceinline__ void copy_row(const uint4* __restrict__ src, long long orow, int row_vecs, int lane,
                                         uint4* __restrict__ x_out, const LnFuse& ln) {
    if constexpr (std::is_void<LT>::value) {
        uint4* dst = x_out + orow * row_vecs;
        float s1 = 0.f, s2 = 0.f;
        for (int base = 0; base < row_vecs; base += 32 * MAXV) {
            uint4 v[MAXV];
#pragma unroll
            for (int j = 0; j < MAXV; ++j) {
                const int iv = base + j * 32 + lane;
                if (iv < row_vecs) v[j] = __ldg(src + iv);
            }
#pragma unroll
            for (int j = 0; j < MAXV; ++j) {
                const int iv = base + j * 32 + lane;
                if (iv < row_vecs) {
                    dst[iv] = v[j];
                    if (ln.stats) {                  // bf16 rows only (the caller's business)
                        const uint32_t w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float y0 = __uint_as_float(w[e] << 16), y1 = __uint_as_float(w[e] & 0xffff0000u);
                            s1 += y0 + y1;
                            s2 = fmaf(y0, y0, fmaf(y1, y1, s2));
                        }
                    }
                }
            }
        }
        if (ln.stats) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            if (lane == 0) { ln.stats[2 * orow] = s1; ln.stats[2 * orow + 1] = s2; }
        }
    } else {
        uint4 v[MAXV];
#pragma unroll
        for (int j = 0; j < MAXV; ++j) {
            const int iv = j * 32 + lane;
            if (iv < row_vecs) v[j] = __ldg(src + iv);
        }
        if (x_out) {
            uint4* dst = x_out + orow * row_vecs;
#pragma unroll
            for (int j = 0; j < MAXV; ++j) {
                const int iv = j * 32 + lane;
                if (iv < row_vecs) dst[iv] = v[j];
            }
        }
        const int D = row_vecs * Vec16<LT>::N;
        layernorm_row<LT, LT, MAXV>(v, row_vecs, lane, ln.gamma, ln.beta, ln.eps, D, reinterpret_cast<LT*>(ln.out) + orow * D);
    }
}

// Sum and sum of squares of a row of bf16 values held by a warp as 16-byte pieces (zeros where a lane has none),
// to out[0], out[1]: the statistics of a LayerNorm folded into the next product.
template <int NV>
__device__ __forceinline__ void row_sums(const uint4 (&v)[NV], int lane, float* __restrict__ out) {
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
        const uint32_t w[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float y0 = __uint_as_float(w[e] << 16), y1 = __uint_as_float(w[e] & 0xffff0000u);
            s1 += y0 + y1;
            s2 = fmaf(y0, y0, fmaf(y1, y1, s2));
        }
    }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    if (lane == 0) { out[0] = s1; out[1] = s2; }
}

// Nothing dropped (K == N): every token is kept, in order; only the scores remain to be
// finished when they arrive as per-tile partial sums of squares.
__global__ void __launch_bounds__(256)
keep_all_kernel(const float* __restrict__ scores, int nparts, float* __restrict__ scores_out, long long T, int N,
                int32_t* __restrict__ keep_idx) {
    grid_dep_launch();
    grid_dep_wait();
    const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
    if (t >= T) return;
    if (nparts > 0 && scores_out) scores_out[t] = finish_score(scores + t * partial_stride(nparts), nparts);
    keep_idx[t] = (int32_t)(t % N);
}

// x_out[b, j, :] = x[b, keep_idx[b, j], :] (zeros where the index is -1); with LT given, LN of the row to ln.out.
// One warp per row, 16-byte pieces, all loads of a row issued before the first store.
template <int MAXV, typename LT>
__global__ void __launch_bounds__(256)
gather_kernel(const uint4* __restrict__ x, const int32_t* __restrict__ keep_idx, unsigned rows, int N,
              unsigned K, int row_vecs, uint4* __restrict__ x_out, const LnFuse ln) {
    grid_dep_launch();
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const unsigned row = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int src = __ldg(keep_idx + row);
    if (src < 0) {
        if (x_out)
            for (int iv = lane; iv < row_vecs; iv += 32) x_out[(long long)row * row_vecs + iv] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    copy_row<MAXV, LT>(x + ((long long)(row / K) * N + src) * row_vecs, row, row_vecs, lane, x_out, ln);
}

// The same for rows of at most 32 * VPR pieces, RPW = 4 / VPR rows per warp, so that a lane has four loads in
// flight whatever the width (a row of 192 bf16 is 24 pieces: one load per lane).  Bound by HBM / L2: 256 x 181 rows
// of 192 bf16 3.8 us after the selection = 9.3 TB/s out of L2.
template <int VPR>
__global__ void __launch_bounds__(256)
gather_short_kernel(const uint4* __restrict__ x, const int32_t* __restrict__ keep_idx, unsigned rows, int N,
                    unsigned K, int row_vecs, uint4* __restrict__ x_out, float* __restrict__ stats) {
    constexpr int RPW = 4 / VPR;
    grid_dep_launch();
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const unsigned row0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * RPW;
    if (row0 >= rows) return;
    const int mine = lane < RPW && row0 + lane < rows ? __ldg(keep_idx + row0 + lane) : -1;
    uint4 v[RPW][VPR];
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        const int src = __shfl_sync(0xffffffffu, mine, r);
        const uint4* s = x + ((long long)((row0 + r) / K) * N + (src < 0 ? 0 : src)) * row_vecs;
#pragma unroll
        for (int j = 0; j < VPR; ++j) {
            v[r][j] = make_uint4(0u, 0u, 0u, 0u);
            if (src >= 0 && j * 32 + lane < row_vecs) v[r][j] = __ldg(s + j * 32 + lane);
        }
    }
#pragma unroll
    for (int r = 0; r < RPW; ++r) {
        if (row0 + r >= rows) break;
        uint4* dst = x_out + (long long)(row0 + r) * row_vecs;
#pragma unroll
        for (int j = 0; j < VPR; ++j)
            if (j * 32 + lane < row_vecs) dst[j * 32 + lane] = v[r][j];
        if (stats) row_sums<VPR>(v[r], lane, stats + 2 * (long long)(row0 + r));
    }
}

// Line-wise pruning of an H x W token grid (Sec. 4, CNN variant L-W): the shift is averaged over
// every row and every column of the full grid, and the lines with the lowest averages go.  Grid
// (G, B): every CTA of sample b repeats the cheap part — one thread per line sums its line in
// fp64 in index order (the order a plain loop takes, so the averages are the same doubles on any
// machine), ranks it among its peers by counting (larger average first, lower index on a tie, NaN
// last) and the kept lines are numbered by a count over the flags — and then copies its share of
// the Hk x Wk kept positions, a warp per position.  CTA 0 of the sample writes the two index lists.
constexpr int kLineMax = 256;
constexpr int kMapMax = 8192;               // scores of one sample staged in shared memory (32 KB)

__device__ __forceinline__ bool line_outranks(double a, int ia, double b, int ib) {
    if (a != a) return (b != b) && ia < ib;
    if (b != b) return true;
    return a > b || (a == b && ia < ib);
}

template <int MAXV>
__global__ void __launch_bounds__(256)
linewise_kernel(const float* __restrict__ scores, int H, int W, int Hk, int Wk, int32_t* __restrict__ keep_rows,
                int32_t* __restrict__ keep_cols, const uint4* __restrict__ x, int row_vecs, uint4* __restrict__ x_out) {
    __shared__ double mean[2 * kLineMax];      // rows, then columns
    __shared__ int32_t kept[2 * kLineMax];
    __shared__ unsigned char flag[2 * kLineMax];
    __shared__ float smap[kMapMax];
    grid_dep_launch();
    grid_dep_wait();
    const int b = blockIdx.y;
    const float* s = scores + (long long)b * H * W;
    // a map of up to kMapMax scores is staged in shared memory first (coalesced, all threads), so
    // that the per-line loops below do not wait on global memory one element at a time
    const bool staged = H * W <= kMapMax;
    if (staged) {
        for (int i = threadIdx.x; i < H * W; i += blockDim.x) smap[i] = s[i];
        __syncthreads();
    }
    const float* sv = staged ? smap : s;
    for (int l = threadIdx.x; l < H + W; l += blockDim.x) {
        double acc = 0.0;
        if (l < H) {
            for (int w = 0; w < W; ++w) acc += (double)sv[l * W + w];
            mean[l] = acc / (double)W;
        } else {
            const int c = l - H;
            for (int h = 0; h < H; ++h) acc += (double)sv[h * W + c];
            mean[kLineMax + c] = acc / (double)H;
        }
    }
    __syncthreads();
    for (int l = threadIdx.x; l < H + W; l += blockDim.x) {
        const bool row = l < H;
        const int i = row ? l : l - H, n = row ? H : W, want = row ? Hk : Wk;
        const double* m = mean + (row ? 0 : kLineMax);
        const double mine = m[i];
        int rank = 0;
        for (int j = 0; j < n; ++j) rank += (j != i) && line_outranks(m[j], j, mine, i);
        flag[(row ? 0 : kLineMax) + i] = rank < want;
    }
    __syncthreads();
    for (int l = threadIdx.x; l < H + W; l += blockDim.x) {
        const bool row = l < H;
        const int i = row ? l : l - H, off = row ? 0 : kLineMax;
        if (!flag[off + i]) continue;
        int pos = 0;
        for (int j = 0; j < i; ++j) pos += flag[off + j];
        kept[off + pos] = i;
        if (blockIdx.x == 0) (row ? keep_rows + (long long)b * Hk : keep_cols + (long long)b * Wk)[pos] = i;
    }
    __syncthreads();
    if (!x) return;
    const int P = Hk * Wk, G = gridDim.x, per = (P + G - 1) / G;
    const int lo = blockIdx.x * per, hi = min(lo + per, P);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    const LnFuse none = {nullptr, nullptr, 0.f, nullptr, nullptr};
    auto src_of = [&](int p) {
        const int i = p / Wk, j = p - i * Wk;
        return x + (((long long)b * H + kept[i]) * W + kept[kLineMax + j]) * row_vecs;
    };
    if (row_vecs <= 32) {
        // short rows (up to 512 bytes): a warp takes 32 / rv positions side by side (rv = the row's
        // 16-byte pieces rounded up to a power of two) and four such groups per step, so that every
        // lane has four loads in flight
        int rv = 1;
        while (rv < row_vecs) rv <<= 1;
        const int side = 32 / rv, sub = lane / rv, v = lane - sub * rv, step = side * 4;
        for (int p0 = lo + warp * step; p0 < hi; p0 += nwarps * step) {
            uint4 val[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + u * side + sub;
                if (p < hi && v < row_vecs) val[u] = __ldg(src_of(p) + v);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + u * side + sub;
                if (p < hi && v < row_vecs) x_out[((long long)b * P + p) * row_vecs + v] = val[u];
            }
        }
        return;
    }
    for (int p = lo + warp; p < hi; p += nwarps)
        copy_row<MAXV, void>(src_of(p), (long long)b * P + p, row_vecs, lane, x_out, none);
}

}  // namespace

cudaError_t launch_select(const float* scores, int nparts, float* scores_out, int B, int N, int K, int has_cls,
                          int32_t* keep_idx, int32_t* row_map, cudaStream_t st, const int32_t* seq_lens,
                          const int32_t* drops, int32_t* lens_out) {
    if (B == 0) return cudaSuccess;
    if (K == N && !seq_lens) {
        const long long T = (long long)B * N;
        return launch_pdl(keep_all_kernel, dim3((unsigned)((T + 255) / 256)), dim3(256), 0, st, scores, nparts, scores_out, T, N, keep_idx);
    }
    const Ragged rg = {seq_lens, drops, lens_out};
    // keys per thread: the fewest that leave at most 1024 threads (latency is what counts: more threads per
    // sample mean fewer keys to compare per step), whole warps
#define RS_SEL_CASE(KPT)                                                                                            \
    if (N <= KPT * kSelMaxThreads)                                                                                  \
        return launch_pdl(select_kernel<KPT>, dim3(B), dim3(((N + KPT - 1) / KPT + 31) / 32 * 32), 0, st, scores,   \
                          nparts, scores_out, N, K, has_cls, keep_idx, row_map, rg)
    RS_SEL_CASE(1);
    RS_SEL_CASE(2);
    RS_SEL_CASE(5);
    RS_SEL_CASE(16);
    RS_SEL_CASE(32);
#undef RS_SEL_CASE
    return cudaErrorInvalidValue;
}

bool ln_fusable(rs_dtype dtype, int D) { return (size_t)D * dtype_size(dtype) / 16 <= 32 * 4; }

cudaError_t launch_gather(rs_dtype dtype, const void* x, const int32_t* keep_idx, int B, int N, int K,
                          int D, void* x_out, const LnFuse* ln, cudaStream_t st) {
    const long long rows = (long long)B * K;
    if (rows == 0) return cudaSuccess;
    if (rows >= (1ll << 31)) return cudaErrorInvalidValue;
    const int row_vecs = (int)((size_t)D * dtype_size(dtype) / 16);
    const bool norm = ln && ln->gamma;               // else ln, if given, only asks for the row sums of the copy
    if ((norm && !ln_fusable(dtype, D)) || (!x_out && !norm)) return cudaErrorInvalidValue;
    const LnFuse none = {nullptr, nullptr, 0.f, nullptr, nullptr};
#define RS_G_CASE(LT)                                                                                                 \
    launch_pdl(gather_kernel<4, LT>, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, (const uint4*)x, keep_idx,   \
               (unsigned)rows, N, (unsigned)K, row_vecs, (uint4*)x_out, ln ? *ln : none)
#define RS_GS_CASE(VPR)                                                                                               \
    launch_pdl(gather_short_kernel<VPR>, dim3((unsigned)((rows + 32 / VPR - 1) / (32 / VPR))), dim3(256), 0, st,      \
               (const uint4*)x, keep_idx, (unsigned)rows, N, (unsigned)K, row_vecs, (uint4*)x_out, ln ? ln->stats : nullptr)
    if (!norm) return row_vecs <= 32 ? RS_GS_CASE(1) : row_vecs <= 64 ? RS_GS_CASE(2) : RS_G_CASE(void);
    return dtype == RS_BF16 ? RS_G_CASE(__nv_bfloat16) : RS_G_CASE(float);
#undef RS_GS_CASE
#undef RS_G_CASE
}

int linewise_max_lines() { return kLineMax; }

cudaError_t launch_linewise(const float* scores, int B, int H, int W, int Hk, int Wk, int32_t* keep_rows,
                            int32_t* keep_cols, rs_dtype dtype, const void* x, int D, void* x_out, int sm_count,
                            cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int row_vecs = x ? (int)((size_t)D * dtype_size(dtype) / 16) : 0;
    // about eight CTAs per SM in all (measured best between six and twelve), at least 16 positions
    // each; one CTA per sample for the indices alone
    int G = 1;
    if (x) {
        G = (8 * sm_count + B - 1) / B;
        const int cap = (Hk * Wk + 15) / 16;
        if (G > cap) G = cap;
        if (G < 1) G = 1;
    }
    return launch_pdl(linewise_kernel<4>, dim3(G, B), dim3(256), 0, st, scores, H, W, Hk, Wk, keep_rows, keep_cols,
                      (const uint4*)x, row_vecs, (uint4*)x_out);
}

}  // namespace rs
