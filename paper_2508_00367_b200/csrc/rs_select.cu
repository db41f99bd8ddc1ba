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
// Sixteen parts are loaded before the first is added, so a token costs one round trip to L2 (adding as they came
// left two to four loads in flight and made the scores half of the selection's time).
__device__ __forceinline__ float finish_score(const float* __restrict__ p, int enc) {
    const int nparts = enc & 0xffff, dist = enc >> 16;
    if (dist == RS_DIST_COS) {
        float uv = 0.f, uu = 0.f, vv = 0.f;
        for (int j = 0; j < nparts; ++j) { uv += p[3 * j]; uu += p[3 * j + 1]; vv += p[3 * j + 2]; }
        return 1.f - uv / fmaxf(sqrtf(uu) * sqrtf(vv), 1e-12f);
    }
    float acc = 0.f;
    for (int j0 = 0; j0 < nparts; j0 += 16) {
        float v[16];
        if ((nparts & 3) == 0) {             // rows start on 16-byte boundaries
#pragma unroll
            for (int j = 0; j < 16; j += 4)
                if (j0 + j < nparts) {
                    const float4 t = __ldg(reinterpret_cast<const float4*>(p + j0 + j));
                    v[j] = t.x; v[j + 1] = t.y; v[j + 2] = t.z; v[j + 3] = t.w;
                }
        } else {
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (j0 + j < nparts) v[j] = __ldg(p + j0 + j);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j0 + j < nparts) acc += v[j];
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
            if (i >= n_b) {                // padding of a batch with a count per sample: its rows may not even have been computed
                s = 0.f;
                if (nparts > 0 && scores_out) scores_out[(long long)b * N + i] = s;
            } else if (nparts > 0) {       // partial sums from the GEMM epilogue
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

// Adds the eight bf16 values of a 16-byte piece and their squares: the statistics of a LayerNorm folded into the
// next product.
__device__ __forceinline__ void add_row_sums(const uint4& v, float& s1, float& s2) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float y0 = __uint_as_float(w[e] << 16), y1 = __uint_as_float(w[e] & 0xffff0000u);
        s1 += y0 + y1;
        s2 = fmaf(y0, y0, fmaf(y1, y1, s2));
    }
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
                    if (ln.stats) add_row_sums(v[j], s1, s2);    // bf16 rows only (the caller's business)
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

// Source row of output row `row` (-1: the output row is zeros).  TokenRows: row j of sample b is token
// keep_idx[b, j].  GridRows: position (i, j) of the kept grid is position (keep_rows[i], keep_cols[j]).
struct TokenRows {
    const int32_t* keep_idx;
    unsigned K;
    int N;
    __device__ __forceinline__ long long operator()(unsigned row) const {
        const int t = __ldg(keep_idx + row);
        return t < 0 ? -1 : (long long)(row / K) * N + t;
    }
};
struct GridRows {
    const int32_t *keep_rows, *keep_cols;
    unsigned Hk, Wk;
    int H, W;
    __device__ __forceinline__ long long operator()(unsigned row) const {
        const unsigned line = row / Wk, j = row - line * Wk, b = line / Hk;        // line = b * Hk + i
        return ((long long)b * H + __ldg(keep_rows + line)) * W + __ldg(keep_cols + b * Wk + j);
    }
};

// x_out[row, :] = x[src(row), :]; with LT given, LN of the row to ln.out.
// One warp per row, 16-byte pieces, all loads of a row issued before the first store.  CTAs take the rows from
// the last to the first: what the kernel before this one touched last is what the L2 still holds of an input
// larger than it (512 x 197 tokens of 768 bf16 after their scores: 43 -> 41 us, 6.9 TB/s read and written; an
// evict-first hint on the writes as well cost 2 us).
template <int MAXV, typename LT, typename Src>
__global__ void __launch_bounds__(256)
gather_kernel(const uint4* __restrict__ x, const Src src_of, unsigned rows, int row_vecs, uint4* __restrict__ x_out, const LnFuse ln) {
    grid_dep_launch();
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const unsigned row = (gridDim.x - 1 - blockIdx.x) * 8 + (threadIdx.x >> 5);
    if (row >= rows) return;
    const long long src = src_of(row);
    if (src < 0) {
        if (x_out)
            for (int iv = lane; iv < row_vecs; iv += 32) x_out[(long long)row * row_vecs + iv] = make_uint4(0u, 0u, 0u, 0u);
        return;
    }
    copy_row<MAXV, LT>(x + src * row_vecs, row, row_vecs, lane, x_out, ln);
}

// The same copy for rows of at most 32 * VPR pieces: a lane keeps four loads in flight whatever the width.
// VPR 2: two rows per warp.  VPR 1: four groups of 32 >> lsh rows side by side, 1 << lsh lanes (the pieces of a
// row rounded up to a power of two) per row.  Bound by HBM / L2: 256 x 181 rows of 192 bf16 take 3.8 us after the
// selection = 9.3 TB/s out of L2.
template <int VPR, typename Src>
__global__ void __launch_bounds__(256)
gather_short_kernel(const uint4* __restrict__ x, const Src src_of, unsigned rows, int row_vecs, int lsh,
                    uint4* __restrict__ x_out, float* __restrict__ stats) {
    constexpr int U = 4 / VPR;
    grid_dep_launch();
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    if (VPR > 1) lsh = 5;
    const unsigned side = 32u >> lsh, sub = (unsigned)lane >> lsh;
    const int v0 = lane & ((1 << lsh) - 1);
    const unsigned row0 = ((gridDim.x - 1 - blockIdx.x) * 8 + (threadIdx.x >> 5)) * U * side + sub;
    uint4 v[U][VPR];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const unsigned row = row0 + u * side;
        const long long src = row < rows ? src_of(row) : -1;
#pragma unroll
        for (int j = 0; j < VPR; ++j) {
            v[u][j] = make_uint4(0u, 0u, 0u, 0u);
            if (src >= 0 && j * 32 + v0 < row_vecs) v[u][j] = __ldg(x + src * row_vecs + j * 32 + v0);
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const unsigned row = row0 + u * side;
#pragma unroll
        for (int j = 0; j < VPR; ++j)
            if (row < rows && j * 32 + v0 < row_vecs) x_out[(long long)row * row_vecs + j * 32 + v0] = v[u][j];
        if (stats) {
            float s1 = 0.f, s2 = 0.f;
#pragma unroll
            for (int j = 0; j < VPR; ++j) add_row_sums(v[u][j], s1, s2);
            for (int o = 1 << lsh >> 1; o > 0; o >>= 1) {
                s1 += __shfl_xor_sync(0xffffffffu, s1, o);
                s2 += __shfl_xor_sync(0xffffffffu, s2, o);
            }
            if (v0 == 0 && row < rows) reinterpret_cast<float2*>(stats)[row] = make_float2(s1, s2);
        }
    }
}

// Line-wise pruning of an H x W token grid (Sec. 4, CNN variant L-W): the shift is averaged over
// every row and every column of the full grid, and the lines with the lowest averages go.  One CTA per
// sample finds the kept lines -- one thread per line sums it in fp64 in index order (the order a plain loop
// takes, so the averages are the same doubles on any machine), ranks it among its peers by counting (larger
// average first, lower index on a tie, NaN last) and takes its position from the flags' ballots -- and the
// gather kernels above move the kept positions.  (Repeating the selection in every CTA that copied positions
// left room for five CTAs of 256 threads per SM and made all of them start with it: 64 maps of 56 x 56 x 256
// took 52 us that way, 150 MB at 2.9 TB/s; the two kernels take 30.)
constexpr int kLineMax = 256;
constexpr int kMapMax = 8192;               // scores of one sample staged in shared memory (33 KB)

// A double as a key that sorts like it: NaN below every number, -0 = +0.
__device__ __forceinline__ unsigned long long line_key(double a) {
    if (a != a) return 0ull;
    if (a == 0.0) a = 0.0;
    const unsigned long long b = (unsigned long long)__double_as_longlong(a);
    return b >> 63 ? ~b : b | (1ull << 63);
}

__global__ void __launch_bounds__(2 * kLineMax)
line_select_kernel(const float* __restrict__ scores, int H, int W, int Hk, int Wk, int32_t* __restrict__ keep_rows,
                   int32_t* __restrict__ keep_cols) {
    __shared__ unsigned long long key[2][kLineMax];    // rows, then columns
    __shared__ unsigned mask[2][kLineMax / 32];
    __shared__ float smap[kMapMax + kLineMax];
    grid_dep_launch();
    grid_dep_wait();
    const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
    const float* s = scores + (long long)b * H * W;
    // a map of up to kMapMax scores is staged in shared memory first (coalesced, all threads; an odd row
    // stride keeps the row sums free of bank conflicts), so that the sums do not wait on global memory
    const bool staged = H * W <= kMapMax;
    const int ld = staged ? W | 1 : W;
    if (staged) {
        for (int i = tid; i < H * W; i += 2 * kLineMax) {
            const int r = i / W;
            smap[r * ld + (i - r * W)] = s[i];
        }
        __syncthreads();
    }
    const float* sv = staged ? smap : s;
    const int kind = tid / kLineMax, l = tid - kind * kLineMax;        // threads 0 .. 255: rows, the rest: columns
    const int n = kind ? W : H, len = kind ? H : W, want = kind ? Wk : Hk;
    if (l < n) {
        const float* p = sv + (kind ? l : l * ld);
        const int step = kind ? ld : 1;
        double acc = 0.0;
#pragma unroll 8
        for (int e = 0; e < len; ++e) acc += (double)p[e * step];
        key[kind][l] = line_key(acc / (double)len);
    }
    __syncthreads();
    bool keep = false;
    if (l < n) {
        const unsigned long long mine = key[kind][l];
        int rank = 0;
#pragma unroll 4
        for (int j = 0; j < n; ++j) rank += key[kind][j] > mine || (key[kind][j] == mine && j < l);
        keep = rank < want;
    }
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) mask[kind][l >> 5] = m;
    __syncthreads();
    if (!keep) return;
    int pos = __popc(m & ((1u << lane) - 1u));
    for (int w = 0; w < l >> 5; ++w) pos += __popc(mask[kind][w]);
    (kind ? keep_cols + (long long)b * Wk : keep_rows + (long long)b * Hk)[pos] = l;
}

// Launch of the copy: several narrow rows per warp, else a warp per row.  Few narrow rows are done sooner with a warp each,
// too: several / one to a warp, us with the selection kernel before it, 200 x 192 bf16 3.1 / 2.5, 6000 x 192 3.7 / 3.3,
// 8000 x 192 3.7 / 3.9, 40000 x 192 6.2 / 8.9; two / one to a warp 200 x 384 2.7 / 2.5, 4000 x 384 3.2 / 3.4.
template <typename Src>
cudaError_t launch_copy(const void* x, const Src& src, long long rows, int row_vecs, void* x_out, const LnFuse& ln, int sm_count, cudaStream_t st) {
    const int vpr = row_vecs <= 32 ? 1 : 2;
    if (row_vecs <= 64 && rows > (vpr == 1 ? 48ll : 20ll) * sm_count) {
        int lsh = 0;
        while (lsh < 5 && (1 << lsh) < row_vecs) ++lsh;
        const unsigned per_cta = vpr == 1 ? 8 * 4 * (32u >> lsh) : 16;
        const dim3 grid((unsigned)((rows + per_cta - 1) / per_cta));
        return vpr == 1 ? launch_pdl(gather_short_kernel<1, Src>, grid, dim3(256), 0, st, (const uint4*)x, src, (unsigned)rows, row_vecs, lsh, (uint4*)x_out, ln.stats)
                        : launch_pdl(gather_short_kernel<2, Src>, grid, dim3(256), 0, st, (const uint4*)x, src, (unsigned)rows, row_vecs, lsh, (uint4*)x_out, ln.stats);
    }
    return launch_pdl(gather_kernel<4, void, Src>, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, (const uint4*)x, src, (unsigned)rows, row_vecs, (uint4*)x_out, ln);
}

// launch(first sample, rows) over whole samples of `per_sample` rows: the kernels count the rows of a launch in 32 bits, so a
// batch of 2^31 rows or more goes in several launches.
template <typename F> cudaError_t by_samples(int B, int per_sample, F launch) {
    const long long most = ((1ll << 31) - 1) / per_sample;
    for (long long b0 = 0; b0 < B; b0 += most) {
        const cudaError_t e = launch(b0, (B - b0 < most ? B - b0 : most) * per_sample);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_select(const float* scores, int nparts, float* scores_out, int B, int N, int K, int has_cls,
                          int32_t* keep_idx, int32_t* row_map, int sm_count, cudaStream_t st, const int32_t* seq_lens,
                          const int32_t* drops, int32_t* lens_out) {
    if (B == 0) return cudaSuccess;
    if (K == N && !seq_lens) {
        const long long T = (long long)B * N;
        return launch_pdl(keep_all_kernel, dim3((unsigned)((T + 255) / 256)), dim3(256), 0, st, scores, nparts, scores_out, T, N, keep_idx);
    }
    const Ragged rg = {seq_lens, drops, lens_out};
    // keys per thread: the fewest that leave at most 1024 threads (latency is what counts: more threads per
    // sample mean fewer keys to compare per step), whole warps.  With samples for two rounds and more it is samples at a time
    // that count: more than 512 threads of the kernel's 64 registers leave room for one CTA on an SM, so that 2561 to 5120
    // tokens take sixteen keys a thread there.  Five / sixteen, us: 256 x 4097 18.2 / 20.1, 512 x 2561 25.8 / 20.1, 512 x 4097
    // 32.2 / 27.6, 2048 x 4097 111 / 81.
    const bool many = B >= 2 * sm_count && N > 2560;
#define RS_SEL_CASE(KPT)                                                                                            \
    if (N <= KPT * kSelMaxThreads)                                                                                  \
        return launch_pdl(select_kernel<KPT>, dim3(B), dim3(((N + KPT - 1) / KPT + 31) / 32 * 32), 0, st, scores,   \
                          nparts, scores_out, N, K, has_cls, keep_idx, row_map, rg)
    RS_SEL_CASE(1);
    RS_SEL_CASE(2);
    if (!many) RS_SEL_CASE(5);
    RS_SEL_CASE(16);
    RS_SEL_CASE(32);
#undef RS_SEL_CASE
    return cudaErrorInvalidValue;
}

bool ln_fusable(rs_dtype dtype, int D) { return (size_t)D * dtype_size(dtype) / 16 <= 32 * 4; }

cudaError_t launch_gather(rs_dtype dtype, const void* x, const int32_t* keep_idx, int B, int N, int K,
                          int D, void* x_out, const LnFuse* ln, int sm_count, cudaStream_t st) {
    if (B == 0 || K == 0) return cudaSuccess;
    const int row_vecs = (int)((size_t)D * dtype_size(dtype) / 16);
    const bool norm = ln && ln->gamma;               // else ln, if given, only asks for the row sums of the copy
    if ((norm && !ln_fusable(dtype, D)) || (!x_out && !norm)) return cudaErrorInvalidValue;
    const LnFuse none = {nullptr, nullptr, 0.f, nullptr, nullptr};
    return by_samples(B, K, [&](long long b0, long long rows) {
        const uint4* xb = (const uint4*)x + b0 * N * row_vecs;
        uint4* ob = x_out ? (uint4*)x_out + b0 * K * row_vecs : nullptr;
        LnFuse lb = ln ? *ln : none;
        if (norm) lb.out = (char*)ln->out + (size_t)b0 * K * D * dtype_size(dtype);
        if (lb.stats) lb.stats += 2 * b0 * K;
        const TokenRows src = {keep_idx + b0 * K, (unsigned)K, N};
        if (!norm) return launch_copy(xb, src, rows, row_vecs, ob, lb, sm_count, st);
        const dim3 grid((unsigned)((rows + 7) / 8));
        if (dtype == RS_BF16)
            return launch_pdl(gather_kernel<4, __nv_bfloat16, TokenRows>, grid, dim3(256), 0, st, xb, src, (unsigned)rows, row_vecs, ob, lb);
        return launch_pdl(gather_kernel<4, float, TokenRows>, grid, dim3(256), 0, st, xb, src, (unsigned)rows, row_vecs, ob, lb);
    });
}

int linewise_max_lines() { return kLineMax; }

cudaError_t launch_line_select(const float* scores, int B, int H, int W, int Hk, int Wk, int32_t* keep_rows,
                               int32_t* keep_cols, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    return launch_pdl(line_select_kernel, dim3(B), dim3(2 * kLineMax), 0, st, scores, H, W, Hk, Wk, keep_rows, keep_cols);
}

cudaError_t launch_line_gather(rs_dtype dtype, const void* x, const int32_t* keep_rows, const int32_t* keep_cols, int B, int H,
                               int W, int Hk, int Wk, int D, void* x_out, int sm_count, cudaStream_t st) {
    if (B == 0) return cudaSuccess;
    const int row_vecs = (int)((size_t)D * dtype_size(dtype) / 16);
    const LnFuse none = {nullptr, nullptr, 0.f, nullptr, nullptr};
    return by_samples(B, Hk * Wk, [&](long long b0, long long rows) {
        const GridRows src = {keep_rows + b0 * Hk, keep_cols + b0 * Wk, (unsigned)Hk, (unsigned)Wk, H, W};
        return launch_copy((const uint4*)x + b0 * H * W * row_vecs, src, rows, row_vecs, (uint4*)x_out + b0 * Hk * Wk * row_vecs, none, sm_count, st);
    });
}

}  // namespace rs
