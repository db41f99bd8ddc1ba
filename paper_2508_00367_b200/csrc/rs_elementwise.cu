// HBM-bound row kernels: LayerNorm, the representation-shift score (Sec. 3.2)
// and the residual-add epilogue with the score fused in.  One warp owns one
// token row; rows move as 16-byte vectors, several in flight per lane.
#include <type_traits>

#include "rs_internal.h"
#include "rs_device.cuh"
#include "rs_gemm.cuh"

namespace rs {

namespace {

constexpr int kWarpsPerCta = 8;

// ---------------------------------------------------------------- LayerNorm
// LN of Eq. att / Eq. MLP: mean and biased variance over D, then affine.  One warp per row; the
// row stays in registers as packed 16-byte pieces (unpacked once per pass over it), which keeps
// the kernel at 48 to 64 registers so that four or five CTAs per SM cover the memory latency.
template <typename TI, typename TO, int MAXV>
__global__ void __launch_bounds__(kWarpsPerCta * 32, MAXV <= 4 ? 5 : 4)
layernorm_kernel(const TI* __restrict__ x, const float* __restrict__ gamma,
                 const float* __restrict__ beta, float eps, long long T, int D, TO* __restrict__ out,
                 const int32_t* __restrict__ row_map, const int first, const int32_t* __restrict__ lens, unsigned seq_n) {
    constexpr int VN = Vec16<TI>::N;
    if (!first) grid_dep_launch();
    grid_dep_wait();
    if (first) grid_dep_launch();
    const int lane = threadIdx.x & 31;
    const long long row = (long long)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
    if (row >= T) return;
    if (lens) {                                  // padding that neither the products nor attention read
        const unsigned b = (unsigned)row / seq_n, i = (unsigned)row - b * seq_n;
        if ((int)i >= gemm::rows_needed(lens, b, seq_n)) return;
    }
    const int nvec = D / VN;
    const long long src = row_map ? (long long)row_map[row] : row;
    const uint4* xr = reinterpret_cast<const uint4*>(x + src * D);
    uint4 raw[MAXV];
#pragma unroll
    for (int j = 0; j < MAXV; ++j) {
        const int iv = j * 32 + lane;
        if (iv < nvec) raw[j] = ld_stream(xr + iv);
    }
    layernorm_row<TI, TO, MAXV>(raw, nvec, lane, gamma, beta, eps, D, out + row * D);
}

// The same for fp32 rows of at most 256 values, as LN2 reads them (x', D = 192): half a warp per row, VPL pieces per
// lane, two rows of a half in flight.  A whole warp per row issues as many instructions for 48 pieces as for 64, two
// reductions of five steps each among them, and was bound by that: after the projection of
// 50432 x 192 rows 15.2 -> 10.0 us, 25216 x 128 7.4 -> 5.3, 25216 x 256 8.7 -> 8.4.
constexpr int kNarrowRows = 4 * kWarpsPerCta;            // rows per CTA
template <int VPL>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 4)
layernorm_narrow_kernel(const float* __restrict__ x, const float* __restrict__ gamma, const float* __restrict__ beta, float eps,
                        long long T, int D, __nv_bfloat16* __restrict__ out, const int32_t* __restrict__ lens, unsigned seq_n) {
    grid_dep_launch();
    grid_dep_wait();
    const int l16 = threadIdx.x & 15, nvec = D / 4;
    const long long row0 = (long long)blockIdx.x * kNarrowRows + (threadIdx.x >> 5) * 4 + ((threadIdx.x >> 4) & 1);
    float4 v[2][VPL];
    bool on[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const long long row = row0 + 2 * u;
        on[u] = row < T;
        if (on[u] && lens) {                     // padding that neither the products nor attention read
            const unsigned b = (unsigned)row / seq_n, i = (unsigned)row - b * seq_n;
            on[u] = (int)i < gemm::rows_needed(lens, b, seq_n);
        }
        const float* xr = x + (on[u] ? row : 0) * D;
#pragma unroll
        for (int j = 0; j < VPL; ++j) {
            v[u][j] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (on[u] && j * 16 + l16 < nvec) {
                const uint4 t = ld_stream(reinterpret_cast<const uint4*>(xr) + j * 16 + l16);
                v[u][j] = make_float4(__uint_as_float(t.x), __uint_as_float(t.y), __uint_as_float(t.z), __uint_as_float(t.w));
            }
        }
    }
    float mu[2], rstd[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        float sum = 0.f;
#pragma unroll
        for (int j = 0; j < VPL; ++j) sum += (v[u][j].x + v[u][j].y) + (v[u][j].z + v[u][j].w);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        mu[u] = sum / (float)D;
        float sq = 0.f;
#pragma unroll
        for (int j = 0; j < VPL; ++j)
            if (j * 16 + l16 < nvec) {
                const float a = v[u][j].x - mu[u], b = v[u][j].y - mu[u], c = v[u][j].z - mu[u], d = v[u][j].w - mu[u];
                sq += (a * a + b * b) + (c * c + d * d);
            }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
        rstd[u] = rsqrtf(sq / (float)D + eps);
    }
#pragma unroll
    for (int j = 0; j < VPL; ++j) {
        const int iv = j * 16 + l16;
        if (iv >= nvec) continue;
        const float4 g = __ldg(reinterpret_cast<const float4*>(gamma) + iv), bt = __ldg(reinterpret_cast<const float4*>(beta) + iv);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if (!on[u]) continue;
            const float y[4] = {(v[u][j].x - mu[u]) * rstd[u] * g.x + bt.x, (v[u][j].y - mu[u]) * rstd[u] * g.y + bt.y,
                                (v[u][j].z - mu[u]) * rstd[u] * g.z + bt.z, (v[u][j].w - mu[u]) * rstd[u] * g.w + bt.w};
            store_n<__nv_bfloat16, 4>(out + (row0 + 2 * u) * D + iv * 4, y);
        }
    }
}

// ---------------------------------------------------------------- shift score
// s = D(F(x), x) per token (Sec. 3.2); DIST 0: L2, 1: L1, 2: cosine distance.
// Bound by HBM.  The 16-byte pieces stay packed in registers until they are reduced, so that eight loads per
// lane are in flight at about 48 registers per thread and enough warps fit an SM to cover the HBM latency.
// With HINT `before` is read with an evict-first hint: what the L2 can keep of the two is then `after`, whose kept rows
// the compaction reads next.  Inputs that the L2 holds anyway go without it: 5000 x 256 bf16 2.3 us with, 1.9 without,
// 20000 x 768 7.0 / 6.45 (the cosine's three sums are scheduled better with it, 2.5 / 2.9: always on there).
template <typename T, int DIST> struct ShiftSums {
    float acc = 0.f, aa = 0.f, bb = 0.f;
    __device__ __forceinline__ void add(const uint4& ra, const uint4& rb) {
        constexpr int VN = Vec16<T>::N;
        float va[VN], vb[VN];
        unpack16<T>(ra, va);
        unpack16<T>(rb, vb);
#pragma unroll
        for (int e = 0; e < VN; ++e) {
            if (DIST == 0) { const float d = va[e] - vb[e]; acc = fmaf(d, d, acc); }
            else if (DIST == 1) { acc += fabsf(va[e] - vb[e]); }
            else {
                acc = fmaf(va[e], vb[e], acc);
                aa = fmaf(va[e], va[e], aa);
                bb = fmaf(vb[e], vb[e], bb);
            }
        }
    }
    // over the lanes whose numbers differ below `width` (a power of two)
    __device__ __forceinline__ float finish(int width) {
        for (int o = width >> 1; o > 0; o >>= 1) {
            acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (DIST == 2) {
                aa += __shfl_xor_sync(0xffffffffu, aa, o);
                bb += __shfl_xor_sync(0xffffffffu, bb, o);
            }
        }
        return DIST == 0 ? sqrtf(acc) : DIST == 1 ? acc : 1.f - acc / fmaxf(sqrtf(aa) * sqrtf(bb), 1e-12f);
    }
};

// One warp per token.
template <typename T, int DIST, bool HINT>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 5)
shift_score_kernel(const T* __restrict__ after, const T* __restrict__ before, long long rows, int D,
                   float* __restrict__ scores) {
    constexpr int UNROLL = 4;
    grid_dep_launch();
    grid_dep_wait();
    const uint64_t once = evict_first_policy();
    const int lane = threadIdx.x & 31;
    const long long row = (long long)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int nvec = D / Vec16<T>::N;
    const uint4* a = reinterpret_cast<const uint4*>(after + row * D);
    const uint4* b = reinterpret_cast<const uint4*>(before + row * D);
    ShiftSums<T, DIST> s;
    for (int base = 0; base < nvec; base += 32 * UNROLL) {
        uint4 ra[UNROLL], rb[UNROLL];
#pragma unroll
        for (int u = 0; u < UNROLL; ++u) {
            const int iv = base + u * 32 + lane;
            if (iv < nvec) { ra[u] = ld_stream(a + iv); rb[u] = HINT ? ld_stream(b + iv, once) : ld_stream(b + iv); }
        }
#pragma unroll
        for (int u = 0; u < UNROLL; ++u)
            if (base + u * 32 + lane < nvec) s.add(ra[u], rb[u]);
    }
    const float d = s.finish(32);
    if (lane == 0) scores[row] = d;
}

// Tokens of at most 32 * VPR pieces (VPR 1 or 2), many of them (launch_shift_score): 4 / VPR groups of 32 >> lsh tokens
// side by side per warp, 1 << lsh lanes per token, so that a lane has eight loads in flight here too (a warp per token of 256 bf16 had two:
// 64 x 56 x 56 positions took 56 us = 3.7 TB/s; this takes 36 = 5.7 TB/s).
template <typename T, int DIST, int VPR, bool HINT>
__global__ void __launch_bounds__(kWarpsPerCta * 32, 5)
shift_score_short_kernel(const T* __restrict__ after, const T* __restrict__ before, long long rows, int D, int lsh,
                         float* __restrict__ scores) {
    constexpr int U = 4 / VPR;
    grid_dep_launch();
    grid_dep_wait();
    const uint64_t once = evict_first_policy();
    const int lane = threadIdx.x & 31;
    if (VPR > 1) lsh = 5;
    const int nvec = D / Vec16<T>::N, side = 32 >> lsh, v0 = lane & ((1 << lsh) - 1);
    const long long row0 = ((long long)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5)) * (U * side) + (lane >> lsh);
    uint4 ra[U][VPR], rb[U][VPR];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const long long row = row0 + u * side;
#pragma unroll
        for (int j = 0; j < VPR; ++j) {
            const int iv = j * 32 + v0;
            ra[u][j] = rb[u][j] = make_uint4(0u, 0u, 0u, 0u);
            if (row < rows && iv < nvec) {
                ra[u][j] = ld_stream(reinterpret_cast<const uint4*>(after + row * D) + iv);
                const uint4* p = reinterpret_cast<const uint4*>(before + row * D) + iv;
                rb[u][j] = HINT ? ld_stream(p, once) : ld_stream(p);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const long long row = row0 + u * side;
        ShiftSums<T, DIST> s;
#pragma unroll
        for (int j = 0; j < VPR; ++j) s.add(ra[u][j], rb[u][j]);
        const float d = s.finish(1 << lsh);
        if (v0 == 0 && row < rows) scores[row] = d;
    }
}

// ---------------------------------------------------------------- residual add + score
// x_hat = m + x' and the score of the chosen pair of representations (Sec. 3.3 "Operation
// choice"): MODE 0 |m - x'| (ii), 1 |m|, 2 |SA(LN(x)) - x| = |x' - 2x| (i), 3 |x_hat - x| (iii).
// The score rides on the residual-add pass, which already has the operands in registers.
template <typename TO, typename TX, int MODE>
__global__ void __launch_bounds__(kWarpsPerCta * 32)
residual_score_kernel(const float* __restrict__ m, const float* __restrict__ xp, const TX* __restrict__ x0,
                      long long rows, int D, int dist, TO* __restrict__ x_hat, float* __restrict__ scores) {
    grid_dep_launch();
    grid_dep_wait();
    const int lane = threadIdx.x & 31;
    const long long row = (long long)blockIdx.x * kWarpsPerCta + (threadIdx.x >> 5);
    if (row >= rows) return;
    const int nvec = D / 4;
    float acc = 0.f, uu = 0.f, vv = 0.f;
    for (int iv = lane; iv < nvec; iv += 32) {
        const float4 a = *reinterpret_cast<const float4*>(m + row * D + iv * 4);
        const float4 b = *reinterpret_cast<const float4*>(xp + row * D + iv * 4);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
        float y[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            y[e] = av[e] + bv[e];
            float u, v;                              // the scored pair
            if (MODE == 0) { u = av[e]; v = bv[e]; }
            else if (MODE == 1) { u = y[e]; v = bv[e]; }
            else {
                const float x = to_float(x0[row * D + iv * 4 + e]);
                u = MODE == 2 ? bv[e] - x : y[e];    // SA(LN(x)) = x' - x
                v = x;
            }
            if (dist == RS_DIST_L2) { const float d = u - v; acc = fmaf(d, d, acc); }
            else if (dist == RS_DIST_L1) acc += fabsf(u - v);
            else { acc = fmaf(u, v, acc); uu = fmaf(u, u, uu); vv = fmaf(v, v, vv); }
        }
        store_n<TO, 4>(x_hat + row * D + iv * 4, y);
    }
    acc = warp_sum(acc);
    float sc = dist == RS_DIST_L2 ? sqrtf(acc) : acc;
    if (dist == RS_DIST_COS) {
        uu = warp_sum(uu); vv = warp_sum(vv);
        sc = 1.f - acc / fmaxf(sqrtf(uu) * sqrtf(vv), 1e-12f);
    }
    if (lane == 0 && scores) scores[row] = sc;
}

inline unsigned row_grid(long long rows) { return (unsigned)((rows + kWarpsPerCta - 1) / kWarpsPerCta); }

template <typename TI, typename TO>
cudaError_t ln_dispatch(const void* x, const float* g, const float* b, float eps, long long T, int D,
                        void* out, const int32_t* row_map, bool first, cudaStream_t st, const int32_t* lens, int seq_n) {
    const int nvec = D / Vec16<TI>::N;
    const dim3 grid(row_grid(T)), block(kWarpsPerCta * 32);
    if constexpr (std::is_same<TI, float>::value && std::is_same<TO, __nv_bfloat16>::value) {
        const dim3 narrow((unsigned)((T + kNarrowRows - 1) / kNarrowRows));
#define RS_LN_CASE(VPL)                                                                                                    \
    if (!row_map && !first && nvec <= 16 * VPL)                                                                            \
        return launch_pdl(layernorm_narrow_kernel<VPL>, narrow, block, 0, st, (const float*)x, g, b, eps, T, D,            \
                          (__nv_bfloat16*)out, lens, (unsigned)seq_n)
        RS_LN_CASE(2);
        RS_LN_CASE(3);
        RS_LN_CASE(4);
#undef RS_LN_CASE
    }
    if (nvec <= 32 * 4)
        return launch_pdl(layernorm_kernel<TI, TO, 4>, grid, block, 0, st, (const TI*)x, g, b, eps, T, D, (TO*)out, row_map, (int)first, lens, (unsigned)seq_n);
    else if (nvec <= 32 * 8)
        return launch_pdl(layernorm_kernel<TI, TO, 8>, grid, block, 0, st, (const TI*)x, g, b, eps, T, D, (TO*)out, row_map, (int)first, lens, (unsigned)seq_n);
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_layernorm(rs_dtype in_dtype, rs_dtype out_dtype, const void* x, const float* gamma,
                             const float* beta, float eps, long long T, int D, void* out,
                             const int32_t* row_map, bool first, cudaStream_t st, const int32_t* lens, int seq_n) {
    if (T == 0) return cudaSuccess;
    if (in_dtype == RS_F32 && out_dtype == RS_F32) return ln_dispatch<float, float>(x, gamma, beta, eps, T, D, out, row_map, first, st, lens, seq_n);
    if (in_dtype == RS_F32 && out_dtype == RS_BF16) return ln_dispatch<float, __nv_bfloat16>(x, gamma, beta, eps, T, D, out, row_map, first, st, lens, seq_n);
    if (in_dtype == RS_BF16 && out_dtype == RS_BF16) return ln_dispatch<__nv_bfloat16, __nv_bfloat16>(x, gamma, beta, eps, T, D, out, row_map, first, st, lens, seq_n);
    return ln_dispatch<__nv_bfloat16, float>(x, gamma, beta, eps, T, D, out, row_map, first, st, lens, seq_n);
}

cudaError_t launch_shift_score(rs_dtype dtype, rs_dist dist, long long T, int D, const void* after,
                               const void* before, float* scores, int sm_count, cudaStream_t st) {
    if (T == 0) return cudaSuccess;
    const int nvec = (int)((size_t)D * dtype_size(dtype) / 16);
    int lsh = 0;
    while (lsh < 5 && (1 << lsh) < nvec) ++lsh;
    // Tokens of up to 32 pieces go several to a warp once a warp per token would take more than one round of the 40 warps
    // that an SM holds (two and a half for 17 to 32 pieces, of which a warp takes four one after the other, half of one for one
    // or two pieces); fewer tokens are done sooner with a warp each.  Several to a warp / a warp each, us, L2 of bf16:
    // 1000 x 256 2.3 / 1.8, 6000 x 128 2.5 / 2.7, 6000 x 256 3.1 / 2.7, 12000 x 256 4.1 / 3.9, 16000 x 256 4.3 / 4.7,
    // 40000 x 256 6.6 / 9.4.
    // Of 33 to 64 pieces two go to a warp from ten tokens per SM on (the cosine of 100 x 384 1.8 / 1.6, 2000 x 384 2.1 / 2.3).
    const bool several = nvec <= 32 && 2 * T > 40ll * sm_count * (lsh <= 1 ? 1 : lsh < 5 ? 2 : 5), two = nvec > 32 && nvec <= 64 && T > 10ll * sm_count;
    const long long per_cta = kWarpsPerCta * (several ? 4 * (32 >> lsh) : two ? 2 : 1);
    const bool hint = dist == RS_DIST_COS || 2 * T * D * (long long)dtype_size(dtype) > (64ll << 20);      // half of the L2
    const dim3 grid((unsigned)((T + per_cta - 1) / per_cta)), block(kWarpsPerCta * 32);
#define RS_SCORE_HINT(TT, DD, HH)                                                                                                       \
    return several ? launch_pdl(shift_score_short_kernel<TT, DD, 1, HH>, grid, block, 0, st, (const TT*)after, (const TT*)before, T, D, lsh, scores) \
           : two   ? launch_pdl(shift_score_short_kernel<TT, DD, 2, HH>, grid, block, 0, st, (const TT*)after, (const TT*)before, T, D, lsh, scores) \
                   : launch_pdl(shift_score_kernel<TT, DD, HH>, grid, block, 0, st, (const TT*)after, (const TT*)before, T, D, scores)
#define RS_SCORE_CASE(TT, DD)                                \
    do {                                                     \
        if (hint) RS_SCORE_HINT(TT, DD, true);               \
        RS_SCORE_HINT(TT, DD, (DD == 2));                    \
    } while (0)
    if (dtype == RS_BF16) {
        if (dist == RS_DIST_L2) RS_SCORE_CASE(__nv_bfloat16, 0);
        else if (dist == RS_DIST_L1) RS_SCORE_CASE(__nv_bfloat16, 1);
        else RS_SCORE_CASE(__nv_bfloat16, 2);
    } else {
        if (dist == RS_DIST_L2) RS_SCORE_CASE(float, 0);
        else if (dist == RS_DIST_L1) RS_SCORE_CASE(float, 1);
        else RS_SCORE_CASE(float, 2);
    }
#undef RS_SCORE_CASE
#undef RS_SCORE_HINT
    return cudaGetLastError();
}

cudaError_t launch_residual_score(const float* m, const float* x_prime, const void* x, rs_dtype x_dtype,
                                  long long T, int D, rs_score_mode mode, rs_dist dist, rs_dtype out_dtype,
                                  void* x_hat, float* scores, cudaStream_t st) {
    if (T == 0) return cudaSuccess;
    const dim3 grid(row_grid(T)), block(kWarpsPerCta * 32);
#define RS_RES_CASE(TO, TX, MD)                                                                                  \
    return launch_pdl(residual_score_kernel<TO, TX, MD>, grid, block, 0, st, m, x_prime, (const TX*)x, T, D, (int)dist, (TO*)x_hat, scores)
#define RS_RES_MODE(TO, TX)                                     \
    do {                                                        \
        if (mode == RS_SCORE_MLP) RS_RES_CASE(TO, TX, 0);       \
        else if (mode == RS_SCORE_MLP_DELTA) RS_RES_CASE(TO, TX, 1); \
        else if (mode == RS_SCORE_ATTN) RS_RES_CASE(TO, TX, 2); \
        else RS_RES_CASE(TO, TX, 3);                            \
    } while (0)
    if (out_dtype == RS_BF16) {
        if (x_dtype == RS_BF16) RS_RES_MODE(__nv_bfloat16, __nv_bfloat16); else RS_RES_MODE(__nv_bfloat16, float);
    } else {
        if (x_dtype == RS_BF16) RS_RES_MODE(float, __nv_bfloat16); else RS_RES_MODE(float, float);
    }
#undef RS_RES_MODE
#undef RS_RES_CASE
    return cudaGetLastError();
}

// LayerNorm folded into the projection that follows: one warp per output row n of W [n_out, K].
namespace {
__global__ void __launch_bounds__(256)
ln_fold_prep_kernel(const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias, const float* __restrict__ g,
                    const float* __restrict__ beta, int n_out, int K, __nv_bfloat16* __restrict__ w_out,
                    float* __restrict__ c_out, float* __restrict__ b_out) {
    const int n = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (n >= n_out) return;
    float c = 0.f, bb = 0.f;
    for (int k = lane; k < K; k += 32) {
        const float w = __bfloat162float(W[(size_t)n * K + k]);
        const __nv_bfloat16 ws = __float2bfloat16_rn(w * g[k]);
        w_out[(size_t)n * K + k] = ws;
        c += __bfloat162float(ws);
        bb = fmaf(w, beta[k], bb);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        c += __shfl_xor_sync(0xffffffffu, c, o);
        bb += __shfl_xor_sync(0xffffffffu, bb, o);
    }
    if (lane == 0) {
        c_out[n] = c;
        b_out[n] = bb + (bias ? bias[n] : 0.f);
    }
}
}  // namespace

cudaError_t launch_ln_fold_prep(const void* W, const float* bias, const float* g, const float* beta, int n_out, int K,
                                void* w_out, float* c_out, float* b_out, cudaStream_t st) {
    ln_fold_prep_kernel<<<(n_out + 7) / 8, 256, 0, st>>>((const __nv_bfloat16*)W, bias, g, beta, n_out, K,
                                                         (__nv_bfloat16*)w_out, c_out, b_out);
    return cudaGetLastError();
}

}  // namespace rs
