// bf16 GEMM for few rows on the tensor cores, with the epilogues of rs_gemm_tc.cu (which includes this file):
//     out[M, N] = epilogue(A[M, K] . W[N, K]^T)
// With a few hundred rows the 256-row pair tiles of rs_gemm_tc.cu leave most SMs idle and each of the few busy
// ones walks the whole of K: one image of 197 tokens has 6 pair tiles in its second MLP product, 48 dependent
// K steps long, 17 us for 5 MB of weights.  Here a tile is 128 x 64 and a cluster of `splits` CTAs shares its K,
// so that about every SM streams a slice of the weights; what bounds the kernel then is latency (launch, one
// round trip to memory, a few MMAs, the reduction), not a rate.  The partial accumulators go from tensor memory
// to shared memory and are added in rank order through distributed shared memory, each CTA finishing every
// splits-th row of the tile.
// Weights do not depend on the kernel before this one, so their first slabs are requested before the grid
// dependency is waited for (args.weights_ready: the caller knows that nothing still running writes them).
// Measured: see gemm_small_plan.
#pragma once
#include "rs_internal.h"
#include "rs_gemm.cuh"
#include "rs_device.cuh"
#include "rs_once.h"
#include "rs_tc.cuh"

namespace rs {
namespace few {

// Whether a shape goes to this kernel, and the CTAs that share the K of a tile.
constexpr int kSmallBN = 64;
struct SmallPlan { bool use; int splits; };

namespace {

using namespace tc;
using namespace gemm;

constexpr int BM = 128, BN = kSmallBN, BK = 64, STAGES = 4;
constexpr int kThreads = 256;                          // warp 0: TMA, warp 1: MMA, all eight: reduction and epilogue
constexpr int A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int RED_LD = BN + 4;                         // floats per row of the partial tile: 16-byte accesses of eight rows hit all banks
constexpr int OFF_BAR = STAGES * STAGE_BYTES;          // (the partial tile reuses the stages)
constexpr int OFF_ROWS = OFF_BAR + 256;                // float2 [BM]
constexpr size_t kSmem = (size_t)OFF_ROWS + BM * 8 + 1024 /*alignment slack*/;
static_assert(BM * RED_LD * 4 <= STAGES * STAGE_BYTES, "partial tile");
static_assert(2 * (kSmem + 1024) <= 228 * 1024, "two CTAs per SM");

__device__ __forceinline__ void unpack4(const uint2& t, float (&v)[4]) {
    v[0] = __uint_as_float(t.x << 16); v[1] = __uint_as_float(t.x & 0xffff0000u);
    v[2] = __uint_as_float(t.y << 16); v[3] = __uint_as_float(t.y & 0xffff0000u);
}

template <int EPI, typename OutT>
__global__ void __launch_bounds__(kThreads, 2)
gemm_small_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs args,
                  const int splits, OutT* __restrict__ out, const int weights_ready) {
    constexpr bool SCORE = EPI == EPI_SCORE || EPI == EPI_SCORE_STATS;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* full = reinterpret_cast<uint64_t*>(smem + OFF_BAR);       // [STAGES] operands landed
    uint64_t* empty = full + STAGES;                                    // [STAGES] the MMAs reading the stage retired
    uint64_t* tfull = full + 2 * STAGES;                                // accumulator complete
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(full + 2 * STAGES + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rank = blockIdx.x, n0 = blockIdx.y * BN, m0 = blockIdx.z * BM, num_n = gridDim.y;   // the cluster spans grid dimension x
    const int kblocks = args.K / BK, kb0 = kblocks * rank / splits, nkb = kblocks * (rank + 1) / splits - kb0;

    if (tid == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(tfull, 1);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc(tmem_slot, BN);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    const bool producer = warp == 0 && elect_one();
    auto load_w = [&](int i) { tma_load_2d(smem + (i % STAGES) * STAGE_BYTES + A_BYTES, &tmB, &full[i % STAGES], (kb0 + i) * BK, n0); };
    const int ahead = min(STAGES, nkb);
    if (producer)
        for (int i = 0; i < ahead; ++i) {
            mbar_expect_tx(&full[i], STAGE_BYTES);
            if (weights_ready) load_w(i);
        }
    if (producer && weights_ready)                                      // the rest of this CTA's slice on its way to the L2
        for (int i = ahead; i < nkb; ++i) tma_prefetch_2d(&tmB, (kb0 + i) * BK, n0);
    // four columns at cl of each row this thread finishes; bias and column sums are weights too
    const int cl = (tid & 15) * 4, col = n0 + cl;
    float4 bias = make_float4(0.f, 0.f, 0.f, 0.f), csum = bias;
    auto load_cols = [&]() {
        if (args.bias) bias = *reinterpret_cast<const float4*>(args.bias + col);
        if (EPI == EPI_BIAS_LN) csum = *reinterpret_cast<const float4*>(args.colsum + col);
    };
    if (weights_ready) load_cols();
    grid_dep_launch();
    grid_dep_wait();
    if (!weights_ready) load_cols();

    if (producer) {
        bool ok = true;
        for (int i = 0; i < nkb; ++i) {
            const int s = i % STAGES;
            if (i >= STAGES) {
                if (!mbar_wait(&empty[s], ((i / STAGES) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                mbar_expect_tx(&full[s], STAGE_BYTES);
            }
            if (i >= STAGES || !weights_ready) load_w(i);
            tma_load_2d(smem + s * STAGE_BYTES, &tmA, &full[s], (kb0 + i) * BK, m0);
        }
        (void)ok;      // every copy started here is consumed by the MMAs that tfull, waited for below, stands for
    } else if (warp == 1 && elect_one()) {
        constexpr uint32_t idesc = idesc_bf16(BM, BN, 0, 0);
        bool ok = true;
        for (int i = 0; i < nkb && ok; ++i) {
            const int s = i % STAGES;
            ok = mbar_wait(&full[s], (i / STAGES) & 1u, abort_flag);
            if (!ok) break;
            tc_fence_after();
            const uint64_t da = smem_desc_sw128(smem_u32(smem + s * STAGE_BYTES), 16, 1024);
            const uint64_t db = smem_desc_sw128(smem_u32(smem + s * STAGE_BYTES + A_BYTES), 16, 1024);
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
                mma_ss(tmem_base, da + 2u * k, db + 2u * k, idesc, (i | k) != 0);
            mma_commit(&empty[s]);
        }
        if (ok) mma_commit(tfull);
    }
    __syncwarp();

    // Rows finished by this thread: rank + splits * (pass * 16 + tid / 16); the operands of the first pass are
    // fetched while the accumulator is still being computed.
    const int rl = tid >> 4;
    const int rows_here = (BM - rank + splits - 1) / splits;
    float2* mr = reinterpret_cast<float2*>(smem + OFF_ROWS);             // EPI_BIAS_LN: mean and 1 / deviation of the CTA's rows
    if (EPI == EPI_BIAS_LN) {
        const int i = tid >> 1, row = m0 + rank + splits * i;            // two threads per row
        if (rank + splits * (warp * 16) < BM) {                          // (whole warps)
            const float2* sp = reinterpret_cast<const float2*>(args.stats_in) + (size_t)(row < args.M ? row : 0) * args.stats_parts;
            float s1 = 0.f, s2 = 0.f;
#pragma unroll 8
            for (int p = tid & 1; p < args.stats_parts; p += 2) {
                const float2 t = __ldg(sp + p);
                s1 += t.x; s2 += t.y;
            }
            s1 += __shfl_xor_sync(0xffffffffu, s1, 1);
            s2 += __shfl_xor_sync(0xffffffffu, s2, 1);
            const float inv_d = 1.f / (float)args.K, mu = s1 * inv_d;
            if (!(tid & 1)) mr[i] = make_float2(mu, rsqrtf(fmaxf(s2 * inv_d - mu * mu, 0.f) + args.ln_eps));
        }
    }
    auto fetch_row = [&](int i) {
        float4 res = make_float4(0.f, 0.f, 0.f, 0.f);
        const int row = m0 + rank + splits * i;
        const bool ok = i < rows_here && row < args.M;
        if (EPI == EPI_RESID && ok) {
            const int src = args.row_map ? __ldg(args.row_map + row) : row;
            float v[4];
            unpack4(__ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(args.residual) + (size_t)src * args.N + col)), v);
            res = make_float4(v[0], v[1], v[2], v[3]);
        }
        if (SCORE && ok) res = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(args.residual) + (size_t)row * args.N + col));
        return res;
    };
    float4 cur = fetch_row(rl);

    mbar_wait(tfull, 0, abort_flag);                                     // on a time-out the flag is set: carry on, the status says so
    __syncwarp();
    tc_fence_after();
    float* red = reinterpret_cast<float*>(smem);
    {
        uint32_t r[32];
        const int q = warp & 3, half = warp >> 2;                        // tensor-memory lanes and columns of this warp
        tmem_ld_32x32(tmem_base + ((uint32_t)(q * 32) << 16) + half * 32, r);
        tmem_wait_ld();
        float* dst = red + (q * 32 + lane) * RED_LD + half * 32;
#pragma unroll
        for (int j = 0; j < 32; j += 4)
            *reinterpret_cast<uint4*>(dst + j) = make_uint4(r[j], r[j + 1], r[j + 2], r[j + 3]);
    }
    tc_fence_before();
    if (splits > 1) cluster_sync(); else __syncthreads();

    for (int i = rl; i - rl < rows_here; i += 16) {                      // the same number of passes for every thread
        const float4 res = cur;
        const float2 ln = EPI == EPI_BIAS_LN && i < rows_here ? mr[i] : make_float2(0.f, 0.f);
        if (i + 16 - rl < rows_here) cur = fetch_row(i + 16);
        const int lr = rank + splits * i, row = m0 + lr;
        const bool valid = i < rows_here && row < args.M;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (valid) {
            const float* p = red + lr * RED_LD + cl;
            if (splits == 1) {
                acc = *reinterpret_cast<const float4*>(p);
            } else {
                const uint32_t a = smem_u32(p);
                float4 t[8];                                             // all in flight before the first is added
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    if (s < splits) t[s] = ld_cluster(map_to_cta(a, s));
#pragma unroll
                for (int s = 0; s < 8; ++s)
                    if (s < splits) { acc.x += t[s].x; acc.y += t[s].y; acc.z += t[s].z; acc.w += t[s].w; }
            }
        }
        float v[4] = {acc.x, acc.y, acc.z, acc.w};
        const float bv[4] = {bias.x, bias.y, bias.z, bias.w}, cv[4] = {csum.x, csum.y, csum.z, csum.w};
        const float xs[4] = {res.x, res.y, res.z, res.w};
        float sq = 0.f, sq1 = 0.f, sq2 = 0.f, st1 = 0.f, st2 = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e)
            v[e] = EPI == EPI_BIAS_LN ? fmaf(ln.y, fmaf(-ln.x, cv[e], v[e]), bv[e]) : v[e] + bv[e];
        if (EPI == EPI_BIAS_GELU) {
#pragma unroll
            for (int e = 0; e < 4; ++e) v[e] = gelu_erf(v[e]);
        } else if (EPI == EPI_RESID) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (args.partials) score_acc(args.dist, v[e], xs[e], sq, sq1, sq2);          // (u, v) = (SA(LN(x)), x)
                v[e] += xs[e];
            }
        } else if (SCORE) {
            float x0[4] = {0.f, 0.f, 0.f, 0.f};
            if (args.score_kind == 2 && valid) {
                const int xrow = args.row_map ? __ldg(args.row_map + row) : row;
                unpack4(__ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(args.residual2) + (size_t)xrow * args.N + col)), x0);
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float m = v[e], y = m + xs[e];
                score_acc(args.dist, args.score_kind ? y : m, args.score_kind == 2 ? x0[e] : xs[e], sq, sq1, sq2);
                v[e] = y;
            }
        }
        if (valid) store_n<OutT, 4>(out + (size_t)row * args.N + col, v);
        if (EPI == EPI_SCORE_STATS) {
            // the statistics are those of the values as stored: the next block reads these bf16 numbers
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const float y = to_float(from_float<OutT>(v[e]));
                st1 += y;
                st2 = fmaf(y, y, st2);
            }
        }
        // one set of sums per row of the tile (sixteen lanes)
        if (SCORE || (EPI == EPI_RESID && args.partials)) {
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
                sq += __shfl_xor_sync(0xffffffffu, sq, o);
                if (args.dist == RS_DIST_COS) {
                    sq1 += __shfl_xor_sync(0xffffffffu, sq1, o);
                    sq2 += __shfl_xor_sync(0xffffffffu, sq2, o);
                }
                if (EPI == EPI_SCORE_STATS) {
                    st1 += __shfl_xor_sync(0xffffffffu, st1, o);
                    st2 += __shfl_xor_sync(0xffffffffu, st2, o);
                }
            }
            if (valid && (tid & 15) == 0) {
                const size_t pi = (size_t)row * num_n + blockIdx.y;
                if (args.dist == RS_DIST_COS) {
                    args.partials[3 * pi] = sq; args.partials[3 * pi + 1] = sq1; args.partials[3 * pi + 2] = sq2;
                } else {
                    args.partials[pi] = sq;
                }
                if (EPI == EPI_SCORE_STATS) reinterpret_cast<float2*>(args.stats_out)[pi] = make_float2(st1, st2);
            }
        }
    }
    if (splits > 1) cluster_leave(); else __syncthreads();               // no CTA leaves while a peer reads its partial tile
    if (*abort_flag && tid == 0) atomicExch(args.status, RS_DEV_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem_base, BN);
    }
}

template <int EPI, typename OutT>
cudaError_t launch_one(const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& args, int splits, void* out, bool weights_ready, cudaStream_t st) {
    static PerDeviceOnce attr_once;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = (cudaError_t)attr_once.run(dev, [] {
        return (int)cudaFuncSetAttribute(gemm_small_kernel<EPI, OutT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    });
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)splits, (unsigned)(args.N / BN), (unsigned)((args.M + BM - 1) / BM));
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_small_kernel<EPI, OutT>, tmA, tmB, args, splits, (OutT*)out, (int)weights_ready);
}

}  // namespace

// Which shapes: those with few tiles, where a tile count is what fills the SMs.  Up to 100 tiles of 128 x 64 (two
// thirds of the SMs) this kernel is the faster one whatever K is; past that the pair tiles of rs_gemm_tc.cu are,
// except for a K of a few slabs, where their prologue is what counts and the line lies at 220.  Whole pruned
// forwards of 12 blocks (20 % dropped three times), all products on pair tiles / line at 60 / 100 / 150 / 220
// tiles, us: 1 x 197 x 768 633 / 496 / 492 / 496 / 493; 4 x 197 x 768 651 / 554 / 552 / 561 / 561; 8 x 197 x 768
// 659 / 659 / 648 / 668 / 676; 1 x 577 x 1024 738 / 671 / 653 / 650 / 645; 3 x 577 x 1024 857 / 857 / 857 / 938 / 972;
// 2 x 69 x 1024 709 / 511 / 489 / 486 / 486; 8 x 197 x 192 510 / 446 / 433 / 426 / 424.  The residual epilogue stays at 100 for
// every K: its fp32 rows cost more here than the short prologue gains (few rows / pair tiles, us: 5000 x 256 x 256 7.1 / 5.6,
// 9000 x 192 x 192 7.0 / 6.4, 1576 x 1024 x 64 6.3 / 5.1; six blocks of 47 x 197 x 192 303 / 301, of 25 x 197 x 256 268 / 264).
// Splits: as many as leave three slabs of K to a CTA and 4 / 3 CTAs to an SM (the second MLP product of one image of
// 197 tokens: 20 us unsplit, 12.6 by two, 8.7 by four, 7.3 by eight; 17.4 on pair tiles).
SmallPlan gemm_small_plan(int epi, long long M, int N, int K, int sms) {
    const long long tiles = ((M + BM - 1) / BM) * (N / BN);
    int s = 1;
    while (s < 8 && tiles * (s + 1) <= sms + sms / 3 && K / BK >= 3 * (s + 1)) ++s;
    return {tiles <= (K <= 256 && epi != EPI_RESID ? 220 : 100), s};
}

// tmA: boxes of 128 rows; tmB: boxes of kSmallBN rows; both 64 columns, 128-byte swizzle.
cudaError_t launch_gemm_small(int epi, const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& args, int splits, void* out,
                              rs_dtype out_dtype, bool weights_ready, cudaStream_t st) {
    switch (epi) {
        case EPI_BIAS: return launch_one<EPI_BIAS, __nv_bfloat16>(tmA, tmB, args, splits, out, weights_ready, st);
        case EPI_BIAS_GELU: return launch_one<EPI_BIAS_GELU, __nv_bfloat16>(tmA, tmB, args, splits, out, weights_ready, st);
        case EPI_RESID: return launch_one<EPI_RESID, float>(tmA, tmB, args, splits, out, weights_ready, st);
        case EPI_SCORE:
            if (out_dtype == RS_F32) return launch_one<EPI_SCORE, float>(tmA, tmB, args, splits, out, weights_ready, st);
            return launch_one<EPI_SCORE, __nv_bfloat16>(tmA, tmB, args, splits, out, weights_ready, st);
        case EPI_SCORE_STATS: return launch_one<EPI_SCORE_STATS, __nv_bfloat16>(tmA, tmB, args, splits, out, weights_ready, st);
        case EPI_BIAS_LN: return launch_one<EPI_BIAS_LN, __nv_bfloat16>(tmA, tmB, args, splits, out, weights_ready, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace few
}  // namespace rs
