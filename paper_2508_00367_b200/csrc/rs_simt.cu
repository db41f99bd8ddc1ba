// fp32-FMA contraction path: a tiled GEMM with the block's epilogues and a streaming-softmax attention.  It
// serves the RS_F32 storage type (tensor cores have no fp32 x fp32 mode with fp32 products), bf16 shapes
// outside the tensor-core kernels, and is the on-device cross-check for the tcgen05 kernels.
// Both are bound by the FMA pipes (128 fp32 FMAs per cycle and SM).  Products are issued as packed pairs
// (fma.rn.f32x2) along the contracted dimension: a pair's two halves are the sums over the even and the odd
// terms, both operands come out of shared memory as 16-byte pieces ready for it, and half the issue slots
// are left for the loads.
#include <math.h>

#include "rs_internal.h"
#include "rs_attn.cuh"
#include "rs_device.cuh"
#include "rs_once.h"
#include "rs_tc.cuh"

namespace rs {

namespace {

using attn::fadd2;
using attn::ffma2;
using attn::pack2;
using attn::unpack2;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Four consecutive values of T as two packed fp32 pairs.
struct Quad { uint64_t lo, hi; };
__device__ __forceinline__ Quad load_quad(const float* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return {v.x, v.y};
}
__device__ __forceinline__ Quad load_quad(const __nv_bfloat16* p) {
    const uint2 v = *reinterpret_cast<const uint2*>(p);
    return {pack2(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u)),
            pack2(__uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u))};
}
__device__ __forceinline__ float pair_sum(uint64_t v) {
    float a, b;
    unpack2(v, a, b);
    return a + b;
}

// ---------------------------------------------------------------- GEMM
// out[M, N] = act(A[M, K] . W[N, K]^T + bias) + residual.  A warp owns a 32 x 8 NJ patch of the output (8 x NJ
// per thread), a CTA WM x WN patches with WK warps to a patch that split the K of every slab, and a cluster of
// S CTAs may split K further (small outputs would leave most SMs idle); the WK * S partial patches are added in a
// fixed order at the end, through (distributed) shared memory.  Slabs of 32 along K come in by 16-byte cp.async,
// four to seven stages deep; rows are padded by 16 bytes, which keeps the 16-byte reads of eight rows apart free
// of bank conflicts.
template <typename T, int WM, int WN, int WK, int NJ> struct SimtCfg {
    static constexpr int TM = 32 * WM, TN = 8 * NJ * WN, THREADS = 32 * WM * WN * WK;
    static constexpr int BK = 32;
    static constexpr int ROW_BYTES = BK * (int)sizeof(T) + 16, STAGE_BYTES = (TM + TN) * ROW_BYTES;
    static constexpr int STAGES = STAGE_BYTES <= 10240 ? 7 : STAGE_BYTES <= 20480 ? 5 : 4;
    static constexpr int RED_LD = TN + 8, RED_BYTES = WK * TM * RED_LD * 4;
    static constexpr int SMEM = STAGES * STAGE_BYTES > RED_BYTES ? STAGES * STAGE_BYTES : RED_BYTES;
};

struct SimtArgs {
    const void *A, *W;
    const float* bias;
    const void* residual;
    void* out;
    long long M;
    int N, K, gelu, res_bf16, out_bf16, splits;
    int weights_ready;       // W may be read before the kernel waits for its predecessor (no earlier kernel still running writes it)
};

template <typename T, int WM, int WN, int WK, int NJ>
__global__ void __launch_bounds__(SimtCfg<T, WM, WN, WK, NJ>::THREADS, 2)
gemm_simt_kernel(const SimtArgs args) {
    using C = SimtCfg<T, WM, WN, WK, NJ>;
    constexpr int CHUNK = 16 / (int)sizeof(T), CPR = C::BK / CHUNK;      // values per 16 bytes, 16-byte pieces per row
    extern __shared__ __align__(16) uint8_t smem[];
    grid_dep_launch();
    if (!args.weights_ready) grid_dep_wait();
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wk = warp / (WM * WN), wm = (warp % (WM * WN)) / WN, wn = warp % WN;
    const int ty = lane >> 3, tx = lane & 7;
    // grid dimension x: the clusters of `splits` (a power of two) along N -- x alone has room for every N --, y: along M
    const int rank = blockIdx.x & (args.splits - 1);
    const long long m0 = (long long)blockIdx.y * C::TM;
    const int n0 = (blockIdx.x >> (__ffs(args.splits) - 1)) * C::TN;
    const T* A = reinterpret_cast<const T*>(args.A);
    const T* W = reinterpret_cast<const T*>(args.W);
    const int K = args.K, slabs = (K + C::BK - 1) / C::BK;
    const int s_begin = (int)((long long)slabs * rank / args.splits), s_end = (int)((long long)slabs * (rank + 1) / args.splits);

    // a thread copies the same 16-byte column of every ROWS_PER_PASS-th row of a slab
    constexpr int ROWS_PER_PASS = C::THREADS / CPR;
    static_assert(C::THREADS % CPR == 0 && C::TM % ROWS_PER_PASS == 0 && C::TN % ROWS_PER_PASS == 0, "copy pattern");
    const int fr = tid / CPR, fc = tid - fr * CPR;
    const T* pa = A + (m0 + fr) * K + fc * CHUNK;
    const T* pw = W + (long long)(n0 + fr) * K + fc * CHUNK;
    const long long row_step = (long long)ROWS_PER_PASS * K;
    const uint32_t dst0 = tc::smem_u32(smem) + fr * C::ROW_BYTES + fc * 16;
    auto fetch_a = [&](int slab, int stage) {
        const uint32_t dst = dst0 + stage * C::STAGE_BYTES;
        const int k0 = slab * C::BK;
        const bool kok = k0 + fc * CHUNK < K;
        const T* a = pa + k0;
#pragma unroll
        for (int i = 0; i < C::TM / ROWS_PER_PASS; ++i, a += row_step) {
            const bool ok = kok && m0 + fr + i * ROWS_PER_PASS < args.M;
            cp_async16(dst + i * ROWS_PER_PASS * C::ROW_BYTES, ok ? a : A, ok);
        }
    };
    auto fetch_w = [&](int slab, int stage) {
        const uint32_t dst = dst0 + stage * C::STAGE_BYTES;
        const int k0 = slab * C::BK;
        const bool kok = k0 + fc * CHUNK < K;
        const T* w = pw + k0;
#pragma unroll
        for (int i = 0; i < C::TN / ROWS_PER_PASS; ++i, w += row_step) {
            const bool ok = kok && n0 + fr + i * ROWS_PER_PASS < args.N;
            cp_async16(dst + (C::TM + i * ROWS_PER_PASS) * C::ROW_BYTES, ok ? w : W, ok);
        }
    };

    uint64_t acc[8][NJ];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j) acc[i][j] = 0ull;

    // Weights do not depend on the kernel before this one: the first slabs' are requested before it is waited for (they belong to
    // the first group, which is waited for as a whole).  The four products of a ViT-S block, 2 x 197: 92.8 -> 89.5 us for the block.
#pragma unroll
    for (int s = 0; s < C::STAGES - 1; ++s)
        if (s_begin + s < s_end) fetch_w(s_begin + s, s);
    if (args.weights_ready) grid_dep_wait();
#pragma unroll
    for (int s = 0; s < C::STAGES - 1; ++s) {
        if (s_begin + s < s_end) fetch_a(s_begin + s, s);
        cp_async_commit();
    }
    int stage = 0;
    for (int slab = s_begin; slab < s_end; ++slab) {
        cp_async_wait<C::STAGES - 2>();
        __syncthreads();                                                 // the slab landed, and everyone is done with the stage refilled next
        const int ahead = stage + C::STAGES - 1;
        if (slab + C::STAGES - 1 < s_end) {
            const int to = ahead >= C::STAGES ? ahead - C::STAGES : ahead;
            fetch_a(slab + C::STAGES - 1, to);
            fetch_w(slab + C::STAGES - 1, to);
        }
        cp_async_commit();
        const uint8_t* base = smem + stage * C::STAGE_BYTES;
        const uint8_t* arow = base + (wm * 32 + ty) * C::ROW_BYTES + wk * (C::BK / WK) * (int)sizeof(T);
        const uint8_t* brow = base + (C::TM + wn * (8 * NJ) + tx) * C::ROW_BYTES + wk * (C::BK / WK) * (int)sizeof(T);
#pragma unroll
        for (int k = 0; k < C::BK / WK; k += 4) {
            Quad b[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) b[j] = load_quad(reinterpret_cast<const T*>(brow + 8 * j * C::ROW_BYTES) + k);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const Quad a = load_quad(reinterpret_cast<const T*>(arow + 4 * i * C::ROW_BYTES) + k);
#pragma unroll
                for (int j = 0; j < NJ; ++j) acc[i][j] = ffma2(a.hi, b[j].hi, ffma2(a.lo, b[j].lo, acc[i][j]));
            }
        }
        if (++stage == C::STAGES) stage = 0;
    }
    cp_async_wait<0>();
    __syncthreads();                                                     // the stages become the partial patches

    float* red = reinterpret_cast<float*>(smem);
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < NJ; ++j)
            red[(wk * C::TM + wm * 32 + ty + 4 * i) * C::RED_LD + wn * (8 * NJ) + tx + 8 * j] = pair_sum(acc[i][j]);
    if (args.splits > 1) tc::cluster_sync(); else __syncthreads();

    // each CTA of the cluster finishes its share of the tile's rows
    const int rows = C::TM / args.splits, r0 = rank * rows;
    for (int e = tid; e < rows * (C::TN / 4); e += C::THREADS) {
        const int r = r0 + e / (C::TN / 4), c = (e % (C::TN / 4)) * 4;
        const long long gm = m0 + r;
        const int gn = n0 + c;
        if (gm >= args.M || gn >= args.N) continue;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int s = 0; s < args.splits; ++s)
#pragma unroll
            for (int w = 0; w < WK; ++w) {
                const float* p = red + (w * C::TM + r) * C::RED_LD + c;
                const float4 t = args.splits > 1 ? tc::ld_cluster(tc::map_to_cta(tc::smem_u32(p), s)) : *reinterpret_cast<const float4*>(p);
                v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
            }
        if (args.bias) {
            const float4 t = __ldg(reinterpret_cast<const float4*>(args.bias + gn));
            v.x += t.x; v.y += t.y; v.z += t.z; v.w += t.w;
        }
        float o[4] = {v.x, v.y, v.z, v.w};
        if (args.gelu) {
#pragma unroll
            for (int x = 0; x < 4; ++x) o[x] = 0.5f * o[x] * (1.f + erff(o[x] * 0.70710678118654752f));
        }
        const long long at = gm * args.N + gn;
        if (args.residual) {
            if (args.res_bf16) {
                const uint2 t = *reinterpret_cast<const uint2*>((const __nv_bfloat16*)args.residual + at);
                o[0] += __uint_as_float(t.x << 16); o[1] += __uint_as_float(t.x & 0xffff0000u);
                o[2] += __uint_as_float(t.y << 16); o[3] += __uint_as_float(t.y & 0xffff0000u);
            } else {
                const float4 t = *reinterpret_cast<const float4*>((const float*)args.residual + at);
                o[0] += t.x; o[1] += t.y; o[2] += t.z; o[3] += t.w;
            }
        }
        if (args.out_bf16) store_n<__nv_bfloat16, 4>((__nv_bfloat16*)args.out + at, o);
        else store_n<float, 4>((float*)args.out + at, o);
    }
    if (args.splits > 1) tc::cluster_leave();                            // no CTA leaves while a peer reads its patches
}

template <typename T, int WM, int WN, int WK, int NJ>
cudaError_t launch_simt(const SimtArgs& args, cudaStream_t st) {
    using C = SimtCfg<T, WM, WN, WK, NJ>;
    static PerDeviceOnce attr_once;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = (cudaError_t)attr_once.run(dev, [] {
        return (int)cudaFuncSetAttribute(gemm_simt_kernel<T, WM, WN, WK, NJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    });
    if (e != cudaSuccess) return e;
    const long long mt = (args.M + C::TM - 1) / C::TM;
    if (mt > 65535) return cudaErrorInvalidValue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)args.splits * (unsigned)(((long long)args.N + C::TN - 1) / C::TN), (unsigned)mt, 1);
    cfg.blockDim = dim3(C::THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)args.splits;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_simt_kernel<T, WM, WN, WK, NJ>, args);
}

// Tile and cluster split.  What a CTA's FMAs take at full rate is known; the rate an SM reaches depends on how many
// CTAs it holds (one warp per scheduler issues a third of the time), the work per SM on the CTA count and its
// rounding, and each resident round adds about a microsecond (pipeline fill, reduction, epilogue).  Rates and
// constants fitted to a sweep of fifteen shapes from 50 x 192 x 192 to 12000 x 4096 x 1024.
// Measured against 64 x 64 tiles with 4 x 4 per thread and unpipelined loads: 394 x 1152 x 384 91 -> 15.5 us;
// 12000 x 4096 x 1024 runs at 47 TFLOP/s.
struct SimtPick { int cfg, splits; };
SimtPick simt_pick(long long M, int N, int K, int sms) {
    static const struct { int tm, tn, resident; double rate[3]; } cfg[4] = {
        {64, 128, 2, {0.31, 0.60, 0.60}}, {64, 64, 2, {0.31, 0.60, 0.60}}, {32, 32, 3, {0.19, 0.38, 0.56}}, {128, 64, 2, {0.32, 0.58, 0.58}}};
    SimtPick best = {3, 1};                              // the tallest tile: any M up to 2^23 fits its grid
    double best_t = -1.0;
    const int slabs = (K + 31) / 32;
    for (int c = 0; c < 4; ++c) {
        if ((M + cfg[c].tm - 1) / cfg[c].tm > 65535) continue;
        const double tiles = (double)((M + cfg[c].tm - 1) / cfg[c].tm) * ((N + cfg[c].tn - 1) / cfg[c].tn);
        for (int s = 1; s <= 4 && (s == 1 || slabs >= 3 * s); s *= 2) {
            const double load = tiles * s / sms, per = ceil(load);
            const int held = per < cfg[c].resident ? (int)per : cfg[c].resident;
            const double us = (double)cfg[c].tm * cfg[c].tn * ((slabs + s - 1) / s) * 32 / (128.0 * 1900.0) / cfg[c].rate[held - 1];
            const double t = us * 0.5 * (load + per) + ceil(per / cfg[c].resident) * (s > 1 ? 1.5 : 1.0);
            if (best_t < 0 || t < best_t) { best_t = t; best = {c, s}; }
        }
    }
    return best;
}

template <typename T> cudaError_t dispatch_simt(SimtArgs& args, int sms, cudaStream_t st) {
    const SimtPick p = simt_pick(args.M, args.N, args.K, sms);
    args.splits = p.splits;
    switch (p.cfg) {
        case 0: return launch_simt<T, 2, 2, 1, 8>(args, st);
        case 1: return launch_simt<T, 2, 1, 2, 8>(args, st);
        case 2: return launch_simt<T, 1, 1, 4, 4>(args, st);
        default: return launch_simt<T, 4, 2, 1, 4>(args, st);
    }
}

// ---------------------------------------------------------------- attention
// Eq. sa with a running max / running sum (no N x N buffer).  A CTA takes 32 query rows of one (sample, head), eight
// to a warp (16 and four where that leaves SMs short of CTAs); keys and values come through shared memory 64 at a
// time, two stages.  Per key tile a lane computes the scores of its two keys against the warp's rows (pairs along
// the head dimension), the warp agrees on the rows' maxima, and the probabilities go through the warp's own shared
// memory, key-major, to the second product: there a lane owns four output columns and every other key (pairs along
// the query rows).
// (One thread per query row with q and o in registers, the form this replaces, kept 24 of 148 SMs busy at 2 x 197
// tokens of six heads and took 92 us.)
// GROUPS: with a CTA or two to an SM a warp or two per scheduler walk through the key tiles one after the other, a chain of loads,
// shuffles and exponentials each.  Then GROUPS times four warps share a CTA's rows, each group every GROUPS-th key tile in buffers of its own;
// the groups' maxima, sums and outputs are merged through shared memory.
// A first key tile may hold scores of -infinity only: the maximum starts from the lowest finite number, which makes all of its weights zeros.
constexpr int AKV = 64, AWARPS = 4, ADH = 64;
constexpr int KLD = ADH + 4;                                  // padded row length (floats): conflict-free 16-byte accesses
constexpr int ATT_KV_FLOATS = AKV * KLD + AKV * ADH;          // one stage: keys (padded), values
constexpr int OLD = ADH + 4;                                  // floats per row of a group's result: output, maximum, sum
template <int AROWS, int GROUPS> struct AttnSimt {
    static constexpr int AQ = AWARPS * AROWS, PLD = AROWS == 8 ? 12 : 4, STAGES = GROUPS > 1 ? 1 : 2, THREADS = 32 * AWARPS * GROUPS;
    static constexpr int SMEM = (AQ * ADH + GROUPS * (STAGES * ATT_KV_FLOATS + AWARPS * AKV * PLD)) * 4;
    static_assert(AQ * OLD <= ATT_KV_FLOATS && SMEM <= 227 * 1024, "a group's result takes the place of its keys");
};

template <typename T, int AROWS, int GROUPS>
__global__ void __launch_bounds__((AttnSimt<AROWS, GROUPS>::THREADS), GROUPS == 1 ? 2 : 1)
attn_simt_kernel(const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                 T* __restrict__ out, int N, int H, float scale, long long qb, long long qr,
                 long long qh, long long kb, long long kr, long long kh, long long vb, long long vr,
                 long long vh) {
    using A = AttnSimt<AROWS, GROUPS>;
    constexpr int AQ = A::AQ, PLD = A::PLD, STAGES = A::STAGES;
    extern __shared__ __align__(16) float sm[];
    grid_dep_launch();
    grid_dep_wait();
    const int group = GROUPS == 1 ? 0 : threadIdx.x / (32 * AWARPS);
    const int tid = threadIdx.x - group * 32 * AWARPS, warp = tid >> 5, lane = tid & 31;     // within the group
    float* Qs = sm;                                            // [AQ][64], scaled
    float* const KV0 = sm + AQ * ADH;                          // a group: [stages][keys 64 x 68 | values 64 x 64]
    float* KV = KV0 + group * STAGES * ATT_KV_FLOATS;
    float* Ps = KV0 + GROUPS * STAGES * ATT_KV_FLOATS + (group * AWARPS + warp) * AKV * PLD;     // [64 keys][AROWS] of this warp
    auto group_sync = [&]() {
        if (GROUPS == 1) __syncthreads();
        else tc::named_barrier(1 + group, 32 * AWARPS);
    };
    const int h = blockIdx.y, b = blockIdx.z, q0 = blockIdx.x * AQ;
    const T* kp = k + b * kb + h * kh;
    const T* vp = v + b * vb + h * vh;
    const int tiles = (N + AKV - 1) / AKV;

    // rows past N are zeros: keys there are masked below, their values meet zero weights
    auto fetch = [&](int t, int stage) {
        float* Ks = KV + stage * ATT_KV_FLOATS;
        float* Vs = Ks + AKV * KLD;
        for (int e = tid; e < AKV * (ADH / 4); e += 32 * AWARPS) {
            const int r = e / (ADH / 4), c = (e % (ADH / 4)) * 4, j = t * AKV + r;
            const bool ok = j < N;
            const T* ks = kp + (long long)(ok ? j : 0) * kr + c;
            const T* vs = vp + (long long)(ok ? j : 0) * vr + c;
            if constexpr (sizeof(T) == 4) {
                cp_async16(tc::smem_u32(Ks + r * KLD + c), ks, ok);
                cp_async16(tc::smem_u32(Vs + r * ADH + c), vs, ok);
            } else {
                const Quad kq = load_quad(ks), vq = load_quad(vs);
                *reinterpret_cast<ulonglong2*>(Ks + r * KLD + c) = ok ? make_ulonglong2(kq.lo, kq.hi) : make_ulonglong2(0, 0);
                *reinterpret_cast<ulonglong2*>(Vs + r * ADH + c) = ok ? make_ulonglong2(vq.lo, vq.hi) : make_ulonglong2(0, 0);
            }
        }
    };
    if (group < tiles) fetch(group, 0);
    cp_async_commit();
    for (int e = threadIdx.x; e < AQ * ADH; e += A::THREADS) {
        const int r = e / ADH, c = e % ADH, i = q0 + r;
        Qs[e] = i < N ? to_float(q[b * qb + (long long)i * qr + h * qh + c]) * scale : 0.f;
    }

    float m[AROWS], l[AROWS];                                  // running maximum (the warp's), this lane's share of the sum
    uint64_t o[AROWS / 2][4];                                  // rows (2p, 2p + 1) x columns 4 (lane & 15) .. + 3, keys of this half warp
#pragma unroll
    for (int r = 0; r < AROWS; ++r) { m[r] = attn::kLowest; l[r] = 0.f; }
#pragma unroll
    for (int p = 0; p < AROWS / 2; ++p)
#pragma unroll
        for (int c = 0; c < 4; ++c) o[p][c] = 0ull;

    if (GROUPS > 1) __syncthreads();                           // Q is there
    for (int t = group, n = 0; t < tiles; t += GROUPS, ++n) {
        const int stage = STAGES == 1 ? 0 : n & 1;
        if (STAGES > 1) {
            if (t + GROUPS < tiles) fetch(t + GROUPS, stage ^ 1);
        } else if (n) {
            fetch(t, 0);
        }
        cp_async_commit();
        cp_async_wait<STAGES - 1>();
        group_sync();
        const float* Ks = KV + stage * ATT_KV_FLOATS;
        const float* Vs = Ks + AKV * KLD;
        const int valid = min(AKV, N - t * AKV);

        // scores of keys lane and lane + 32 against the warp's rows
        uint64_t s2[AROWS][2];
#pragma unroll
        for (int r = 0; r < AROWS; ++r) s2[r][0] = s2[r][1] = 0ull;
#pragma unroll 4
        for (int c = 0; c < ADH; c += 4) {
            const Quad k0 = load_quad(Ks + lane * KLD + c), k1 = load_quad(Ks + (lane + 32) * KLD + c);
#pragma unroll
            for (int r = 0; r < AROWS; ++r) {
                const Quad qv = load_quad(Qs + (warp * AROWS + r) * ADH + c);
                s2[r][0] = ffma2(qv.hi, k0.hi, ffma2(qv.lo, k0.lo, s2[r][0]));
                s2[r][1] = ffma2(qv.hi, k1.hi, ffma2(qv.lo, k1.lo, s2[r][1]));
            }
        }
        float p0[AROWS], p1[AROWS], corr[AROWS];
        bool raised = false;
#pragma unroll
        for (int r = 0; r < AROWS; ++r) {
            p0[r] = lane < valid ? pair_sum(s2[r][0]) : -INFINITY;
            p1[r] = lane + 32 < valid ? pair_sum(s2[r][1]) : -INFINITY;
            const float mx = fmaxf(m[r], warp_max(fmaxf(p0[r], p1[r])));
            corr[r] = expf(m[r] - mx);                         // 0 on the first tile
            raised |= mx > m[r];
            m[r] = mx;
            p0[r] = expf(p0[r] - mx);
            p1[r] = expf(p1[r] - mx);
            l[r] = l[r] * corr[r] + (p0[r] + p1[r]);
        }
        if (raised) {                                          // the same for the whole warp
#pragma unroll
            for (int p = 0; p < AROWS / 2; ++p) {
                const uint64_t cc = pack2(corr[2 * p], corr[2 * p + 1]);
#pragma unroll
                for (int c = 0; c < 4; ++c) o[p][c] = ffma2(o[p][c], cc, 0ull);
            }
        }
        __syncwarp();                                          // the warp is done with the last tile's probabilities
#pragma unroll
        for (int r = 0; r < AROWS; r += 4) {
            *reinterpret_cast<float4*>(Ps + lane * PLD + r) = make_float4(p0[r], p0[r + 1], p0[r + 2], p0[r + 3]);
            *reinterpret_cast<float4*>(Ps + (lane + 32) * PLD + r) = make_float4(p1[r], p1[r + 1], p1[r + 2], p1[r + 3]);
        }
        __syncwarp();
        const int half = lane >> 4, col = (lane & 15) * 4;
#pragma unroll 4
        for (int j = half; j < valid + half; j += 2) {          // past an odd `valid`: weight 0, a value of zeros
            const float4 vv = *reinterpret_cast<const float4*>(Vs + j * ADH + col);
            const uint64_t vd[4] = {pack2(vv.x, vv.x), pack2(vv.y, vv.y), pack2(vv.z, vv.z), pack2(vv.w, vv.w)};
#pragma unroll
            for (int p = 0; p < AROWS / 2; p += 2) {
                const Quad pq = load_quad(Ps + j * PLD + 2 * p);
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    o[p][c] = ffma2(pq.lo, vd[c], o[p][c]);
                    o[p + 1][c] = ffma2(pq.hi, vd[c], o[p + 1][c]);
                }
            }
        }
        group_sync();                                          // everyone is done with this stage
    }
#pragma unroll
    for (int r = 0; r < AROWS; ++r) l[r] = warp_sum(l[r]);
    const int half = lane >> 4, col = (lane & 15) * 4;
    float scale_o[AROWS];                                      // what this group's output is multiplied by
    if (GROUPS > 1) {
        // a row's result, [64 outputs | maximum, sum], where the group's keys were
        auto result = [&](int g, int r) { return KV0 + g * STAGES * ATT_KV_FLOATS + (warp * AROWS + r) * OLD; };
        if (lane == 0) {
#pragma unroll
            for (int r = 0; r < AROWS; ++r) *reinterpret_cast<float2*>(result(group, r) + ADH) = make_float2(m[r], l[r]);
        }
        if (group) {
#pragma unroll
            for (int p = 0; p < AROWS / 2; ++p) {
                float ra[4], rb[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) {
                    o[p][c] = fadd2(o[p][c], __shfl_xor_sync(0xffffffffu, o[p][c], 16));
                    unpack2(o[p][c], ra[c], rb[c]);
                }
                *reinterpret_cast<float4*>(result(group, 2 * p + half) + col) = half ? make_float4(rb[0], rb[1], rb[2], rb[3]) : make_float4(ra[0], ra[1], ra[2], ra[3]);
            }
        }
        __syncthreads();
        if (group) return;
#pragma unroll
        for (int r = 0; r < AROWS; ++r) {
            float2 ml[GROUPS];
            float mx = m[r];
#pragma unroll
            for (int g = 1; g < GROUPS; ++g) {
                ml[g] = *reinterpret_cast<const float2*>(result(g, r) + ADH);
                mx = fmaxf(mx, ml[g].x);
            }
            scale_o[r] = expf(m[r] - mx);
            float sum = scale_o[r] * l[r];
#pragma unroll
            for (int g = 1; g < GROUPS; ++g) sum += expf(ml[g].x - mx) * ml[g].y;
            const float inv = 1.f / sum;
            scale_o[r] *= inv;
            l[r] = inv;
            m[r] = mx;
        }
    } else {
#pragma unroll
        for (int r = 0; r < AROWS; ++r) scale_o[r] = 1.f / l[r];
    }
#pragma unroll
    for (int p = 0; p < AROWS / 2; ++p) {
        float ra[4], rb[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            o[p][c] = fadd2(o[p][c], __shfl_xor_sync(0xffffffffu, o[p][c], 16));
            unpack2(o[p][c], ra[c], rb[c]);
        }
        // the lower half warp stores row 2p, the upper row 2p + 1
        const int i = q0 + warp * AROWS + 2 * p + half;
        const float f = half ? scale_o[2 * p + 1] : scale_o[2 * p];
        float w[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) w[c] = (half ? rb[c] : ra[c]) * f;
        if (GROUPS > 1) {
            const float mx = half ? m[2 * p + 1] : m[2 * p], inv = half ? l[2 * p + 1] : l[2 * p];
#pragma unroll
            for (int g = 1; g < GROUPS; ++g) {
                const float* rp = KV0 + g * STAGES * ATT_KV_FLOATS + (warp * AROWS + 2 * p + half) * OLD;
                const float fg = expf(rp[ADH] - mx) * inv;
                const float4 og = *reinterpret_cast<const float4*>(rp + col);
                w[0] = fmaf(og.x, fg, w[0]); w[1] = fmaf(og.y, fg, w[1]); w[2] = fmaf(og.z, fg, w[2]); w[3] = fmaf(og.w, fg, w[3]);
            }
        }
        if (i < N) store_n<T, 4>(out + ((long long)b * N + i) * ((long long)H * ADH) + h * ADH + col, w);
    }
}

template <typename T, int AROWS, int GROUPS>
cudaError_t attn_launch(const rs_attn_desc& d, const void* q, const void* k, const void* v, void* out, cudaStream_t st) {
    using A = AttnSimt<AROWS, GROUPS>;
    static PerDeviceOnce attr_once;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = (cudaError_t)attr_once.run(dev, [] {
        return (int)cudaFuncSetAttribute(attn_simt_kernel<T, AROWS, GROUPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, A::SMEM);
    });
    if (e != cudaSuccess) return e;
    const float scale = d.scale != 0.f ? d.scale : 1.f / sqrtf((float)d.head_dim);
    const dim3 grid((d.N + A::AQ - 1) / A::AQ, d.H, d.B);
    return launch_pdl(attn_simt_kernel<T, AROWS, GROUPS>, grid, dim3(A::THREADS), A::SMEM, st, (const T*)q, (const T*)k, (const T*)v, (T*)out, d.N, d.H,
                      scale, d.q_batch_stride, d.q_row_stride, d.q_head_stride, d.k_batch_stride, d.k_row_stride,
                      d.k_head_stride, d.v_batch_stride, d.v_row_stride, d.v_head_stride);
}

template <typename T>
cudaError_t attn_dispatch(const rs_attn_desc& d, const void* q, const void* k, const void* v, void* out, int sms, cudaStream_t st) {
    const long long ctas32 = (long long)((d.N + 31) / 32) * d.H * d.B, ctas16 = (long long)((d.N + 15) / 16) * d.H * d.B;
    const int tiles = (d.N + AKV - 1) / AKV;
    // Four groups where the CTAs fit the SMs one to each, of sixteen rows or else of 32.  One group / four, us: 1 x 3 x 65 6.2 / 5.2, 1 x 3 x 130 8.1 / 6.4,
    // 1 x 3 x 577 21.3 / 17.3, 2 x 6 x 197 (84 CTAs of 32 rows) 17.0 / 12.4; with more CTAs they lose: 4 x 6 x 197 18.2 / 23.1, 1 x 12 x 577 40.6 / 50.6.
    // Two groups: 15.6 at 2 x 6 x 197.  Error against 64 bits 2.50e-7 -> 2.09e-7 there, 3.53e-7 -> 2.43e-7 at 1 x 3 x 577 (shorter sums).
    if (tiles >= 2 && ctas16 <= sms) return attn_launch<T, 4, 4>(d, q, k, v, out, st);
    if (tiles >= 3 && ctas32 <= sms) return attn_launch<T, 8, 4>(d, q, k, v, out, st);
    return ctas32 < 2ll * sms ? attn_launch<T, 4, 1>(d, q, k, v, out, st) : attn_launch<T, 8, 1>(d, q, k, v, out, st);
}

}  // namespace

cudaError_t launch_gemm_simt(rs_dtype in_dtype, const void* A, const void* W, const float* bias,
                             int gelu, const void* residual, rs_dtype res_dtype, void* out,
                             rs_dtype out_dtype, long long M, int N, int K, int sm_count, cudaStream_t st, bool weights_ready) {
    if (M == 0 || N == 0) return cudaSuccess;
    SimtArgs args = {A, W, bias, residual, out, M, N, K, gelu, res_dtype == RS_BF16, out_dtype == RS_BF16, 1, weights_ready ? 1 : 0};
    return in_dtype == RS_BF16 ? dispatch_simt<__nv_bfloat16>(args, sm_count, st) : dispatch_simt<float>(args, sm_count, st);
}

cudaError_t launch_attn_simt(const rs_attn_desc& d, const void* q, const void* k, const void* v,
                             void* out, int sm_count, cudaStream_t st) {
    if (d.B == 0 || d.N == 0) return cudaSuccess;
    return d.dtype == RS_BF16 ? attn_dispatch<__nv_bfloat16>(d, q, k, v, out, sm_count, st)
                              : attn_dispatch<float>(d, q, k, v, out, sm_count, st);
}

}  // namespace rs
