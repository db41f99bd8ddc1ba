// Projection and MLP of a block of 192 columns in one kernel (Eq. att, Eq. MLP, Sec. 3.2), included by rs_gemm_tc.cu:
//     x' = o Wo^T + bo + x,   m = GELU(LN(x') W1^T + b1) W2^T + b2,   out = m + x',   the scored pair's partial sums, row sums
// As four kernels such a block moves x' (fp32) three times, LN(x') twice and the hidden layer, four times as wide as the
// tokens, twice through memory, and with K of three slabs the products are bound by their epilogues.  A tile of 192 columns
// holds whole rows, and a pair of CTAs has room for all that 256 rows need from o to out:
//   * P = o Wo^T in tensor memory; sixteen warps (four to a row quadrant, 48 columns each) add bias and residual, keep x' in
//     shared memory and write LN(x') where o was, as a K-major operand;
//   * the hidden layer goes by in chunks of 128 columns: S = LN(x') W1c^T (two buffers in turn); the sixteen warps read it (32
//     columns each), apply bias and GELU and write it, rounded to bf16, as the tensor-memory A operand of O += h W2c^T, where
//     P was;
//   * they take O and x' out.
// The weights stream through a TMA ring, each CTA of the pair loading its half of every piece (no multicast).  LN(x') and the
// hidden layer are rounded to bf16, and x' is fp32, as where they go through memory.
// What bounds it: see tail_tc_use.
#pragma once
#include "rs_internal.h"
#include "rs_gemm.cuh"
#include "rs_device.cuh"
#include "rs_once.h"
#include "rs_tc.cuh"

namespace rs {
namespace tail {

constexpr int D = 192, C = 128;                          // columns of a token; hidden columns per chunk
constexpr int kMaxHidden = 768;                          // b1 is held in shared memory
constexpr int kParts = 4, kPartCols = D / kParts;        // partial sums per row, one per 48 columns

struct TailArgs {
    int T, Dm;
    const float *bo, *ln_g, *ln_b, *b1, *b2;             // biases: or null
    float ln_eps;
    const __nv_bfloat16* x;                              // block input, through row_map if that is given
    const int* row_map;
    float* attn_partials;                                // sums of the pair (SA(LN(x)), x), or null
    float* partials;                                     // sums of the pair score_kind names, or null
    float* stats_out;                                    // [T, kParts][2] or null
    void* out;                                           // [T, D]
    int score_kind, dist;
    const int* lens;
    int seq_n;
    int* status;
};

namespace {

using namespace tc;
using namespace gemm;

constexpr int BM = 128, BK = 64;                         // rows per CTA, columns of a slab
// warp 0: weights and o by TMA, warp 1: MMA (leader CTA), warp 2: x, warp 3: none, 4-19: rows
constexpr int kRow0 = 4, kRowWarps = 16, kThreads = 32 * (kRow0 + kRowWarps);
constexpr int TILE_BYTES = BM * D * 2;                   // 48 KB: three slabs of 128 rows x 128 bytes, 128-byte swizzle
constexpr int SLAB_BYTES = BM * 128;
constexpr int STAGE_BYTES = C * D;                       // 24 KB: this CTA's half of a [128, 192] or [192, 128] piece of a weight
constexpr int STAGES = 3;
// o and then LN(x') | x (three slabs) and then x' (six slabs of 32 columns of fp32) and then out in its place | weights
constexpr int OFF_O = 0, OFF_U = 0, OFF_X = TILE_BYTES, OFF_STAGE = OFF_X + 2 * TILE_BYTES;
constexpr int OFF_BAR = OFF_STAGE + STAGES * STAGE_BYTES;
constexpr int OFF_VEC = OFF_BAR + 256;                   // float bo, ln_g, ln_b, b2 [D] each, b1 [kMaxHidden]
constexpr int OFF_RED = OFF_VEC + (4 * D + kMaxHidden) * 4;      // float [2][kParts][BM]: sums of a row's quarters
constexpr int OFF_MASK = OFF_RED + 2 * kParts * BM * 4;
constexpr size_t SMEM = (size_t)OFF_MASK + kMaskWords * 4;       // the window itself must be 1024-byte aligned
static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
static_assert(D == 3 * BK && C == 2 * BK, "boxes of the weights");
constexpr int P_COL = 0, O_COL = 0, S_COL = D, H_COL = D + 2 * C;    // tensor memory: P and then O | two chunks | a chunk after GELU
static_assert(H_COL + C / 2 <= 512, "tensor memory");

// Sixteen columns as packed pairs.
using attn::pack2; using attn::unpack2; using attn::ffma2; using attn::fadd2; using attn::fmul2;
__device__ __forceinline__ void pairs(const uint32_t (&v)[16], uint64_t (&y)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) y[j] = pack2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
}
__device__ __forceinline__ void unpairs(const uint64_t (&y)[8], uint32_t (&v)[16]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        float a, b;
        unpack2(y[j], a, b);
        v[2 * j] = __float_as_uint(a);
        v[2 * j + 1] = __float_as_uint(b);
    }
}
__device__ __forceinline__ float both(uint64_t s) {
    float a, b;
    unpack2(s, a, b);
    return a + b;
}
__device__ __forceinline__ void add_vec(uint64_t (&y)[8], const float* b) {
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
        const float4 t = *reinterpret_cast<const float4*>(b + 2 * j);
        y[j] = fadd2(y[j], pack2(t.x, t.y));
        y[j + 1] = fadd2(y[j + 1], pack2(t.z, t.w));
    }
}
// Adds the pairs (u, v) to the sums of the chosen distance.
__device__ __forceinline__ void score16(int dist, const uint64_t (&u)[8], const float (&v)[16], float& s0, float& s1, float& s2) {
    if (dist == RS_DIST_L2) {
        uint64_t s = pack2(s0, 0.f);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const uint64_t d = fadd2(u[j], pack2(-v[2 * j], -v[2 * j + 1]));
            s = ffma2(d, d, s);
        }
        s0 = both(s);
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float a, b;
            unpack2(u[j], a, b);
            score_acc(dist == RS_DIST_L1 ? RS_DIST_L1 : RS_DIST_COS, a, v[2 * j], s0, s1, s2);
            score_acc(dist == RS_DIST_L1 ? RS_DIST_L1 : RS_DIST_COS, b, v[2 * j + 1], s0, s1, s2);
        }
    }
}

template <typename OutT>
__global__ void __launch_bounds__(kThreads, 1)
tail_kernel(const __grid_constant__ CUtensorMap tmO, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmWo,
            const __grid_constant__ CUtensorMap tmW1, const __grid_constant__ CUtensorMap tmW2, OutT* __restrict__ out, const TailArgs args) {
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;
    if (smem_u32(smem) & 1023u) {
        if (threadIdx.x == 0) atomicExch(args.status, RS_DEV_SMEM_ALIGN);
        return;
    }
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
    uint64_t* full = bars;                       // [STAGES] leader's: both CTAs' weights landed
    uint64_t* empty = full + STAGES;             // [STAGES] per CTA: the products reading the stage retired
    uint64_t* a_full = empty + STAGES;           // leader's: o of the tile landed in both CTAs
    uint64_t* p_full = a_full + 1;               // per CTA: P complete (and o read)
    uint64_t* u_full = p_full + 1;               // leader's: LN(x') written (one arrival per row warp of either CTA)
    uint64_t* s_full = u_full + 1;               // [2] per CTA: S of a chunk complete
    uint64_t* s_free = s_full + 2;               // [2] leader's: S read (one arrival per row warp of either CTA)
    uint64_t* h_ready = s_free + 2;              // leader's: the chunk after GELU written (likewise)
    uint64_t* h_free = h_ready + 1;              // per CTA: the product reading it retired
    uint64_t* u_free = h_free + 1;               // per CTA: the first layer's products of the tile retired
    uint64_t* o_full = u_free + 1;               // per CTA: O of the tile complete
    uint64_t* o_empty = o_full + 1;              // leader's: O read by all row warps of both CTAs
    uint64_t* x_full = o_empty + 1;              // per CTA: x of the tile landed
    uint64_t* x_empty = x_full + 1;              // per CTA: the output that replaced x' has been taken out
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(x_empty + 1);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    float* vec = reinterpret_cast<float*>(smem + OFF_VEC);
    float *bo_s = vec, *g_s = vec + D, *be_s = vec + 2 * D, *b2_s = vec + 3 * D, *b1_s = vec + 4 * D;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();
    const int pair = (int)cluster_id_x(), npairs = (int)cluster_count_x();
    const int num_m = (args.T + 2 * BM - 1) / (2 * BM), NC = args.Dm / C;

    if (threadIdx.x == 0) {
        prefetch_tmap(&tmO); prefetch_tmap(&tmX); prefetch_tmap(&tmWo); prefetch_tmap(&tmW1); prefetch_tmap(&tmW2);
        for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        mbar_init(a_full, 1);
        mbar_init(p_full, 1);
        mbar_init(u_full, 2 * kRowWarps);
        for (int b = 0; b < 2; ++b) {
            mbar_init(&s_full[b], 1);
            mbar_init(&s_free[b], 2 * kRowWarps);
        }
        mbar_init(h_ready, 2 * kRowWarps);
        mbar_init(h_free, 1);
        mbar_init(u_free, 1);
        mbar_init(o_full, 1);
        mbar_init(o_empty, 2 * kRowWarps);
        mbar_init(x_full, args.row_map ? 32 : 1);        // by the lane that starts the TMA copies, or by each lane's own copies
        mbar_init(x_empty, kRowWarps);
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, 512);
        tmem_relinquish_pair();
    }
    for (int i = threadIdx.x; i < D; i += kThreads) {
        bo_s[i] = args.bo ? __ldg(args.bo + i) : 0.f;
        g_s[i] = __ldg(args.ln_g + i);
        be_s[i] = __ldg(args.ln_b + i);
        b2_s[i] = args.b2 ? __ldg(args.b2 + i) : 0.f;
    }
    for (int i = threadIdx.x; i < args.Dm; i += kThreads) b1_s[i] = args.b1 ? __ldg(args.b1 + i) : 0.f;
    tc_fence_before();
    __syncthreads();
    cluster_sync();                              // the peer's barriers exist before anything signals them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    grid_dep_launch();
    // Weights do not depend on the kernel before this one (TailCall): the producer fills the ring first (below), unless a mask of row
    // tiles has to be made with the whole CTA.
    const bool early = !args.lens;
    if (!(warp == 0 && early)) grid_dep_wait();

    int tiles = num_m;
    uint32_t* mask = args.lens ? reinterpret_cast<uint32_t*>(smem + OFF_MASK) : nullptr;
    if (mask) tiles = mark_row_tiles(mask, args.lens, args.seq_n, args.T, warp, lane, kThreads);
    const int mine = tiles > pair ? (tiles - pair + npairs - 1) / npairs : 0;      // tiles pair, pair + npairs, ...
    RowTiles row_tiles = {mask};                 // (each role walks its own copy)
    auto row0 = [&](int t) { return row_tiles.at(pair + t * npairs) * (2 * BM) + (int)rank * BM; };

    if (warp == 0) {
        // ---------------- weights and o (both CTAs; each loads its own halves) ----------------
        if (elect_one()) {
            uint32_t it = 0;
            bool ok = true, waited = !early;
            auto load_o = [&](int t) {           // the first layer has read LN(x') of the tile before
                if (t > 0) ok = ok && mbar_wait(u_free, (t - 1) & 1u, abort_flag);
                if (!ok) return;
                const uint32_t lead = map_to_cta(smem_u32(a_full), 0);
                const int m = row0(t);
                if (rank == 0) mbar_expect_tx(a_full, 2 * TILE_BYTES);
#pragma unroll
                for (int kb = 0; kb < D / BK; ++kb) tma_load_2d_pair(smem + OFF_O + kb * SLAB_BYTES, &tmO, lead, kb * BK, m);
            };
            // kind 0: slabs 2 i and 2 i + 1 of Wo, 1: chunk i of W1, 2: chunk i of W2
            auto piece = [&](int kind, int i) {
                if (!waited && it == STAGES) {   // the ring is full: now o of the first tile
                    grid_dep_wait();
                    waited = true;
                    load_o(0);
                }
                const int s = it % STAGES;
                ok = ok && mbar_wait(&empty[s], ((it / STAGES) & 1u) ^ 1u, abort_flag);
                if (!ok) return;
                uint8_t* dst = smem + OFF_STAGE + s * STAGE_BYTES;
                const uint32_t lead_full = map_to_cta(smem_u32(&full[s]), 0);
                const int boxes = kind == 1 ? D / BK : kind == 0 && i == 1 ? 1 : 2, box_bytes = kind == 1 ? (C / 2) * 128 : (D / 2) * 128;
                if (rank == 0) mbar_expect_tx(&full[s], 2 * boxes * box_bytes);
                for (int k = 0; k < boxes; ++k) {
                    if (kind == 1) tma_load_2d_pair(dst + k * box_bytes, &tmW1, lead_full, k * BK, i * C + (int)rank * (C / 2));
                    else tma_load_2d_pair(dst + k * box_bytes, kind == 0 ? &tmWo : &tmW2, lead_full, (2 * i + k) * BK, (int)rank * (D / 2));
                }
                ++it;
            };
            if (waited && mine > 0) load_o(0);
            for (int t = 0; t < mine && ok; ++t) {
                piece(0, 0);
                piece(0, 1);
                piece(1, 0);
                for (int c = 0; c < NC && ok; ++c) {
                    if (c + 1 < NC) piece(1, c + 1);
                    piece(2, c);
                }
                if (t + 1 < mine) load_o(t + 1);
            }
            if (!waited) grid_dep_wait();
            // every stage filled here has been read (and its copies have landed) before the CTA may exit
            const uint32_t issued = it;
            for (uint32_t s = 0; s < STAGES && s < issued && ok; ++s) {
                const uint32_t last = ((issued - 1 - s) / STAGES) * STAGES + s;
                ok = mbar_wait(&empty[s], (last / STAGES) & 1u, abort_flag);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA only) ----------------
        if (rank == 0 && elect_one()) {
            constexpr uint32_t idesc_c = idesc_bf16(2 * BM, C, 0, 0), idesc_d = idesc_bf16(2 * BM, D, 0, 0);
            uint32_t it = 0;
            bool ok = true;
            auto next_stage = [&](uint64_t& db) {
                const int s = it % STAGES;
                ok = ok && mbar_wait(&full[s], (it / STAGES) & 1u, abort_flag);
                ++it;
                tc_fence_after();
                db = smem_desc_sw128(smem_u32(smem + OFF_STAGE + s * STAGE_BYTES), 16, 1024);
                return &empty[s];
            };
            const uint64_t da_u = smem_desc_sw128(smem_u32(smem + OFF_U), 16, 1024);         // (o and LN(x') in turn)
            auto first = [&](int g, bool last) { // S = LN(x') W1c^T
                const int b = g & 1;
                if (g >= 2) ok = ok && mbar_wait(&s_free[b], ((g >> 1) - 1) & 1u, abort_flag);
                uint64_t db;
                uint64_t* done = next_stage(db);
                if (!ok) return;
#pragma unroll
                for (int k = 0; k < D / 16; ++k)
                    mma_ss_pair(tmem_base + S_COL + b * C, da_u + (k / 4) * (SLAB_BYTES >> 4) + 2 * (k % 4), db + (k / 4) * ((C / 2) * 128 >> 4) + 2 * (k % 4), idesc_c, k != 0);
                mma_commit_pair(done, 3);
                mma_commit_pair(&s_full[b], 3);
                if (last) mma_commit_pair(u_free, 3);
            };
            for (int t = 0, g = 0; t < mine && ok; ++t) {
                // P = o Wo^T, over what the warps have read of the tile before
                ok = mbar_wait(a_full, t & 1u, abort_flag) && (t == 0 || mbar_wait(o_empty, (t - 1) & 1u, abort_flag));
                for (int i = 0; i < 2 && ok; ++i) {
                    uint64_t db;
                    uint64_t* done = next_stage(db);
                    if (!ok) break;
                    for (int kb = 2 * i; kb < D / BK && kb < 2 * i + 2; ++kb)
#pragma unroll
                        for (int k = 0; k < 4; ++k)
                            mma_ss_pair(tmem_base + P_COL, da_u + kb * (SLAB_BYTES >> 4) + 2 * k, db + (kb - 2 * i) * ((D / 2) * 128 >> 4) + 2 * k, idesc_d, (kb | k) != 0);
                    mma_commit_pair(done, 3);
                }
                if (!ok) break;
                mma_commit_pair(p_full, 3);
                ok = mbar_wait<true>(u_full, t & 1u, abort_flag);    // LN(x') of the peer's rows too
                if (ok) first(g, NC == 1);
                for (int c = 0; c < NC && ok; ++c, ++g) {
                    if (c + 1 < NC) first(g + 1, c + 2 == NC);
                    ok = ok && mbar_wait(h_ready, g & 1u, abort_flag);
                    uint64_t db;
                    uint64_t* done = next_stage(db);
                    if (!ok) break;
#pragma unroll
                    for (int k = 0; k < C / 16; ++k)     // O (+)= h W2c^T
                        mma_ts_pair(tmem_base + O_COL, tmem_base + H_COL + 8 * k, db + (k / 4) * ((D / 2) * 128 >> 4) + 2 * (k % 4), idesc_d, (c | k) != 0);
                    mma_commit_pair(done, 3);
                    mma_commit_pair(h_free, 3);
                    if (c == NC - 1) mma_commit_pair(o_full, 3);
                }
            }
            // arrivals on this CTA's barriers that nothing above waited for
            const int chunks = mine * NC;
            for (int g = chunks > 2 ? chunks - 2 : 0; g < chunks && ok; ++g) ok = mbar_wait(&s_free[g & 1], (g >> 1) & 1u, abort_flag);
            if (mine > 0 && ok) mbar_wait(o_empty, (mine - 1) & 1u, abort_flag);
        }
    } else if (warp == 2) {
        // ---------------- x of the tiles, a tile ahead ----------------
        for (int t = 0; t < mine; ++t) {
            const int m = row0(t);
            if (t > 0 && !args.row_map && lane == 0)     // (x lands when x' of the tile before has been used, and should come from the L2 then)
                for (int kb = 0; kb < D / BK; ++kb) tma_prefetch_2d(&tmX, kb * BK, m);
            if (t > 0 && !__all_sync(0xffffffffu, mbar_wait(x_empty, (t - 1) & 1u, abort_flag))) break;
            if (!args.row_map) {
                if (lane == 0) {
                    mbar_expect_tx(x_full, TILE_BYTES);
                    for (int kb = 0; kb < D / BK; ++kb) tma_load_2d(smem + OFF_X + kb * SLAB_BYTES, &tmX, x_full, kb * BK, m);
                }
                continue;
            }
            // through the row map: 16-byte asynchronous copies, a row's pieces by eight neighbouring lanes, in the layout of the
            // tensor map's swizzle; rows past T become zeros
            const int p = lane & 7;
            for (int i = lane >> 3; i < BM; i += 4) {
                const int row = m + i, sr = row < args.T ? __ldg(args.row_map + row) : -1;
#pragma unroll
                for (int kb = 0; kb < D / BK; ++kb)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                                 ::"r"(smem_u32(smem + OFF_X + kb * SLAB_BYTES + i * 128 + ((p ^ (i & 7)) << 4))),
                                 "l"(args.x + (size_t)(sr < 0 ? 0 : sr) * D + kb * BK + p * 8), "r"(sr < 0 ? 0 : 16) : "memory");
            }
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(x_full)) : "memory");
        }
        // every copy started here has landed (and has been used) before the CTA may exit
        if (mine > 0) mbar_wait(x_empty, (mine - 1) & 1u, abort_flag);
    } else if (warp >= kRow0) {
        // ---------------- rows: bias, residual, LayerNorm; GELU; output ----------------
        // A wait that ran out is not acted on here: the values are void, the status says so, and all sixteen warps still come to
        // the same barriers.
        const int q = warp & 3, grp = (warp - kRow0) >> 2;           // rows of the tile; columns 48 grp .. + 47, or 32 grp .. + 31 of a chunk
        const int r = q * 32 + lane, c0 = grp * kPartCols, swz = r & 7;
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t s_addr = lane_addr + S_COL + grp * 32, h_addr = lane_addr + H_COL + grp * 16;
        const uint32_t lead_u = map_to_cta(smem_u32(u_full), 0), lead_oe = map_to_cta(smem_u32(o_empty), 0);
        const uint32_t lead_h = map_to_cta(smem_u32(h_ready), 0), lead_s[2] = {map_to_cta(smem_u32(&s_free[0]), 0), map_to_cta(smem_u32(&s_free[1]), 0)};
        float* red = reinterpret_cast<float*>(smem + OFF_RED);
        // 16-byte piece i of this thread's 48 columns in a tile of bf16
        auto piece = [&](int base, int i) { const int p = grp * (kPartCols / 8) + i; return smem + base + (p >> 3) * SLAB_BYTES + r * 128 + (((p & 7) ^ swz) << 4); };
        // piece i of four fp32 columns from column col on, of row rr, in the tile of x'
        auto piece32 = [&](int rr, int col, int i) { return smem + OFF_X + (col >> 5) * SLAB_BYTES + rr * 128 + (((((col & 31) >> 2) + i) ^ (rr & 7)) << 4); };
        // the row's total from its four quarters, in one order (named barrier of the row quadrant's 128 threads)
        auto row_sum = [&](int which, float s) {
            red[(which * kParts + grp) * BM + r] = s;
            named_barrier(1 + q, 128);
            const float* p = red + which * kParts * BM + r;
            return (p[0] + p[BM]) + (p[2 * BM] + p[3 * BM]);
        };
        auto put_bf16 = [&](const uint64_t (&y)[8], int base, int i) {           // sixteen columns, pieces i and i + 1
            uint32_t w[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                float a, b;
                unpack2(y[j], a, b);
                w[j] = pack_bf16(a, b);
            }
            *reinterpret_cast<uint4*>(piece(base, i)) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4*>(piece(base, i + 1)) = make_uint4(w[4], w[5], w[6], w[7]);
        };
        auto put_sums = [&](float* out, int row, float sq, float sq1, float sq2) {
            float* p = out + ((size_t)row * kParts + grp) * (args.dist == RS_DIST_COS ? 3 : 1);
            p[0] = sq;
            if (args.dist == RS_DIST_COS) { p[1] = sq1; p[2] = sq2; }
        };
        int g = 0;
        for (int t = 0; t < mine; ++t) {
            const int m0 = row0(t), row = m0 + r;
            const bool valid = row < args.T;
            // x' = P + bo + x, back where P was
            mbar_wait(x_full, t & 1u, abort_flag);
            mbar_wait(p_full, t & 1u, abort_flag);
            __syncwarp();
            tc_fence_after();
            float sq = 0.f, sq1 = 0.f, sq2 = 0.f;
            uint64_t sum2 = pack2(0.f, 0.f);
#pragma unroll 1
            for (int i = 0; i < kPartCols; i += 16) {
                uint32_t v[16];
                tmem_ld_32x16(lane_addr + P_COL + c0 + i, v);
                float x[16];
                unpack16<__nv_bfloat16>(*reinterpret_cast<const uint4*>(piece(OFF_X, i / 8)), *reinterpret_cast<float(*)[8]>(x));
                unpack16<__nv_bfloat16>(*reinterpret_cast<const uint4*>(piece(OFF_X, i / 8 + 1)), *reinterpret_cast<float(*)[8]>(x + 8));
                tmem_wait_ld();
                uint64_t y[8];
                pairs(v, y);
                add_vec(y, bo_s + c0 + i);
                if (args.attn_partials) score16(args.dist, y, x, sq, sq1, sq2);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    y[j] = fadd2(y[j], pack2(x[2 * j], x[2 * j + 1]));
                    sum2 = fadd2(sum2, y[j]);
                }
                unpairs(y, v);
                tmem_st_32x16(lane_addr + P_COL + c0 + i, v);
            }
            if (args.attn_partials && valid) put_sums(args.attn_partials, row, sq, sq1, sq2);
            // LN(x') -> the operand of the first layer
            const float mu = row_sum(0, both(sum2)) / (float)D;
            const uint64_t mneg2 = pack2(-mu, -mu);
            tmem_wait_st();
            uint64_t var2 = pack2(0.f, 0.f);
#pragma unroll 1
            for (int i = 0; i < kPartCols; i += 16) {
                uint32_t v[16];
                tmem_ld_32x16(lane_addr + P_COL + c0 + i, v);
                tmem_wait_ld();
                uint64_t y[8];
                pairs(v, y);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const uint64_t d = fadd2(y[j], mneg2);
                    var2 = ffma2(d, d, var2);
                }
            }
            const float rstd = rsqrtf(row_sum(1, both(var2)) / (float)D + args.ln_eps);
            const uint64_t rstd2 = pack2(rstd, rstd);
#pragma unroll 1
            for (int i = 0; i < kPartCols; i += 16) {
                uint32_t v[16];
                tmem_ld_32x16(lane_addr + P_COL + c0 + i, v);
                tmem_wait_ld();
                // (x' takes the place of x, which all of the row's threads have read before the sums)
#pragma unroll
                for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(piece32(r, c0 + i, j)) = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
                uint64_t y[8];
                pairs(v, y);
#pragma unroll
                for (int j = 0; j < 8; j += 2) {
                    const float4 gm = *reinterpret_cast<const float4*>(g_s + c0 + i + 2 * j), bt = *reinterpret_cast<const float4*>(be_s + c0 + i + 2 * j);
                    y[j] = ffma2(fmul2(fadd2(y[j], mneg2), rstd2), pack2(gm.x, gm.y), pack2(bt.x, bt.y));
                    y[j + 1] = ffma2(fmul2(fadd2(y[j + 1], mneg2), rstd2), pack2(gm.z, gm.w), pack2(bt.z, bt.w));
                }
                put_bf16(y, OFF_U, i / 8);
            }
            fence_async_smem();                          // written data visible to the tensor core's reads
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster_release(lead_u);

            // the hidden layer
#pragma unroll 1
            for (int c = 0; c < NC; ++c, ++g) {
                const int b = g & 1;
                const float* bias = b1_s + c * C + grp * 32;
                mbar_wait(&s_full[b], (g >> 1) & 1u, abort_flag);
                __syncwarp();
                tc_fence_after();
                uint32_t v[32], h[16];
                tmem_ld_32x32(s_addr + b * C, v);
                tmem_wait_ld();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_relaxed(lead_s[b]);       // the product of the chunk after next may overwrite S
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 bb = *reinterpret_cast<const float4*>(bias + j);
                    float y0 = __uint_as_float(v[j]) + bb.x, y1 = __uint_as_float(v[j + 1]) + bb.y;
                    float y2 = __uint_as_float(v[j + 2]) + bb.z, y3 = __uint_as_float(v[j + 3]) + bb.w;
                    gelu_erf2(y0, y1);
                    gelu_erf2(y2, y3);
                    h[j / 2] = pack_bf16(y0, y1);
                    h[j / 2 + 1] = pack_bf16(y2, y3);
                }
                if (g > 0) {                             // the product with the chunk before has read its place
                    mbar_wait(h_free, (g - 1) & 1u, abort_flag);
                    __syncwarp();
                    tc_fence_after();
                }
                tmem_st_32x16(h_addr, h);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_relaxed(lead_h);
            }

            // out = O + b2 + x', score, row sums
            const int xrow = (args.score_kind == 2 && args.row_map && valid) ? __ldg(args.row_map + row) : row;
            mbar_wait(o_full, t & 1u, abort_flag);
            __syncwarp();
            tc_fence_after();
            sq = sq1 = sq2 = 0.f;
            uint64_t st1 = pack2(0.f, 0.f), st2 = st1;
#pragma unroll 1
            for (int i = 0; i < kPartCols; i += 16) {
                uint32_t v[16];
                tmem_ld_32x16(lane_addr + O_COL + c0 + i, v);
                float w[16], u[16];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 x4 = *reinterpret_cast<const float4*>(piece32(r, c0 + i, j));
                    w[4 * j] = x4.x; w[4 * j + 1] = x4.y; w[4 * j + 2] = x4.z; w[4 * j + 3] = x4.w;
                }
                tmem_wait_ld();
                if (i + 16 == kPartCols) {               // O fully read by this warp
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive_cluster_relaxed(lead_oe);
                }
                uint64_t y[8];
                pairs(v, y);
                add_vec(y, b2_s + c0 + i);
                if (args.score_kind == 2) {
                    // whole-block shift: x^ - x, with the block input x read here (rows past T: zeros)
                    const uint4* x0p = reinterpret_cast<const uint4*>(args.x + (size_t)xrow * D + c0 + i);
                    unpack16<__nv_bfloat16>(valid ? __ldg(x0p) : make_uint4(0u, 0u, 0u, 0u), *reinterpret_cast<float(*)[8]>(u));
                    unpack16<__nv_bfloat16>(valid ? __ldg(x0p + 1) : make_uint4(0u, 0u, 0u, 0u), *reinterpret_cast<float(*)[8]>(u + 8));
                } else {
#pragma unroll
                    for (int j = 0; j < 16; ++j) u[j] = w[j];
                }
                if (args.partials && args.score_kind == 0) score16(args.dist, y, u, sq, sq1, sq2);
#pragma unroll
                for (int j = 0; j < 8; ++j) y[j] = fadd2(y[j], pack2(w[2 * j], w[2 * j + 1]));
                if (args.partials && args.score_kind != 0) score16(args.dist, y, u, sq, sq1, sq2);
                // a lane's results take the place of its x'
                if constexpr (sizeof(OutT) == 2) {
                    uint32_t pk[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float a, b;
                        unpack2(y[j], a, b);
                        pk[j] = pack_bf16(a, b);
                        if (args.stats_out) {            // sums of the values as stored: the next block reads these bf16 numbers
                            const uint64_t z = pack2(__uint_as_float(pk[j] << 16), __uint_as_float(pk[j] & 0xffff0000u));
                            st1 = fadd2(st1, z);
                            st2 = ffma2(z, z, st2);
                        }
                    }
                    *reinterpret_cast<uint4*>(piece32(r, c0 + i, 0)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
                    *reinterpret_cast<uint4*>(piece32(r, c0 + i, 1)) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; j += 2) {
                        float4 o4;
                        unpack2(y[j], o4.x, o4.y);
                        unpack2(y[j + 1], o4.z, o4.w);
                        *reinterpret_cast<float4*>(piece32(r, c0 + i, j / 2)) = o4;
                    }
                }
            }
            __syncwarp();
            // the warp's 32 rows x 48 columns leave with neighbouring lanes on neighbouring 16-byte pieces of a row: LPR lanes to the
            // sixteen columns of a row, and rows to a quarter of a warp whose pieces lie in different banks
            constexpr int LPR = sizeof(OutT) == 2 ? 2 : 4, ROWS = 32 / LPR, ID = LPR == 2 ? 1 : 2;
            const int sub = lane & (LPR - 1), idx = lane >> ID;
            const int rsub = LPR == 2 ? (idx >> 3) * 8 + (idx & 3) * 2 + ((idx >> 2) & 1) : (idx & 1) * 4 + (idx >> 1);
#pragma unroll
            for (int rb = 0; rb < 32; rb += ROWS) {
                const int rr = q * 32 + rb + rsub;
                uint4 t4[3];
#pragma unroll
                for (int i = 0; i < 3; ++i) t4[i] = *reinterpret_cast<const uint4*>(piece32(rr, c0 + 16 * i, sub));
                char* to = reinterpret_cast<char*>(out + (size_t)(m0 + rr) * D + c0) + sub * 16;
                if (m0 + rr < args.T) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) *reinterpret_cast<uint4*>(to + i * 16 * sizeof(OutT)) = t4[i];
                }
            }
            if (args.partials && valid) put_sums(args.partials, row, sq, sq1, sq2);
            if (args.stats_out && valid) reinterpret_cast<float2*>(args.stats_out)[(size_t)row * kParts + grp] = make_float2(both(st1), both(st2));
            fence_async_smem();                          // (the next x lands over what was written here)
            __syncwarp();
            if (lane == 0) mbar_arrive(x_empty);
        }
        // the last signals on this CTA's barriers that nothing above waited for
        if (mine > 0) {
            mbar_wait(h_free, (mine * NC - 1) & 1u, abort_flag);
            mbar_wait(u_free, (mine - 1) & 1u, abort_flag);
        }
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) atomicExch(args.status, RS_DEV_TIMEOUT);
    cluster_leave();                                     // (each CTA has seen everything that its peer signals to it: see the roles' ends)
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, 512);
    }
}

template <typename OutT>
cudaError_t launch(const CUtensorMap& tmO, const CUtensorMap& tmX, const CUtensorMap& tmWo, const CUtensorMap& tmW1, const CUtensorMap& tmW2,
                   const TailArgs& args, int sm_count, cudaStream_t st) {
    static PerDeviceOnce attr_once;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = (cudaError_t)attr_once.run(dev, [] { return (int)cudaFuncSetAttribute(tail_kernel<OutT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM); });
    if (e != cudaSuccess) return e;
    const int tiles = (args.T + 2 * BM - 1) / (2 * BM), pairs = tiles < sm_count / 2 ? tiles : sm_count / 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, tail_kernel<OutT>, tmO, tmX, tmWo, tmW1, tmW2, (OutT*)args.out, args);
}

}  // namespace
}  // namespace tail
}  // namespace rs
