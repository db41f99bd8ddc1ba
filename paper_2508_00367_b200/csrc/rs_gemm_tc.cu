// bf16 GEMM on the 5th-generation tensor cores with the block's epilogues fused in:
//     out[M, N] = epilogue(A[M, K] . W[N, K]^T)
// A and W are K-major.  Two CTAs on neighbouring SMs form a pair (a cluster of two) that owns
// a 256 x BN output tile: each CTA loads its own 128 rows of A and BN/2 rows of W by TMA
// (128-byte swizzle, no multicast) into a shared-memory ring, and one thread of the pair's
// leader issues tcgen05.mma.cta_group::2, which reads both CTAs' shared memory and accumulates
// each CTA's 128 x BN half in that CTA's tensor memory.  Per byte moved from L2 to the SMs the
// pair tile does twice the arithmetic of a 128 x 128 tile, which is what lifts the kernel off
// the L2 -> SM bandwidth bound.  The fp32 accumulator is double-buffered in tensor memory, so
// the eight epilogue warps of each CTA drain tile i (tcgen05.ld -> bias / GELU / residual /
// score -> swizzled shared memory -> one TMA store per warp and 128-byte column block) while the
// main loop of tile i+1 runs.
//
// Epilogues (Eq. att, Eq. MLP, Sec. 3.2):
//   EPI_BIAS       out = acc + b                          -> bf16      (QKV projection)
//   EPI_BIAS_GELU  out = GELU(acc + b)                    -> bf16      (FC1)
//   EPI_RESID      a = acc + b;  out = a + x              -> fp32      (projection + residual = x');
//                  optionally partial sums of (a - x)^2 per row    (shift through attention, choice (i))
//   EPI_SCORE      m = acc + b;  out = m + x';  partial sums of (m - x')^2, m^2 or (out - x)^2 per row
//                                                          -> bf16/fp32 (FC2 + residual + shift score)
#include <string.h>

#include "rs_internal.h"
#include "rs_attn.cuh"
#include "rs_gemm.cuh"
#include "rs_device.cuh"
#include "rs_once.h"
#include "rs_tc.cuh"

namespace rs {
namespace gemm {

// Exact-erf GELU, v * Phi(v), to fp32 accuracy (max abs error 8e-7 over all v) without erff:
// with q(t) = -log2(Phi(-t)) for t >= 0,  Phi(v) = 2^-q(|v|) for v < 0 and 1 - 2^-q(|v|) for
// v >= 0.  q is smooth (about t^2/2 * log2(e) plus slow terms) and a degree-5 polynomial fitted
// on [0, 7] with weight t * Phi(-t) reproduces GELU to that accuracy; its positive leading
// coefficient keeps 2^-q -> 0 for large |v|.  Coefficients from csrc/fit_gelu.py.
// A value stays above -infinity, so that -infinity gives 0; max.NaN keeps a NaN.
constexpr float kLowest = -3.4e38f;
using attn::max_nan;
__device__ __forceinline__ float ex2_ftz(float x) {
    float e;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x));
    return e;
}
__device__ __forceinline__ float gelu_erf(float v) {
    v = max_nan(v, kLowest);
    const float a = fabsf(v);
    float q = 0.00047694556997157633f;
    q = fmaf(q, a, -0.00711308470266570f);
    q = fmaf(q, a, 0.05190887302160263f);
    q = fmaf(q, a, 0.4598882496356964f);
    q = fmaf(q, a, 1.1508461236953735f);
    q = fmaf(q, a, 1.0000265836715698f);
    const float e = ex2_ftz(-q);
    return v * (v >= 0.f ? 1.f - e : e);
}
// A pair at a time on packed FMAs, with n = -|v|: the polynomial in n gives -q, and GELU = max(v, 0) + n 2^-q for either
// sign: 12 instructions a pair instead of 22, and the 2^x of the special-function unit (16 of its cycles a pair and warp) is
// what is left.  FC1 50432 x 768 x 192 31.9 -> 30.9 us, 25216 x 3072 x 768 80.8 -> 78.3, 16400 x 3072 x 768 56.1 -> 54.2.
__device__ __forceinline__ void gelu_erf2(float& v0, float& v1) {
    using attn::pack2; using attn::unpack2; using attn::ffma2;
    const uint64_t n = pack2(max_nan(-fabsf(v0), kLowest), max_nan(-fabsf(v1), kLowest));
    auto c = [](float x) { return pack2(x, x); };
    uint64_t q = c(0.00047694556997157633f);
    q = ffma2(q, n, c(0.00711308470266570f));
    q = ffma2(q, n, c(0.05190887302160263f));
    q = ffma2(q, n, c(-0.4598882496356964f));
    q = ffma2(q, n, c(1.1508461236953735f));
    q = ffma2(q, n, c(-1.0000265836715698f));
    float q0, q1;
    unpack2(q, q0, q1);
    unpack2(ffma2(n, pack2(ex2_ftz(q0), ex2_ftz(q1)), pack2(fmaxf(v0, 0.f), fmaxf(v1, 0.f))), v0, v1);
}

}  // namespace gemm
}  // namespace rs

#include "rs_gemm_small.cuh"
#include "rs_tail.cuh"

namespace rs {

namespace {

using namespace tc;
using namespace gemm;

constexpr int BM = 128;                       // rows per CTA; the pair's tile has 2 * BM rows
constexpr int BK = 64;
// warp 0: TMA, warp 1: MMA (leader CTA), the others: epilogue, in groups of four that take a range of columns each
constexpr int A_BYTES = BM * BK * 2;          // 16 KB
constexpr int STG_BYTES = 32 * 128;           // one staged output block of a warp: its 32 rows of 128 bytes
constexpr int RES_BOX_BYTES = 32 * 64;         // residual of one 32-column chunk of a warp: 32 rows of 32 bf16

// The list of work of a launch.  Whole tiles go to the pairs round robin; 256-wide tiles left for a last round that
// half of the pairs or fewer would work on are cut in two, so that the round takes a part of a tile's time.  A
// 128-column piece costs about 0.65 of a whole tile: it moves more operand bytes per FLOP and the ring's five stages hold
// less of it in flight, which is why tiles are not narrow to begin with; quarters (0.75 to 0.9) gain nothing more.
// 25104 x 768 x 3072 110 -> 98 us (one tile more than four rounds), 12608 x 768 x 768 24.1 -> 21.5.
template <int BN> struct WorkList {
    int full, rest, pieces, num_n;     // tiles of the full rounds, tiles of the last, the pieces of each of those, tiles per row tile
    __device__ __forceinline__ WorkList(int tiles, int num_n_, int npairs) : num_n(num_n_) {
        full = tiles / npairs * npairs;
        rest = tiles - full;
        pieces = BN == 256 && rest * 2 <= npairs ? 2 : 1;
    }
    __device__ __forceinline__ int count() const { return full + rest * pieces; }
    struct Piece { int row_tile, n0, width; };
    __device__ __forceinline__ Piece at(int i) const {
        int tile = i, part = 0, width = BN;
        if (i >= full && pieces > 1) {
            tile = full + ((i - full) >> 1);
            part = (i - full) & 1;
            width = BN / 2;
        }
        const int mt = tile / num_n;
        return {mt, (tile - mt * num_n) * BN + part * width, width};
    }
};

// EPI_RESID brings the bf16 residual of a warp's rows in by TMA (a row per lane read straight from
// global memory touches 32 lines per load instruction and cost a fifth of the projection's time), two chunks of
// 32 columns ahead, the next tile's first ones included.  It pays for the room with one operand stage less.  (A whole tile's boxes at a
// time left room for one staging buffer per warp only, and a third of the epilogue waited for it: 50432 x 192 x 192
// 19.5 -> 18.8 us, 25216 x 384 x 384 20.0 -> 19.2, 6924 x 1024 x 1024 21.5 -> 21.0.)
// WIDE: four (192 columns: three) groups of epilogue warps with 64 columns each instead of two with half a tile each, for
// products whose K is so short that the epilogue is the longer part: four warps a scheduler instead of two cover
// its latencies.  (Longer ones are slower that way, their stores then come in one burst: see wide_epilogue.)
template <int BN, int EPI, bool WIDE> struct Cfg {
    static constexpr bool RES_TMA = EPI == EPI_RESID;
    static constexpr bool LN = EPI == EPI_BIAS_LN;                 // one staging buffer per warp, room for a second column vector
    static constexpr int B_BYTES = (BN / 2) * BK * 2;              // this CTA's half of the W tile
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = (BN == 128 ? 6 : 5) - (RES_TMA ? 1 : 0);
    static constexpr int TMEM_COLS = (BN == 128) ? 256 : 512;      // two accumulators, a power of two
    static constexpr int SPLIT = (BN == 128) ? 64 : 128;           // epilogue warps 2-5 take columns [0, SPLIT) of a whole tile
    static constexpr int GROUPS = WIDE ? BN / 64 : 2, EPI_WARPS = 4 * GROUPS, THREADS = 64 + 32 * EPI_WARPS;
    static constexpr int STG_PER_WARP = LN || WIDE ? 1 : 2;
    static constexpr int RES_WARP_BYTES = RES_TMA ? 2 * RES_BOX_BYTES : 0;
    static constexpr int OFF_STG = STAGES * STAGE_BYTES;
    static constexpr int OFF_RES = OFF_STG + EPI_WARPS * STG_PER_WARP * STG_BYTES;
    static constexpr int OFF_BAR = OFF_RES + EPI_WARPS * RES_WARP_BYTES;
    static constexpr int OFF_BIAS = OFF_BAR + 256;                 // float [2 tile parities][256]: bias of the tile's columns
    static constexpr int OFF_COLSUM = OFF_BIAS + 2048;             // EPI_BIAS_LN: float [2][256] like the bias
    static constexpr int OFF_MASK = OFF_BIAS + (LN ? 4096 : 2048);  // one bit per row tile (batches with a count per sample)
    static constexpr size_t SMEM = (size_t)OFF_MASK + kMaskWords * 4;   // the window itself must be 1024-byte aligned
    static_assert(SMEM <= 227 * 1024, "shared memory of one CTA");
};

template <int BN, int EPI, typename OutT, bool WIDE>
__global__ void __launch_bounds__((Cfg<BN, EPI, WIDE>::THREADS), 1)
gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmBh, const __grid_constant__ CUtensorMap tmOut,
               const __grid_constant__ CUtensorMap tmRes, const GemmArgs args) {
    using C = Cfg<BN, EPI, WIDE>;
    // The 128-byte swizzle wants 1024-byte aligned stage and staging buffers, and the layout leaves no
    // room to round the base up: a window that is not aligned is reported, and nothing else is done.
    extern __shared__ __align__(1024) uint8_t smem_raw[];
    uint8_t* smem = smem_raw;
    if (smem_u32(smem) & 1023u) {
        if (threadIdx.x == 0) atomicExch(args.status, RS_DEV_SMEM_ALIGN);
        return;
    }
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
    uint64_t* full = bars;                       // [STAGES] leader's: both CTAs' operands landed
    uint64_t* empty = bars + C::STAGES;          // [STAGES] per CTA: the MMAs reading the stage retired
    uint64_t* tfull = bars + 2 * C::STAGES;      // [2] per CTA: accumulator complete
    uint64_t* tempty = bars + 2 * C::STAGES + 2; // [2] leader's: both CTAs' epilogues drained it
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * C::STAGES + 4);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
    volatile int* group_fail = reinterpret_cast<volatile int*>(tmem_slot + 2);   // [GROUPS]
    uint64_t* res_full = bars + 2 * C::STAGES + 6;   // [EPI_WARPS][2] a chunk of the warp's residual landed (EPI_RESID)

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t rank = cluster_ctarank();     // 0 = leader of the pair
    const int num_m = (args.M + 2 * BM - 1) / (2 * BM), num_n = args.N / BN;
    const int kblocks = args.K / BK;
    const int pair = (int)cluster_id_x(), npairs = (int)cluster_count_x();

    if (threadIdx.x == 0) {
        prefetch_tmap(&tmA);
        prefetch_tmap(&tmB);
        prefetch_tmap(&tmOut);
        for (int s = 0; s < C::STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
        for (int a = 0; a < 2; ++a) { mbar_init(&tfull[a], 1); mbar_init(&tempty[a], 2 * C::EPI_WARPS); }
        if (C::RES_TMA) {
            prefetch_tmap(&tmRes);
            // one arrival by the lane that starts the TMA copies, or one by each lane's own indexed copies
            for (int w = 0; w < 2 * C::EPI_WARPS; ++w) mbar_init(&res_full[w], args.row_map ? 32 : 1);
        }
        *abort_flag = 0;
        for (int g = 0; g < C::GROUPS; ++g) group_fail[g] = 0;
        mbar_fence_init();
    }
    if (warp == 1) {
        tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
        tmem_relinquish_pair();
    }
    tc_fence_before();
    __syncthreads();
    cluster_sync();                              // the peer's barriers exist before anything signals them
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // Everything above touched no global memory and may overlap the previous kernel's tail.
    grid_dep_launch();
    grid_dep_wait();

    int tiles = num_m * num_n;
    uint32_t* mask = args.lens ? reinterpret_cast<uint32_t*>(smem + C::OFF_MASK) : nullptr;
    if (mask) tiles = num_n * mark_row_tiles(mask, args.lens, args.seq_n, args.M, warp, lane, C::THREADS);
    RowTiles row_tiles = {mask};                 // (each role walks its own copy)
    const WorkList<BN> list(tiles, num_n, npairs);
    const int works = list.count();

    if (warp == 0) {
        // ---------------- TMA producer (both CTAs; each loads its own halves) ----------------
        if (elect_one()) {
            uint32_t it = 0;
            bool ok = true;
            for (int i = pair; i < works && ok; i += npairs) {
                const auto wk = list.at(i);
                const int m0 = row_tiles.at(wk.row_tile) * (2 * BM) + (int)rank * BM;
                const int n0 = wk.n0 + (int)rank * (wk.width / 2);
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    const int s = it % C::STAGES;
                    const uint32_t ph = (it / C::STAGES) & 1u;
                    if (!mbar_wait(&empty[s], ph ^ 1u, abort_flag)) { ok = false; break; }
                    uint8_t* sa = smem + (size_t)s * C::STAGE_BYTES;
                    const uint32_t lead_full = map_to_cta(smem_u32(&full[s]), 0);
                    if (rank == 0) mbar_expect_tx(&full[s], 2 * A_BYTES + wk.width * BK * 2);
                    tma_load_2d_pair(sa, &tmA, lead_full, kb * BK, m0);
                    tma_load_2d_pair(sa + A_BYTES, wk.width == BN ? &tmB : &tmBh, lead_full, kb * BK, n0);
                }
            }
            // Every stage this thread filled must have been consumed (which implies its copies
            // landed and the leader's commit signals reached this CTA) before the CTA may exit.
            const uint32_t issued = it;
            for (int s = 0; s < C::STAGES && ok; ++s) {
                if ((uint32_t)s >= issued) break;
                const uint32_t last = ((issued - 1 - s) / C::STAGES) * C::STAGES + s;   // last use of stage s
                ok = mbar_wait(&empty[s], (last / C::STAGES) & 1u, abort_flag);
            }
        }
    } else if (warp == 1) {
        // ---------------- MMA issuer (leader CTA only) ----------------
        if (rank == 0 && elect_one()) {
            uint32_t it = 0, tl = 0;
            bool ok = true;
            for (int i = pair; i < works && ok; i += npairs, ++tl) {
                const uint32_t idesc = idesc_bf16(2 * BM, list.at(i).width, 0, 0);
                const uint32_t a = tl & 1u, aph = (tl >> 1) & 1u;
                if (!mbar_wait(&tempty[a], aph ^ 1u, abort_flag)) { ok = false; break; }
                tc_fence_after();
                const uint32_t d_tmem = tmem_base + a * BN;
                for (int kb = 0; kb < kblocks; ++kb, ++it) {
                    const int s = it % C::STAGES;
                    const uint32_t ph = (it / C::STAGES) & 1u;
                    if (!mbar_wait(&full[s], ph, abort_flag)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t sa = smem_u32(smem + (size_t)s * C::STAGE_BYTES);
                    const uint64_t da = smem_desc_sw128(sa, 16, 1024);
                    const uint64_t db = smem_desc_sw128(sa + A_BYTES, 16, 1024);
#pragma unroll
                    for (int k = 0; k < BK / 16; ++k)   // 32 bytes along K per MMA: +2 in the address field
                        mma_ss_pair(d_tmem, da + 2u * k, db + 2u * k, idesc, (kb | k) != 0);
                    mma_commit_pair(&empty[s], 3);      // frees the stage in both CTAs when these MMAs retire
                }
                if (ok) mma_commit_pair(&tfull[a], 3);  // accumulator complete in both CTAs
            }
            // The peer's epilogue hands accumulators back by arrivals on this CTA's barriers that nothing else orders: the last
            // one of either accumulator must have landed before this shared memory can be given to another CTA.  (They
            // come long before the epilogues' last stores, which this CTA waits for anyway.)
            for (uint32_t t = tl > 2 ? tl - 2 : 0; t < tl && ok; ++t)
                ok = mbar_wait(&tempty[t & 1u], (t >> 1) & 1u, abort_flag);
        }
    } else {
        // ---------------- epilogue (both CTAs; each drains its own 128 x BN half) ----------------
        const int q = warp & 3;                          // TMEM lane quadrant this warp may read
        const int group = (warp - 2) >> 2;
        // columns of a tile or piece that this group takes: half of it, or (WIDE) 64 (none of a piece that is narrower)
        int c_begin = 0, c_end = 0;
        auto columns = [&](int width) {
            if (WIDE) {
                c_begin = min(group * 64, width);
                c_end = min(group * 64 + 64, width);
                return;
            }
            const int split = width == BN ? C::SPLIT : BN / 4;
            c_begin = group ? split : 0;
            c_end = group ? width : split;
        };
        constexpr int BLK_COLS = 128 / (int)sizeof(OutT);            // columns in one staged 128-byte row
        constexpr int CHUNKS_PER_BLK = BLK_COLS / 32;                // 32-column TMEM loads per staged block
        const int trow = q * 32 + lane;                  // row inside this CTA's half of the tile
        const uint32_t stg_row = (uint32_t)(lane >> 3) * 1024u + (uint32_t)(lane & 7) * 128u;   // inside the warp's 32-row slab
        const int r8 = lane & 7;
        const int t128 = ((warp - 2) & 3) * 32 + lane;   // this thread's index among the 128 of its group
        const uint32_t lead_tempty[2] = {map_to_cta(smem_u32(&tempty[0]), 0), map_to_cta(smem_u32(&tempty[1]), 0)};
        uint32_t tl = 0, blk_ctr = 0;
        // Where the main loop is the longer part, the plain epilogues wait for a block to be written before they go on to
        // the next: stores in one burst hold up the operand loads.  Together / paced, us: 25216 x 2304 x 768 61.0 / 59.2,
        // 16400 x 2304 x 768 40.9 / 39.4, 16156 x 3072 x 1024 67.8 / 65.7; with less K the epilogue is:
        // 25216 x 1536 x 512 31.5 / 32.3, x 1152 x 384 23.1 / 26.8.  The other epilogues pace themselves by their arithmetic and residuals.
        const bool paced = (EPI == EPI_BIAS || EPI == EPI_BIAS_LN) && kblocks >= 12;
        // EPI_RESID: the residual of this warp's 32 rows x 32 columns, two 64-byte-swizzled boxes in turn
        // (rows past M arrive as zeros)
        uint8_t* res_buf = smem + C::OFF_RES + (warp - 2) * C::RES_WARP_BYTES;
        uint64_t* res_bar = res_full + (warp - 2) * 2;
        RowTiles ahead_tiles = row_tiles;                // the walk of what is fetched a tile ahead
        int m_next = 0, n_next = 0, map_cur = -1, map_next = -1;     // the next piece of work: its first row, this group's first column,
                                                                     // and (row map) the source row of the warp's row `lane`
        // With a row map the box is filled row by row: 16-byte asynchronous copies, a row's pieces by neighbouring
        // lanes, land in the layout the tensor map's 64-byte swizzle would give; rows past M are zero-filled.
        auto issue_res = [&](uint32_t buf, int m, int col, int map) {    // whole warp
            uint8_t* box = res_buf + buf * RES_BOX_BYTES;
            if (!args.row_map) {
                if (lane == 0) {
                    mbar_expect_tx(&res_bar[buf], RES_BOX_BYTES);
                    tma_load_2d(box, &tmRes, &res_bar[buf], col, m + q * 32);
                }
                return;
            }
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                const int r = t * 8 + (lane >> 2), piece = lane & 3, sr = __shfl_sync(0xffffffffu, map, r);
                const __nv_bfloat16* src = reinterpret_cast<const __nv_bfloat16*>(args.residual) + (size_t)(sr < 0 ? 0 : sr) * args.N + col + piece * 8;
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(box + r * 64 + ((piece ^ ((r >> 1) & 3)) << 4))), "l"(src),
                             "r"(sr < 0 ? 0 : 16) : "memory");
            }
            asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&res_bar[buf])) : "memory");
        };
        // The fp32 residual of the scoring epilogues: a warp fetches its 32 rows x 32 columns of the next chunk, the next
        // tile's first one included, with neighbouring lanes on neighbouring 16-byte pieces of a row, into registers while
        // it works on this one, and turns them over to one row per lane through the staging buffer that the results then
        // replace.  A row read per lane from global memory touches 32 lines per load instruction: FC2 50432 x 192 x 768
        // 34.2 -> 31.6 us, 25216 x 384 x 1536 40.8 -> 37.4, 25216 x 768 x 3072 98.6 -> 94.7, 16388 x 1024 x 4096 107.7 -> 105.
        // (EPI_RESID's bf16 rows stay with TMA: this way 50432 x 192 x 192 took 22.6 us instead of 19.6.)
        constexpr bool SCORE = EPI == EPI_SCORE || EPI == EPI_SCORE_STATS;
        constexpr int RES_VECS = EPI == EPI_RESID ? 4 : SCORE ? 8 : 1;   // 16-byte pieces per 32 columns of a row
        uint4 res_next[RES_VECS];
        auto load_res = [&](int m, int col) {            // rows past M: zeros
            const char* base = reinterpret_cast<const char*>(args.residual) + (size_t)col * 4 + (lane & 7) * 16;
#pragma unroll
            for (int j = 0; j < RES_VECS; ++j) {
                const int r = m + q * 32 + 4 * j + (lane >> 3);
                res_next[j] = r < args.M ? __ldg(reinterpret_cast<const uint4*>(base + (size_t)r * args.N * 4)) : make_uint4(0u, 0u, 0u, 0u);
            }
        };
        auto look_ahead = [&](int i) {
            if (!(SCORE || C::RES_TMA) || i >= works) return;
            const auto nw = list.at(i);
            m_next = ahead_tiles.at(nw.row_tile) * (2 * BM) + (int)rank * BM;
            n_next = nw.n0 + (group ? (nw.width == BN ? C::SPLIT : BN / 4) : 0);
            if (C::RES_TMA && args.row_map) {
                const int r = m_next + q * 32 + lane;
                map_next = r < args.M ? __ldg(args.row_map + r) : -1;
            }
        };
        if ((SCORE || C::RES_TMA) && pair < works) {
            look_ahead(pair);
            if (SCORE) {
                load_res(m_next, n_next);
            } else {
                issue_res(0, m_next, n_next, map_next);          // (a half has at least two chunks)
                issue_res(1, m_next, n_next + 32, map_next);
            }
        }
        uint32_t res_ctr = 0;                            // chunks of the residual walked through
        // EPI_BIAS_LN: the partial row sums of this thread's row of the NEXT tile are fetched a tile ahead into
        // registers (up to kLnPre pairs; more are read on the spot), so their way from L2 is never waited for
        constexpr int kLnPre = EPI == EPI_BIAS_LN ? 16 : 1;
        float2 ln_pre[kLnPre];
        auto ln_fetch = [&](int i) {
            const int frow = (i < works ? ahead_tiles.at(list.at(i).row_tile) : 0) * (2 * BM) + (int)rank * BM + trow;
            const bool ok = i < works && frow < args.M && args.stats_parts <= kLnPre;
            const float2* sp = reinterpret_cast<const float2*>(args.stats_in) + (size_t)(ok ? frow : 0) * args.stats_parts;
#pragma unroll
            for (int p = 0; p < kLnPre; ++p) ln_pre[p] = (ok && p < args.stats_parts) ? __ldg(sp + p) : make_float2(0.f, 0.f);
        };
        if (EPI == EPI_BIAS_LN) ln_fetch(pair);
        const int slots = args.N / 64;                   // partial sums per row: one per 64 columns
        for (int i = pair; i < works; i += npairs, ++tl) {
            const auto wk = list.at(i);
            const int m0 = row_tiles.at(wk.row_tile) * (2 * BM) + (int)rank * BM, n0 = wk.n0;
            columns(wk.width);
            const uint32_t a = tl & 1u, aph = (tl >> 1) & 1u;
            const int row = m0 + trow;
            const bool valid = row < args.M;
            // row of the block input x (EPI_SCORE, whole-block shift), possibly through the row map
            const int xrow = (SCORE && args.score_kind == 2 && args.row_map && valid) ? __ldg(args.row_map + row) : row;
            map_cur = map_next;
            look_ahead(i + npairs);
            // EPI_BIAS_LN: mean and reciprocal standard deviation of this thread's row of A from the partial
            // sums its producer left (fetched while the accumulator is still being computed)
            float ln_mu = 0.f, ln_rstd = 0.f;
            if (EPI == EPI_BIAS_LN) {
                float s1 = 0.f, s2 = 0.f;
                if (args.stats_parts <= kLnPre) {
#pragma unroll
                    for (int p = 0; p < kLnPre; ++p) { s1 += ln_pre[p].x; s2 += ln_pre[p].y; }
                    ln_fetch(i + npairs);
                } else if (valid) {
                    const float2* sp = reinterpret_cast<const float2*>(args.stats_in) + (size_t)row * args.stats_parts;
                    for (int p = 0; p < args.stats_parts; ++p) {
                        const float2 t = __ldg(sp + p);
                        s1 += t.x; s2 += t.y;
                    }
                }
                const float inv_d = 1.f / (float)args.K;
                ln_mu = s1 * inv_d;
                ln_rstd = rsqrtf(fmaxf(s2 * inv_d - ln_mu * ln_mu, 0.f) + args.ln_eps);
            }
            float st1 = 0.f, st2 = 0.f;                  // EPI_SCORE_STATS: sums over this thread's columns
            // The four warps of a group decide together whether to go on: the named
            // barriers below have no time limit, so no warp may leave the loop alone.
            // this group's slice of the bias goes to shared memory while the accumulator is still being
            // computed (the barrier below publishes it): the chunk loop then has no global read on its chain.
            // Two copies, by tile parity: a warp may still be reading the last tile's slice.
            float* bias_s = reinterpret_cast<float*>(smem + C::OFF_BIAS) + (tl & 1u) * 256;
            float* cs_s = reinterpret_cast<float*>(smem + C::OFF_COLSUM) + (tl & 1u) * 256;   // EPI_BIAS_LN only
            if (c_begin + t128 < c_end) {
                bias_s[c_begin + t128] = args.bias ? __ldg(args.bias + n0 + c_begin + t128) : 0.f;
                if (EPI == EPI_BIAS_LN) cs_s[c_begin + t128] = __ldg(args.colsum + n0 + c_begin + t128);
            }
            if (!__all_sync(0xffffffffu, mbar_wait(&tfull[a], aph, abort_flag))) group_fail[group] = 1;
            named_barrier(1 + group, 128);
            if (group_fail[group]) break;
            tc_fence_after();
            const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + a * BN;
            float sq = 0.f, sq1 = 0.f, sq2 = 0.f;
            auto hand_back = [&]() {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster_relaxed(lead_tempty[a]);
            };
            if (WIDE && c_begin == c_end) hand_back();
#pragma unroll 1
            for (int c = c_begin; c < c_end; c += 32) {
                const int cb = (c / 32) % CHUNKS_PER_BLK;            // chunk inside the staged block
                uint8_t* stg = smem + C::OFF_STG + ((warp - 2) * C::STG_PER_WARP + (C::STG_PER_WARP == 2 ? (blk_ctr & 1u) : 0u)) * STG_BYTES;
                if (!SCORE && cb == 0) {
                    // the store that last read this buffer (two blocks ago, or the last one) must be done with it
                    if (lane == 0) {
                        // (paced like the plain epilogues: 16156 x 1024 x 1024 34.0 us so, 35.2 with two stores in flight, as one before)
                        if (EPI == EPI_RESID && kblocks >= 16) tma_store_wait_read<0>();
                        else tma_store_wait_read<C::STG_PER_WARP - 1>();
                    }
                    __syncwarp();
                }
                uint4 res[RES_VECS];
                if (C::RES_TMA) {
                    // this lane's row of the chunk's box: 64 bytes, 16-byte pieces XOR-ed with address bits 7-8; then the
                    // box two chunks on takes its place.  (On a time-out the values are void, and the next tile's wait ends the loop.)
                    const uint32_t buf = res_ctr & 1u;
                    mbar_wait(&res_bar[buf], (res_ctr >> 1) & 1u, abort_flag);
                    const uint8_t* rrow = res_buf + buf * RES_BOX_BYTES + lane * 64;
#pragma unroll
                    for (int j = 0; j < RES_VECS; ++j)
                        res[j] = *reinterpret_cast<const uint4*>(rrow + ((j ^ ((lane >> 1) & 3)) << 4));
                    ++res_ctr;
                    __syncwarp();
                    if (c + 64 < c_end) issue_res(buf, m0, n0 + c + 64, map_cur);
                    else if (i + npairs < works) issue_res(buf, m_next, n_next + (c + 64 - c_end), map_next);
                } else if (SCORE) {
                    // the residual passes through the buffer that takes the results, or, where two chunks share that
                    // one (bf16 output), the second chunk's through the other, whose store must have been read by then
                    constexpr bool SHARED = CHUNKS_PER_BLK == 2;
                    uint8_t* tr = smem + C::OFF_STG + ((warp - 2) * 2 + ((blk_ctr + (uint32_t)cb) & 1u)) * STG_BYTES;
                    if (!SHARED || cb) {
                        if (lane == 0) tma_store_wait_read<SHARED ? 0 : 1>();
                        __syncwarp();
                    }
#pragma unroll
                    for (int j = 0; j < RES_VECS; ++j) {
                        const int rr = 4 * j + (lane >> 3);
                        *reinterpret_cast<uint4*>(tr + rr * 128 + (((lane ^ rr) & 7) << 4)) = res_next[j];
                    }
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < RES_VECS; ++j) res[j] = *reinterpret_cast<const uint4*>(tr + stg_row + ((j ^ r8) << 4));
                }
                uint32_t r[32];
                __syncwarp();                            // tcgen05.ld is warp-collective
                tmem_ld_32x32(taddr + c, r);
                tmem_wait_ld();
                if (c + 32 >= c_end) hand_back();        // accumulator fully read by this warp
                if (SCORE) {
                    if (c + 32 < c_end) load_res(m0, n0 + c + 32);
                    else if (i + npairs < works) load_res(m_next, n_next);
                }
                const int col = n0 + c;
                float v[32];
#pragma unroll
                for (int j = 0; j < 32; j += 4) {
                    const float4 b = *reinterpret_cast<const float4*>(bias_s + c + j);
                    if (EPI == EPI_BIAS_LN) {
                        const float4 cc = *reinterpret_cast<const float4*>(cs_s + c + j);
                        v[j] = fmaf(ln_rstd, fmaf(-ln_mu, cc.x, __uint_as_float(r[j])), b.x);
                        v[j + 1] = fmaf(ln_rstd, fmaf(-ln_mu, cc.y, __uint_as_float(r[j + 1])), b.y);
                        v[j + 2] = fmaf(ln_rstd, fmaf(-ln_mu, cc.z, __uint_as_float(r[j + 2])), b.z);
                        v[j + 3] = fmaf(ln_rstd, fmaf(-ln_mu, cc.w, __uint_as_float(r[j + 3])), b.w);
                    } else {
                        v[j] = __uint_as_float(r[j]) + b.x;
                        v[j + 1] = __uint_as_float(r[j + 1]) + b.y;
                        v[j + 2] = __uint_as_float(r[j + 2]) + b.z;
                        v[j + 3] = __uint_as_float(r[j + 3]) + b.w;
                    }
                }
                if (EPI == EPI_BIAS_GELU) {
#pragma unroll
                    for (int j = 0; j < 32; j += 2) gelu_erf2(v[j], v[j + 1]);
                } else if (EPI == EPI_RESID) {
                    float xs[32];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const uint32_t w[4] = {res[j].x, res[j].y, res[j].z, res[j].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            xs[8 * j + 2 * e] = __uint_as_float(w[e] << 16);
                            xs[8 * j + 2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
                        }
                    }
                    if (args.partials)                                // (u, v) = (SA(LN(x)), x)
                        with_dist(args.dist, [&](auto dist) {
#pragma unroll
                            for (int j = 0; j < 32; ++j) score_acc(decltype(dist)::value, v[j], xs[j], sq, sq1, sq2);
                        });
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] += xs[j];
                } else if (SCORE) {
                    float xs[32];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        xs[4 * j] = __uint_as_float(res[j].x); xs[4 * j + 1] = __uint_as_float(res[j].y);
                        xs[4 * j + 2] = __uint_as_float(res[j].z); xs[4 * j + 3] = __uint_as_float(res[j].w);
                    }
                    with_dist(args.dist, [&](auto dist) {
                        if (args.score_kind == 2) {
                            // whole-block shift: x^ - x, with the block input x read here (rows past M: zeros)
                            const uint4* x0p = reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(args.residual2) +
                                                                              (size_t)xrow * args.N + col);
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const uint4 xv = valid ? __ldg(x0p + j) : make_uint4(0u, 0u, 0u, 0u);
                                const uint32_t w[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
                                for (int e = 0; e < 4; ++e) {
                                    float* y = v + 8 * j + 2 * e;
                                    y[0] += xs[8 * j + 2 * e];
                                    y[1] += xs[8 * j + 2 * e + 1];
                                    score_acc(decltype(dist)::value, y[0], __uint_as_float(w[e] << 16), sq, sq1, sq2);
                                    score_acc(decltype(dist)::value, y[1], __uint_as_float(w[e] & 0xffff0000u), sq, sq1, sq2);
                                }
                            }
                        } else {
#pragma unroll
                            for (int j = 0; j < 32; ++j) {
                                const float m = v[j];
                                v[j] = m + xs[j];
                                score_acc(decltype(dist)::value, args.score_kind ? v[j] : m, xs[j], sq, sq1, sq2);
                            }
                        }
                    });
                }
                // stage the 32 values of this row: 16-byte pieces, XOR-swizzled like the TMA box
                if (sizeof(OutT) == 2) {
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        const int piece = cb * 4 + g;
                        const uint4 pk = make_uint4(pack_bf16(v[8 * g], v[8 * g + 1]), pack_bf16(v[8 * g + 2], v[8 * g + 3]),
                                                    pack_bf16(v[8 * g + 4], v[8 * g + 5]), pack_bf16(v[8 * g + 6], v[8 * g + 7]));
                        *reinterpret_cast<uint4*>(stg + stg_row + ((piece ^ r8) << 4)) = pk;
                        if (EPI == EPI_SCORE_STATS) {
                            // the statistics are those of the values as stored: the next block reads these bf16 numbers
                            const uint32_t w[4] = {pk.x, pk.y, pk.z, pk.w};
#pragma unroll
                            for (int e = 0; e < 4; ++e) {
                                const float y0 = __uint_as_float(w[e] << 16), y1 = __uint_as_float(w[e] & 0xffff0000u);
                                st1 += y0 + y1;
                                st2 = fmaf(y0, y0, fmaf(y1, y1, st2));
                            }
                        }
                    }
                } else {
#pragma unroll
                    for (int g = 0; g < 8; ++g)
                        *reinterpret_cast<float4*>(stg + stg_row + ((g ^ r8) << 4)) =
                            make_float4(v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]);
                }
                if (cb == CHUNKS_PER_BLK - 1) {
                    // Every warp stores its own 32 rows: no barrier between the warps of a tile.
                    fence_async_smem();                  // staged data visible to the TMA engine
                    __syncwarp();
                    if (lane == 0) {
                        if (m0 + q * 32 < args.M)        // rows past M are dropped by the tensor map's bounds
                            tma_store_2d(&tmOut, stg, col + 32 - BLK_COLS, m0 + q * 32);
                        tma_store_commit();
                        if (paced) tma_store_wait<0>();
                    }
                    ++blk_ctr;
                }
                if ((c & 32) && (SCORE || (EPI == EPI_RESID && args.partials))) {      // 64 columns done: their sums
                    const size_t pi = (size_t)row * slots + (col >> 6);
                    if (valid) {
                        if (EPI == EPI_SCORE_STATS) reinterpret_cast<float2*>(args.stats_out)[pi] = make_float2(st1, st2);
                        if (args.dist == RS_DIST_COS) {
                            args.partials[3 * pi] = sq; args.partials[3 * pi + 1] = sq1; args.partials[3 * pi + 2] = sq2;
                        } else {
                            args.partials[pi] = sq;
                        }
                    }
                    st1 = st2 = sq = sq1 = sq2 = 0.f;
                }
            }
        }
        if (lane == 0) tma_store_wait<0>();              // all output written before the CTA exits
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) atomicExch(args.status, RS_DEV_TIMEOUT);
    cluster_leave();                                     // (each CTA has seen everything that its peer signals to it: see the roles' ends)
    if (warp == 1) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
    }
}

// Tensor map over a row-major matrix [rows, cols] (cols contiguous) of 2- or 4-byte elements,
// box [box_rows, 128 bytes of columns], 128-byte swizzle.
bool make_tmap_2d(rs_ctx* ctx, CUtensorMap* out, const void* base, int elem_bytes, uint64_t rows, uint64_t cols,
                  uint32_t box_rows) {
    const unsigned long long dims[2] = {cols, rows}, strides[1] = {cols * (uint64_t)elem_bytes};
    const unsigned int box[2] = {(unsigned int)(128 / elem_bytes), box_rows};
    return tc_encode_cached(ctx, out, base, 2, elem_bytes == 2 ? 0 : 1, dims, strides, box, 128);
}

// Tensor map over the bf16 residual [rows, cols] of the projection: box [32 rows, 32 columns = 64 bytes],
// 64-byte swizzle, zeros for rows past the matrix.
bool make_tmap_res(rs_ctx* ctx, CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols) {
    const unsigned long long dims[2] = {cols, rows}, strides[1] = {cols * 2};
    const unsigned int box[2] = {32, 32};
    return tc_encode_cached(ctx, out, base, 2, 0, dims, strides, box, 64);
}

template <int BN, int EPI, typename OutT, bool WIDE = false>
cudaError_t launch_one(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmBh, const CUtensorMap& tmOut,
                       const CUtensorMap& tmRes, const GemmArgs& args, int sm_count, cudaStream_t st) {
    using C = Cfg<BN, EPI, WIDE>;
    static PerDeviceOnce attr_once;   // per instantiation: the attribute is per function and per device
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = (cudaError_t)attr_once.run(dev, [] {
        return (int)cudaFuncSetAttribute(gemm_tc_kernel<BN, EPI, OutT, WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    });
    if (e != cudaSuccess) return e;
    const int tiles = ((args.M + 2 * BM - 1) / (2 * BM)) * (args.N / BN);
    const int most = BN == 256 ? 2 * tiles : tiles, pairs = most < sm_count / 2 ? most : sm_count / 2;     // (WorkList may cut tiles in two)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * pairs, 1, 1);
    cfg.blockDim = dim3(C::THREADS, 1, 1);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // see grid_dep_wait() in the kernel
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<BN, EPI, OutT, WIDE>, tmA, tmB, tmBh, tmOut, tmRes, args);
}

// Where 64 columns to a group of epilogue warps is the faster split (see Cfg): the plain epilogues up to K = 256, GELU, whose
// arithmetic is longer, up to 384.  Halves / 64 columns each, us: QKV 50432 x 576 x 192 18.5 / 17.1, FC1 x 768 x 192 31.3 / 28.6,
// 25216 x 1024 x 256 23.8 / 22.9, x 1536 x 384 35.7 / 33.0; but QKV 25216 x 1152 x 384 22.9 / 23.5, x 2304 x 768 59.9 / 64.5,
// FC1 x 3072 x 768 78 / 84.
// (192 columns with a folded LayerNorm: the two column vectors of 256 do not fit beside sixteen staging buffers.)
bool wide_epilogue(int epi, int bn, int K) {
    if (epi == EPI_BIAS_LN) return bn == 192 && K <= 256;
    return bn >= 192 && ((epi == EPI_BIAS && K <= 256) || (epi == EPI_BIAS_GELU && K <= 384));
}

// Tile width (256, 192 or 128 columns per pair): the one whose rounds over the SM pairs cost least (a round of 192- or
// 128-wide tiles 0.83 or 0.58 of one of 256-wide ones, a last round of halves 0.65; see WorkList).
int pick_bn(long long M, int N, int sm_count) {
    const long long pairs = sm_count / 2, mt = (M + 2 * BM - 1) / (2 * BM);
    const int widths[3] = {256, 192, 128}, round_cost[3] = {100, 83, 58};
    int best = 128;
    long long best_cost = -1;
    for (int i = 0; i < 3; ++i) {
        if (N % widths[i]) continue;
        const long long tiles = mt * (N / widths[i]), full = tiles / pairs, rest = tiles - full * pairs;
        const long long cost = full * round_cost[i] + (rest == 0 ? 0 : widths[i] == 256 && rest * 2 <= pairs ? 65 : round_cost[i]);
        if (best_cost < 0 || cost < best_cost) { best_cost = cost; best = widths[i]; }
    }
    return best;
}

}  // namespace

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

bool tc_encode_cached(rs_ctx* ctx, CUtensorMap* out, const void* base, int rank, int dtype, const unsigned long long* dims,
                      const unsigned long long* strides, const unsigned int* box, int swizzle_bytes) {
    if (!ctx->encode_tiled || rank < 2 || rank > 4) return false;
    rs_tmap_key key;
    memset(&key, 0, sizeof(key));
    key.base = base; key.rank = (unsigned)rank; key.dtype = (unsigned)dtype; key.swizzle = (unsigned)swizzle_bytes;
    for (int i = 0; i < rank; ++i) { key.dims[i] = dims[i]; key.box[i] = box[i]; }
    for (int i = 0; i + 1 < rank; ++i) key.strides[i] = strides[i];
    unsigned long long h = (unsigned long long)(uintptr_t)base * 0x9E3779B97F4A7C15ull;
    for (int i = 0; i < rank; ++i) h = (h ^ key.dims[i] ^ ((unsigned long long)key.box[i] << 40)) * 0x9E3779B97F4A7C15ull;
    h ^= (unsigned long long)swizzle_bytes << 8 | (unsigned long long)dtype;
    // eight neighbouring slots are probed; a new map takes the first free one of them, else the home slot
    const unsigned home = (unsigned)((h >> 32) % kTmapSlots);
    rs_tmap_slot* free_slot = nullptr;
    for (unsigned pr = 0; pr < 8; ++pr) {
        rs_tmap_slot& c = ctx->tmaps[(home + pr) % kTmapSlots];
        if (c.valid && memcmp(&c.key, &key, sizeof(key)) == 0) {
            *out = c.map;
            ctx->tmap_hits += 1;
            return true;
        }
        if (!c.valid && !free_slot) free_slot = &c;
    }
    rs_tmap_slot& slot = free_slot ? *free_slot : ctx->tmaps[home];
    EncodeTiledFn fn = reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled);
    cuuint64_t d[4], st[3];
    cuuint32_t bx[4], estr[4] = {1, 1, 1, 1};
    for (int i = 0; i < rank; ++i) { d[i] = dims[i]; bx[i] = box[i]; }
    for (int i = 0; i + 1 < rank; ++i) st[i] = strides[i];
    const CUtensorMapSwizzle sw = swizzle_bytes == 128 ? CU_TENSOR_MAP_SWIZZLE_128B : swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                                                                         : CU_TENSOR_MAP_SWIZZLE_NONE;
    CUtensorMap m;
    if (fn(&m, dtype == 0 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank,
           const_cast<void*>(base), d, st, bx, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return false;
    slot.map = m; slot.key = key; slot.valid = 1;
    ctx->tmap_misses += 1;
    *out = m;
    return true;
}

void* tc_get_encode_fn() {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
        return nullptr;
    return fn;
}

// Output widths: whole tiles of 128 (256) or of 192 columns, so every D that is a multiple of 128 or of 192
// (192 = three heads: DeiT-T's QKV, projection and MLP are 576, 192 and 768 wide).  Such a block used to fall
// to the fp32-FMA kernels: 12 blocks of D = 192 over 256 x 197 tokens took 21.5 ms there.
bool gemm_tc_supported(long long M, int N, int K) {
    return M >= 1 && M < (1ll << 31) && N >= 128 && ((N % 128) == 0 || (N % 192) == 0) && K >= 64 && (K % 64) == 0;
}

int gemm_tc_score_parts(int N) { return N / 64; }

cudaError_t launch_gemm_tc(rs_ctx* ctx, int epi, const void* A, const void* W, const float* bias,
                           const void* residual, const void* residual2, const int32_t* row_map, void* out, rs_dtype out_dtype,
                           float* partials, int score_kind, int dist, long long M, int N, int K, cudaStream_t st,
                           const GemmLn* ln, bool weights_ready, const GemmRows* rows) {
    if (!ctx->encode_tiled) return cudaErrorNotSupported;
    if (ln && epi == EPI_SCORE && ln->stats_out && out_dtype == RS_BF16) epi = EPI_SCORE_STATS;
    if (ln && epi == EPI_BIAS && ln->stats_in) epi = EPI_BIAS_LN;
    const few::SmallPlan small = few::gemm_small_plan(epi, M, N, K, ctx->sm_count);
    const int bn = small.use ? few::kSmallBN : pick_bn(M, N, ctx->sm_count);
    const int out_bytes = (epi == EPI_RESID || (epi == EPI_SCORE && out_dtype == RS_F32)) ? 4 : 2;
    if (epi == EPI_SCORE_STATS && ln->stats_parts_out) *ln->stats_parts_out = gemm_tc_score_parts(N);
    CUtensorMap tmA, tmB, tmBh, tmOut, tmRes;
    if (epi == EPI_RESID && !row_map && !small.use && !make_tmap_res(ctx, &tmRes, residual, (uint64_t)M, (uint64_t)N)) return cudaErrorInvalidValue;
    if (!make_tmap_2d(ctx, &tmA, A, 2, (uint64_t)M, (uint64_t)K, BM) ||
        !make_tmap_2d(ctx, &tmB, W, 2, (uint64_t)N, (uint64_t)K, (uint32_t)(small.use ? bn : bn / 2)) ||
        (bn == 256 && !make_tmap_2d(ctx, &tmBh, W, 2, (uint64_t)N, (uint64_t)K, 64)) ||
        (!small.use && !make_tmap_2d(ctx, &tmOut, out, out_bytes, (uint64_t)M, (uint64_t)N, 32)))
        return cudaErrorInvalidValue;
    if (bn != 256) tmBh = tmB;                       // unused: only 256-wide tiles are cut
    if (epi != EPI_RESID || row_map) tmRes = tmOut;  // unused by the other epilogues and by the mapped residual
    GemmArgs args;
    args.M = (int)M; args.N = N; args.K = K; args.bias = bias; args.residual = residual;
    args.residual2 = residual2; args.row_map = row_map; args.partials = partials; args.score_kind = score_kind; args.dist = dist; args.status = ctx->d_status;
    args.stats_out = ln ? ln->stats_out : nullptr;
    args.stats_in = ln ? ln->stats_in : nullptr;
    args.colsum = ln ? ln->colsum : nullptr;
    args.stats_parts = ln ? ln->stats_parts : 0;
    args.ln_eps = ln ? ln->eps : 0.f;
    const bool skips = rows && rows->lens && (M + 2 * BM - 1) / (2 * BM) <= kMaskTiles;
    args.lens = skips ? rows->lens : nullptr;
    args.seq_n = skips ? rows->seq_n : 0;
    if (small.use) return few::launch_gemm_small(epi, tmA, tmB, args, small.splits, out, out_dtype, weights_ready, st);
    const int sms = ctx->sm_count;
    if (wide_epilogue(epi, bn, K)) {
        if (epi == EPI_BIAS_LN) return launch_one<192, EPI_BIAS_LN, __nv_bfloat16, true>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st);
        if (epi == EPI_BIAS_GELU)
            return bn == 256 ? launch_one<256, EPI_BIAS_GELU, __nv_bfloat16, true>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st)
                             : launch_one<192, EPI_BIAS_GELU, __nv_bfloat16, true>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st);
        return bn == 256 ? launch_one<256, EPI_BIAS, __nv_bfloat16, true>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st)
                         : launch_one<192, EPI_BIAS, __nv_bfloat16, true>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st);
    }
#define RS_GEMM_CASE(E, T)                                                                       \
    return bn == 256   ? launch_one<256, E, T>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st)           \
           : bn == 192 ? launch_one<192, E, T>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st)           \
                       : launch_one<128, E, T>(tmA, tmB, tmBh, tmOut, tmRes, args, sms, st)
    switch (epi) {
        case EPI_BIAS: RS_GEMM_CASE(EPI_BIAS, __nv_bfloat16);
        case EPI_BIAS_GELU: RS_GEMM_CASE(EPI_BIAS_GELU, __nv_bfloat16);
        case EPI_RESID: RS_GEMM_CASE(EPI_RESID, float);
        case EPI_SCORE:
            if (out_dtype == RS_F32) RS_GEMM_CASE(EPI_SCORE, float);
            RS_GEMM_CASE(EPI_SCORE, __nv_bfloat16);
        case EPI_SCORE_STATS: RS_GEMM_CASE(EPI_SCORE_STATS, __nv_bfloat16);
        case EPI_BIAS_LN: RS_GEMM_CASE(EPI_BIAS_LN, __nv_bfloat16);
    }
#undef RS_GEMM_CASE
    return cudaErrorInvalidValue;
}

// Which blocks take their projection and MLP as one kernel: those of 192 columns with more than two tiles' rows.  Fewer rows
// are done sooner by the four kernels for few rows, which spread a tile's columns over the SMs.  Whole pruned forwards of 12
// blocks (hidden width 768, 20 % dropped three times, captured in a graph below 2500 rows), four kernels / one, us: 1 x 197 388 / 399 and 2 x 197
// 393 / 404 with the line left out; 3 x 173 398 / 395, 5 x 128 400 / 406, 4 x 197 420 / 417, 1 x 785 494 / 497, 6 x 160 405 / 403, 8 x 197 444 / 403,
// 16 x 197 478 / 427, 32 x 197 544 / 458, 1 x 1569 622 / 589, 256 x 197 1301 / 1056.  Without pruning 3 x 173 385 / 385, 1 x 700 482 / 493, 4 x 197
// 435 / 400.  One block a call, hidden width 768: 4 x 197 43.2 / 42.8, 8 x 197 44.1 / 43.5, 16 x 197 50.2 / 44.7; captured in a graph, where a
// launch costs less, up to 2000 rows are the slower for it: 3 x 190 39.0 / 39.3, 4 x 197 39.5 / 40.8, 8 x 197 40.6 / 41.6, 16 x 197 46.0 / 42.1.
// Narrower hidden layers leave less to do in the chunks and gain at all of these: 128 3 x 190 40.7 / 33.6, 4 x 197 42.2 / 34.9; 512 39.9 / 36.8,
// 41.5 / 38.2 (640 at 8 x 197 39.6 / 40.5).
// A tile in mid-launch takes 28000 to 30000 cycles, of which the tensor pipe needs 10400: waiting for x 1300 to 2400, x' and LN(x') 4900, its
// hand-over 1000, the first chunk 3600, five more 2100 each (GELU and its hand-overs), the wait for O 1450, the output 5000 to
// 5800; the first tile of a launch 41000.  Over 197 tiles the schedulers issue in 39 % of the cycles, with the ALU 23, the special-function unit 18 and
// the FMA pipe 17 % busy.  With x' in tensor memory and chunks of 64 columns, two of them under way, a chunk's chain took
// 1500 cycles for half the columns and 256 x 197 1059 us where this form took 1044 (before its hand-over at cluster scope).
bool tail_tc_use(long long T, int D, int Dm) {
    return T > 512 && D == tail::D && Dm >= tail::C && Dm % tail::C == 0 && Dm <= tail::kMaxHidden && T < (1ll << 31);
}
int tail_tc_parts() { return tail::kParts; }

cudaError_t launch_tail_tc(rs_ctx* ctx, const TailCall& c, cudaStream_t st) {
    if (!ctx->encode_tiled) return cudaErrorNotSupported;
    CUtensorMap tmO, tmX, tmWo, tmW1, tmW2;
    constexpr int D = tail::D;
    if (!make_tmap_2d(ctx, &tmO, c.o, 2, (uint64_t)c.T, D, 128) || !make_tmap_2d(ctx, &tmWo, c.wo, 2, D, D, D / 2) ||
        !make_tmap_2d(ctx, &tmW1, c.w1, 2, (uint64_t)c.Dm, D, tail::C / 2) || !make_tmap_2d(ctx, &tmW2, c.w2, 2, D, (uint64_t)c.Dm, D / 2) ||
        (!c.row_map && !make_tmap_2d(ctx, &tmX, c.x, 2, (uint64_t)c.T, D, 128)))
        return cudaErrorInvalidValue;
    if (c.row_map) tmX = tmO;                        // unused: x is read through the map
    tail::TailArgs a;
    a.T = (int)c.T; a.Dm = c.Dm; a.bo = c.bo; a.ln_g = c.ln_g; a.ln_b = c.ln_b; a.b1 = c.b1; a.b2 = c.b2; a.ln_eps = c.ln_eps;
    a.x = reinterpret_cast<const __nv_bfloat16*>(c.x); a.row_map = c.row_map; a.out = c.out;
    a.attn_partials = c.attn_partials; a.partials = c.partials; a.score_kind = c.score_kind; a.dist = c.dist;
    a.stats_out = c.out_dtype == RS_BF16 ? c.stats_out : nullptr;
    if (a.stats_out && c.stats_parts_out) *c.stats_parts_out = tail::kParts;
    const bool skips = c.rows && c.rows->lens && (c.T + 255) / 256 <= kMaskTiles;
    a.lens = skips ? c.rows->lens : nullptr;
    a.seq_n = skips ? c.rows->seq_n : 0;
    a.status = ctx->d_status;
    return c.out_dtype == RS_F32 ? tail::launch<float>(tmO, tmX, tmWo, tmW1, tmW2, a, ctx->sm_count, st)
                                 : tail::launch<__nv_bfloat16>(tmO, tmX, tmWo, tmW1, tmW2, a, ctx->sm_count, st);
}

}  // namespace rs
