// Fused attention on the tensor cores (Eq. sa): three query tiles per CTA.
//
// Same scheme as rs_attn_tc.cu -- S = Q K^T by tcgen05.mma into tensor memory, a softmax warpgroup
// per query tile with a row per thread, P as the tensor-memory A operand of O += P V, lazy
// rescaling -- with the work cut finer so that a third stream fits: key tiles of 64 instead of 128
// keys, hence per query tile 64 columns of S, 32 of P and 64 of O, 480 of the 512 tensor-memory
// columns for three tiles.  With head dimension 64 the special-function unit (the exponentials)
// bounds the kernel, and what keeps that unit from saturating is the serial chain of each
// softmax warp; three warps per scheduler instead of two fill more of its gaps.
// The softmax warps' loop over whole key tiles carries nothing else: no masks, no rescaling of O, no second form of the
// exponentials.  A tile that needs any of these goes through a second, short piece of code (16 columns at a time from tensor
// memory).  What a loop that long also carries is paid for at every tile and in instruction fetches (32 KB at full rate,
// then a third of it): with masked and rescaling forms out of the loop 4 x 16 x 4097 369 -> 337 us, 16 x 12 x 1569 181 -> 160, 32 x 16 x 577 82.8 ->
// 72.3, 64 x 12 x 197 30.5 -> 24.1 (339, 163, 78 and 25.9 with the maximum of the first 128 keys, see walk).  A key tile of three query tiles takes about 1980 cycles
// (647 000 SM cycles by ncu for five items of 65, their ends included), of which 1250 are exponentials.
// An item is three consecutive 128-row query tiles of one (sample, head), which share the K/V
// tiles streamed through the TMA ring, or of consecutive (sample, head)s.
// SPLIT: the weights go to the second product as a bf16 and the bf16 of what that left over, 16 bits of mantissa instead of 8,
// for the blocks that used to have fp32 weights (see rs_block_fwd).  The second parts take columns of the S that they came
// from, so the next Q K^T waits for P V there.  (One after the other through the columns of P, with S handed back early, every key tile went
// to the tensor core and back twice: DeiT-T, 256 images, 1042 -> 992 us for the pass, twelve blocks of 2 x 197 x 192 394 -> 383.)
#include <math.h>

#include "rs_internal.h"
#include "rs_attn.cuh"
#include "rs_device.cuh"
#include "rs_once.h"
#include "rs_tc.cuh"

namespace rs {

namespace {

using namespace tc;
using namespace attn;

constexpr int BQ = 128, BKV = 64, DH = 64, NG = 3;
constexpr int Q_BYTES = BQ * DH * 2;            // 16 KB: a [128, 64] bf16 tile
constexpr int KV_BYTES = BKV * DH * 2;          // 8 KB: a [64, 64] bf16 tile
constexpr int NS = 5;                           // K/V ring stages
constexpr int kThreads = 512;                   // warps 0-3 / 4-7 / 8-11: softmax of tile 0 / 1 / 2, warp 12: TMA, warp 13: Q K^T, warp 14: P V
// the fourth warpgroup (TMA, MMA and two idle warps) hands registers to the three softmax warpgroups
constexpr int kLaunchRegs = 128, kSoftmaxRegs = 152, kOtherRegs = 56;
static_assert(384 * kSoftmaxRegs + 128 * kOtherRegs <= kThreads * kLaunchRegs, "register pool of the CTA");
constexpr int kSCol = 0, kPCol = NG * BKV, kOCol = kPCol + NG * (BKV / 2);   // S 0..191, P 192..287, O 288..479
constexpr int kTmemCols = 512;
constexpr float kRescaleGap = 8.f;              // log2 units the tile maximum may exceed the running one
// shared memory: Q[2 buffers][NG] | K[NS] | V[NS] | output staging | barriers
constexpr int OFF_Q = 0, OFF_K = 2 * NG * Q_BYTES, OFF_V = OFF_K + NS * KV_BYTES;
constexpr int OFF_OST = OFF_V + NS * KV_BYTES;  // output staging: 12 softmax warps x 32 rows x 128 bytes
constexpr int OFF_BAR = OFF_OST + 4 * NG * 4096;
constexpr int kMaxSamples = 256;                 // of a launch with a count per sample
constexpr int OFF_SAMPLES = OFF_BAR + 512;      // what those launches keep of the counts
constexpr size_t kSmem = (size_t)OFF_SAMPLES + 4 * (kMaxSamples + 3) + kMaxSamples + 1024 /*alignment slack*/;
static_assert(kOCol + NG * DH <= kTmemCols, "tensor-memory columns");
static_assert(kSmem <= 232448, "shared memory of one CTA");

// The work: the query tiles of all (sample, head)s in a row, three to an item, whichever heads they belong to; an item that
// meets a head's end takes two K/V streams, a tile of each in turn (with one query tile per head, three).  CTA c takes
// the items c, c + G, ...  The tiles of the last round are spread over the CTAs, `rest` to an item.  Where the plan says so the
// last `cut` query tiles of every head come after all others, one to an item with the keys cut in three: each warpgroup
// takes a third of them for the same queries, and the first merges the three results, which lie in the same tensor-memory
// lanes.  (Always the same tiles of every head: a sample's result does not depend on its place in the batch.)
// RAGGED: items of one sample after the other, the longest first (`order`, `first_item`), each with its own count of tokens.
struct Attn3Args {
    int N, H, B;
    int nt, tiles;           // query tiles per (sample, head) that see all keys at once, and in all
    int cut;                 // and those with the keys cut in three
    uint32_t by_nt, by_h, by_cut;    // 2^32 over nt, H and cut, rounded down: see divide()
    int full, rest;          // items of three tiles that fill whole rounds, tiles per item after those
    int n_whole, n_items;    // items before those with the keys cut, and in all
    const int* lens;         // RAGGED: [B], sample b attends over its first lens[b] tokens only (clamped to 1 .. N)
    __nv_bfloat16* out;      // RAGGED: [B, N, H, 64] where the caller sees the rows past them: zeros; else null
    float scale_log2;        // scale * log2(e)
    int* status;
};

// n / d and its remainder for d's reciprocal as above: the product is the quotient or one less.
__device__ __forceinline__ int divide(int n, int d, uint32_t by_d, int& rest) {
    int quot = (int)__umulhi((uint32_t)n, by_d);
    rest = n - quot * d;
    if (rest >= d) { rest -= d; ++quot; }
    return quot;
}

struct Item3 {
    int b, h, q;             // sample, head and query tile of tile 0
    int ng;                  // query tiles present: 1 .. 3
    int split;               // tiles of the first head; the others belong to the next one (or ones)
    int n, nt, nkv;          // tokens of the sample, its query tiles and key tiles
    int third;               // keys cut in three: key tiles to a warpgroup (the last one may have fewer, or none); else 0
    // how many heads after the item's first one tile g belongs to; whether it is the first or the last tile that a K/V tile serves
    __device__ __forceinline__ int stream(int g) const { return nt == 1 ? g : g >= split; }
    __device__ __forceinline__ bool starts(int g) const { return g == 0 || g == split || nt == 1; }
    __device__ __forceinline__ bool ends(int g) const { return g == ng - 1 || g == split - 1 || nt == 1; }
};
// RAGGED: what the CTA knows of the samples, in shared memory.
struct Samples {
    int items, per;                                      // items in all; query tiles to an item
    int first_item[kMaxSamples + 1];
    unsigned char order[kMaxSamples];
};
static_assert(OFF_SAMPLES + sizeof(Samples) + 1024 <= kSmem, "room for the samples");
__device__ __forceinline__ int sample_len(const Attn3Args& a, int b) { return min(max(__ldg(a.lens + b), 1), a.N); }

template <bool RAGGED, bool CUT> __device__ __forceinline__ Item3 decode_item3(const Attn3Args& a, const Samples* sm, int w) {
    Item3 it;
    if constexpr (RAGGED) {
        int lo = 0, hi = a.B;                            // first_item[lo] <= w < first_item[hi]
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (sm->first_item[mid] <= w) lo = mid;
            else hi = mid;
        }
        it.b = sm->order[lo];
        it.n = sample_len(a, it.b);
        it.nt = (it.n + BQ - 1) / BQ;
        const int tile = (w - sm->first_item[lo]) * sm->per;
        it.ng = min(sm->per, a.H * it.nt - tile);
        it.h = tile / it.nt;
        it.q = tile - it.h * it.nt;
    } else {
        it.n = a.N;
        it.nt = a.nt;
        int bh;
        if (!CUT || w < a.n_whole) {
            const int tile = w < a.full ? w * NG : a.full * NG + (w - a.full) * a.rest;
            it.ng = min(w < a.full ? NG : a.rest, a.tiles - tile);
            bh = divide(tile, a.nt, a.by_nt, it.q);
        } else {
            it.ng = 1;
            bh = divide(w - a.n_whole, a.cut, a.by_cut, it.q);
            it.q += a.nt;
        }
        it.b = divide(bh, a.H, a.by_h, it.h);
    }
    it.split = CUT && w >= a.n_whole ? it.ng : min(it.ng, it.nt - it.q);     // (two or more tiles to a head: three meet one boundary at most)
    it.nkv = (it.n + BKV - 1) / BKV;
    it.third = CUT && w >= a.n_whole ? (it.nkv + NG - 1) / NG : 0;
    return it;
}

// Maximum of N columns of a row of S in registers.
template <int N> __device__ __forceinline__ float row_max(const uint32_t (&r)[N]) {
    float m[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) m[c] = -INFINITY;
#pragma unroll
    for (int i = 0; i < N; i += 16)                 // eight independent chains: latency, not count, is the cost
#pragma unroll
        for (int c = 0; c < 8; ++c) m[c] = max3(m[c], __uint_as_float(r[i + 2 * c]), __uint_as_float(r[i + 2 * c + 1]));
    return max3(max3(m[0], m[1], m[2]), max3(m[3], m[4], m[5]), fmaxf(m[6], m[7]));
}

// p_i = exp2(s_i * sl + mneg) for N values of a row from FROM on, packed to bf16 pairs in place (r[FROM / 2 ...) on return);
// returns the sum of the unrounded p_i.
// Six pairs of the 32 of a key tile go through the FMA pipes: the special-function unit (8 cycles per warp and exponential) is the
// busiest pipe of this kernel, and its idle time does not line up between the three warps of a scheduler.  4 x 16 x
// 4097, an earlier form: 380 us with none, 379 / 371 / 368 / 371 / 382 with 2 / 5 / 6 / 8 / 11 pairs, 435 with all second pairs of four
// elements.  Which six hardly matters (330 to 345 us in the present form).
// SPLIT: lo gets what the bf16s in r leave of the p_i, as bf16 pairs (and the exponentials all go to the special-function
// unit, which is not the busiest pipe there).
template <int FROM, int N, bool SPLIT>
__device__ __forceinline__ float exp_pass(uint32_t (&r)[BKV], uint32_t (&lo)[SPLIT ? BKV / 2 : 1], float sl, float mneg) {
    const uint64_t sl2 = pack2(sl, sl), mneg2 = pack2(mneg, mneg);
    uint64_t l01 = pack2(0.f, 0.f), l23 = l01;
#pragma unroll
    for (int i = FROM; i < FROM + N; i += 4) {
        float x0, x1, x2, x3;
        unpack2(ffma2(pack2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), sl2, mneg2), x0, x1);
        unpack2(ffma2(pack2(__uint_as_float(r[i + 2]), __uint_as_float(r[i + 3])), sl2, mneg2), x2, x3);
        const float p0 = ex2(x0), p1 = ex2(x1);
        float p2, p3;
        constexpr int kByFma = 0x29;                     // which of eight consecutive groups of four send their second pair there
        if (!SPLIT && ((kByFma >> ((i / 4) % 8)) & 1)) ex2_pair_fma(pack2(x2, x3), p2, p3);
        else { p2 = ex2(x2); p3 = ex2(x3); }
        l01 = fadd2(l01, pack2(p0, p1));
        l23 = fadd2(l23, pack2(p2, p3));
        const uint32_t h01 = pack_bf16(p0, p1), h23 = pack_bf16(p2, p3);
        if constexpr (SPLIT) {
            lo[i >> 1] = pack_bf16(p0 - __uint_as_float(h01 << 16), p1 - __uint_as_float(h01 & 0xffff0000u));
            lo[(i >> 1) + 1] = pack_bf16(p2 - __uint_as_float(h23 << 16), p3 - __uint_as_float(h23 & 0xffff0000u));
        }
        r[i >> 1] = h01;
        r[(i >> 1) + 1] = h23;
    }
    float a, b, c, d;
    unpack2(l01, a, b);
    unpack2(l23, c, d);
    return (a + b) + (c + d);
}

// CUT: there are items with the keys cut in three.  (Without, the loops carry nothing of them: 4 x 16 x 3073 205 -> 198 us.)
// FIRST: there are query tiles that see more than 128 keys at once, whose running maximum starts from the first two key tiles (two_first).
// (Without, a short sequence and one with all query tiles cut carry nothing of them: twelve blocks of one image, ViT-B, 477 -> 472 us, where every
// launch fetches the kernel's instructions anew; and with it known, 4 x 16 x 4097 338.5 -> 335.4, 16 x 12 x 539 33.4 -> 32.6.)
template <bool SPLIT, bool RAGGED, bool CUT, bool FIRST>
__global__ void __launch_bounds__(kThreads, 1)
attn_tc3_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO, const Attn3Args args) {
    static_assert(!RAGGED || (!SPLIT && !CUT), "neither comes with a count per sample");
    static_assert(!FIRST || !SPLIT, "weights of 16 bits");
    constexpr bool WHOLE = !CUT || FIRST || SPLIT;       // (else all query tiles have their keys cut)
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + OFF_BAR);
    uint64_t* q_full = bars;                 // [2] Q tiles of the item landed in buffer 0 / 1
    uint64_t* q_empty = bars + 2;            // [2] every Q K^T of the item in that buffer retired
    uint64_t* k_full = bars + 4;             // [NS] K tile landed
    uint64_t* v_full = k_full + NS;          // [NS] V tile landed
    uint64_t* k_empty = k_full + 2 * NS;     // [NS] every Q K^T reading the K stage retired
    uint64_t* v_empty = k_full + 3 * NS;     // [NS] every P V reading the V stage retired
    uint64_t* s_full = k_full + 4 * NS;      // [NG] S of the tile complete in tensor memory
    uint64_t* p_ready = s_full + NG;         // [NG] P written (one arrival per softmax warp)
    uint64_t* o_done = s_full + 2 * NG;      // [NG] O += P V retired
    uint64_t* s_free = s_full + 3 * NG;      // [NG] S row in registers, columns reusable (one arrival per warp)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(s_full + 4 * NG);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

    if (threadIdx.x == 0) {
        prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); prefetch_tmap(&tmO);
        for (int i = 0; i < 2; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); }
        for (int s = 0; s < NS; ++s) { mbar_init(&k_full[s], 1); mbar_init(&v_full[s], 1); mbar_init(&k_empty[s], 1); mbar_init(&v_empty[s], 1); }
        for (int g = 0; g < NG; ++g) { mbar_init(&s_full[g], 1); mbar_init(&p_ready[g], 4); mbar_init(&o_done[g], 1); mbar_init(&s_free[g], 4); }
        *abort_flag = 0;
        mbar_fence_init();
    }
    if (warp == 13) {
        tmem_alloc(tmem_slot, kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = *tmem_slot;
    // Everything above touched no global memory and may overlap the previous kernel's tail.
    grid_dep_launch();
    grid_dep_wait();
    Samples* samples = RAGGED ? reinterpret_cast<Samples*>(smem + OFF_SAMPLES) : nullptr;
    if constexpr (RAGGED) {
        // Samples by key tiles, the most first (its place: how many come before it), and the items before each; a warp to a
        // sample, whose lanes keep what they compare it with in registers.  (A thread to a sample: 30 x 89 tokens 4.7 us for the loops.
        // Tiles and items worked out at each comparison: 256 x 3 x 129 30.6 us instead of
        // 18.6, 256 x 3 x 197 38.3 of 25.9, 64 x 12 x 197 24.0 of 23.0.)
        static_assert(kMaxSamples <= kThreads && kMaxSamples <= 256, "a thread to a sample's count, its index in eight bits");
        constexpr int PER_LANE = kMaxSamples / 32;
        uint32_t* keys = reinterpret_cast<uint32_t*>(smem + OFF_OST);        // (not in use yet)
        int* tiles = reinterpret_cast<int*>(keys + kMaxSamples);
        if (threadIdx.x < kMaxSamples) {
            const int b = threadIdx.x, len = b < args.B ? sample_len(args, b) : 0;
            keys[b] = b < args.B ? min((uint32_t)(len + BKV - 1) / BKV, 0xffffffu) << 8 | (uint32_t)(kMaxSamples - 1 - b) : 0u;
            tiles[b] = args.H * ((len + BQ - 1) / BQ);
        }
        __syncthreads();
        uint32_t key[PER_LANE];
        int items[PER_LANE], n1 = 0, n2 = 0, n3 = 0;                         // items in all with one, two or three query tiles each
#pragma unroll
        for (int i = 0; i < PER_LANE; ++i) {
            key[i] = keys[lane + 32 * i];
            items[i] = tiles[lane + 32 * i];
            n1 += items[i];
            n2 += (items[i] + 1) / 2;
            n3 += (items[i] + 2) / 3;
        }
        // The fewest rounds, an item of one, two or three weighed by what a key tile of it takes (0.62, 0.80 and 1.03 us, and 0.85 for two, since more
        // items also meet more heads' ends: 40 x 12 x 333 tokens with five rounds of two 39.3 us, with four of three 37.3).  With three wherever two left
        // a CTA a second item, and two wherever one did, whatever the items of short samples came to: 24 x 12 x 256 (576 tiles) 19.4 us, so 17.0;
        // 90 x 3 x 134 (276 tiles, in 180 items of two or 93 of three) 13.3, so 11.0.
        auto rounds = [](int n) { return (int)(((unsigned)n + gridDim.x - 1) / gridDim.x); };
        const float t1 = 0.62f * rounds(__reduce_add_sync(0xffffffffu, n1)), t2 = 0.85f * rounds(__reduce_add_sync(0xffffffffu, n2)), t3 = 1.03f * rounds(__reduce_add_sync(0xffffffffu, n3));
        const int per = t1 <= t2 && t1 <= t3 ? 1 : t2 <= t3 ? 2 : 3;
        auto items_of = [&](int t) { return per == 1 ? t : per == 2 ? (t + 1) / 2 : (t + 2) / 3; };
#pragma unroll
        for (int i = 0; i < PER_LANE; ++i) items[i] = items_of(items[i]);
        for (int b = warp; b < args.B; b += kThreads / 32) {
            const uint32_t mine = keys[b];
            int place = 0, before = 0;
#pragma unroll
            for (int i = 0; i < PER_LANE; ++i)
                if (key[i] > mine) { ++place; before += items[i]; }
            place = __reduce_add_sync(0xffffffffu, place);
            before = __reduce_add_sync(0xffffffffu, before);
            if (lane == 0) {
                samples->order[place] = (unsigned char)b;
                samples->first_item[place] = before;
                if (place == args.B - 1) {
                    samples->items = samples->first_item[args.B] = before + items_of(tiles[b]);
                    samples->per = per;
                }
            }
        }
        __syncthreads();
    }
    const int n_items = RAGGED ? samples->items : args.n_items;

    if (warp >= 12) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kOtherRegs));
    if (warp == 12) {
        // ---------------- TMA producer ----------------
        if (elect_one()) {
            uint32_t kv_it = 0, item_n = 0;
            bool ok = true;
            for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x, ++item_n) {
                const Item3 it = decode_item3<RAGGED, CUT>(args, samples, w);
                const uint32_t qb = item_n & 1u;
                if (!mbar_wait(&q_empty[qb], ((item_n >> 1) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                mbar_expect_tx(&q_full[qb], it.ng * Q_BYTES);
                auto next = [&](int& b, int& h) { if (++h == args.H) { h = 0; ++b; } };      // the next (sample, head)
                for (int g = 0, b = it.b, h = it.h; g < it.ng; ++g) {
                    if (g && it.starts(g)) next(b, h);
                    tma_load_4d(smem + OFF_Q + (qb * NG + g) * Q_BYTES, &tmQ, &q_full[qb], 0, h, (it.q + g - it.stream(g) * it.nt) * BQ, b);
                }
                const int streams = it.third ? NG : it.stream(it.ng - 1) + 1, steps = it.third ? it.third : it.nkv;
                for (int j = 0; j < steps && ok; ++j)
                    for (int sm = 0, b = it.b, h = it.h; sm < streams; ++sm, ++kv_it) {
                        const int t = j + sm * it.third;
                        if (t >= it.nkv) break;          // (the last third may be shorter)
                        const int s = kv_it % NS;
                        if (!mbar_wait(&k_empty[s], ((kv_it / NS) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(&k_full[s], KV_BYTES);
                        tma_load_4d(smem + OFF_K + s * KV_BYTES, &tmK, &k_full[s], 0, h, t * BKV, b);
                        if (!mbar_wait(&v_empty[s], ((kv_it / NS) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
                        mbar_expect_tx(&v_full[s], KV_BYTES);
                        tma_load_4d(smem + OFF_V + s * KV_BYTES, &tmV, &v_full[s], 0, h, t * BKV, b);
                        if (!it.third) next(b, h);
                    }
            }
            // every copy started here must have landed before the CTA exits
            for (uint32_t n = item_n > 2 ? item_n - 2 : 0; n < item_n && ok; ++n)
                ok = mbar_wait(&q_full[n & 1u], (n >> 1) & 1u, abort_flag);
            for (uint32_t t = kv_it > NS ? kv_it - NS : 0; t < kv_it && ok; ++t)
                ok = mbar_wait(&k_full[t % NS], (t / NS) & 1u, abort_flag) && mbar_wait(&v_full[t % NS], (t / NS) & 1u, abort_flag);
        }
    } else if (warp == 13) {
        // ---------------- Q K^T issuer: S_g = Q_g K^T, both operands K-major ----------------
        // It runs ahead of the softmax warps as far as the S columns allow: the S of a tile may be
        // overwritten once that tile's softmax warps are done with it.
        if (elect_one()) {
            constexpr uint32_t idesc_s_full = idesc_bf16(BQ, BKV, 0, 0);
            constexpr uint32_t kQ16 = Q_BYTES >> 4, kKV16 = KV_BYTES >> 4;
            const uint32_t desc_hi = smem_desc_hi(smem_desc_sw128(0, 16, 1024));
            const uint32_t q_lo = smem_desc_lo(smem_desc_sw128(smem_u32(smem + OFF_Q), 16, 1024));
            const uint32_t k_lo = smem_desc_lo(smem_desc_sw128(smem_u32(smem + OFF_K), 16, 1024));
            uint32_t ns[NG] = {0, 0, 0};                 // S tiles issued so far per query tile
            uint32_t item_n = 0, t = 0;
            int stage = 0;
            bool ok = true;
            auto next_stage = [&]() {                    // the next K tile of the ring
                stage = t % NS;
                ok = mbar_wait(&k_full[stage], (t / NS) & 1u, abort_flag);
                ++t;
                return ok;
            };
            auto issue = [&](int g, uint32_t dq, uint32_t idesc_s) {
                ok = ns[g] == 0 || mbar_wait(SPLIT ? &o_done[g] : &s_free[g], (ns[g] - 1) & 1u, abort_flag);
                if (!ok) return;
                tc_fence_after();
                const uint32_t dk = k_lo + (uint32_t)stage * kKV16;
#pragma unroll
                for (int k = 0; k < DH / 16; ++k)        // 16 head-dimension columns = 32 bytes per step
                    mma_ss_lh(tmem_base + kSCol + g * BKV, dq + 2u * k, dk + 2u * k, desc_hi, idesc_s, k != 0);
                mma_commit(&s_full[g]);
                ++ns[g];
            };
            for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x, ++item_n) {
                const Item3 it = decode_item3<RAGGED, CUT>(args, samples, w);
                const uint32_t qb = item_n & 1u, q_item = q_lo + qb * NG * kQ16;
                const uint32_t idesc_last = idesc_bf16(BQ, (it.n - (it.nkv - 1) * BKV + 15) & ~15, 0, 0);
                if (!mbar_wait(&q_full[qb], (item_n >> 1) & 1u, abort_flag)) { ok = false; break; }
                if (CUT && it.third) {
                    for (int j = 0; j < it.third && ok; ++j)
#pragma unroll
                        for (int g = 0; g < NG; ++g) {
                            const int tile = j + g * it.third;
                            if (tile >= it.nkv || !ok || !next_stage()) continue;
                            issue(g, q_item, tile == it.nkv - 1 ? idesc_last : idesc_s_full);
                            if (ok) mma_commit(&k_empty[stage]);
                        }
                } else {
                    for (int j = 0; j < it.nkv && ok; ++j) {
                        const uint32_t idesc_s = j == it.nkv - 1 ? idesc_last : idesc_s_full;
#pragma unroll
                        for (int g = 0; g < NG; ++g) {
                            if (g >= it.ng || !ok || (it.starts(g) && !next_stage())) continue;
                            issue(g, q_item + g * kQ16, idesc_s);
                            if (ok && it.ends(g)) mma_commit(&k_empty[stage]);
                        }
                    }
                }
                if (ok) mma_commit(&q_empty[qb]);
            }
        }
    } else if (warp == 14) {
        // ---------------- P V issuer: O_g (+)= P_g V ----------------
        // P from tensor memory (bf16 pairs, 8 columns per 16 keys), V MN-major (head dimension
        // contiguous), 16 keys = 2048 bytes per slab.
        if (elect_one()) {
            constexpr uint32_t idesc_o = idesc_bf16(BQ, DH, 0, 1);
            constexpr uint32_t kKV16 = KV_BYTES >> 4;
            const uint32_t desc_hi = smem_desc_hi(smem_desc_sw128(0, 16, 1024));
            const uint32_t v_lo = smem_desc_lo(smem_desc_sw128(smem_u32(smem + OFF_V), 16, 1024));
            uint32_t np[NG] = {0, 0, 0};                 // P V products issued so far per query tile
            uint32_t t = 0;
            int stage = 0;
            bool ok = true;
            auto next_stage = [&]() {                    // the next V tile of the ring
                stage = t % NS;
                ok = mbar_wait(&v_full[stage], (t / NS) & 1u, abort_flag);
                ++t;
                return ok;
            };
            auto issue = [&](int g, int ksteps, bool first) {
                ok = mbar_wait(&p_ready[g], np[g] & 1u, abort_flag);
                if (!ok) return;
                tc_fence_after();
                const uint32_t dv = v_lo + (uint32_t)stage * kKV16, o_col = tmem_base + kOCol + g * DH, p_col = tmem_base + kPCol + g * (BKV / 2);
                for (int k = 0; k < ksteps; ++k)
                    mma_ts_lh(o_col, p_col + 8 * k, dv + 128u * k, desc_hi, idesc_o, !(first && k == 0));
                if (SPLIT)
                    for (int k = 0; k < ksteps; ++k)
                        mma_ts_lh(o_col, tmem_base + kSCol + g * BKV + 8 * k, dv + 128u * k, desc_hi, idesc_o, 1u);
                mma_commit(&o_done[g]);
                ++np[g];
            };
            for (int w = blockIdx.x; w < n_items && ok; w += gridDim.x) {
                const Item3 it = decode_item3<RAGGED, CUT>(args, samples, w);
                const int ksteps_last = (it.n - (it.nkv - 1) * BKV + 15) >> 4;
                const bool cut = CUT && it.third;
                for (int j = 0, steps = cut ? it.third : it.nkv; j < steps && ok; ++j) {
                    if (cut) {
#pragma unroll
                        for (int g = 0; g < NG; ++g) {
                            const int tile = j + g * it.third;
                            if (tile >= it.nkv || !ok || !next_stage()) continue;
                            issue(g, tile == it.nkv - 1 ? ksteps_last : BKV / 16, j == 0);
                            if (ok) mma_commit(&v_empty[stage]);
                        }
                    } else {
                        const int ksteps = j == it.nkv - 1 ? ksteps_last : BKV / 16;
#pragma unroll
                        for (int g = 0; g < NG; ++g) {
                            if (g >= it.ng || !ok || (it.starts(g) && !next_stage())) continue;
                            issue(g, ksteps, j == 0);
                            if (ok && it.ends(g)) mma_commit(&v_empty[stage]);
                        }
                    }
                }
            }
        }
    } else if (RAGGED && warp == 15 && args.out) {
        zero_padding(args.out, args.lens, args.B, args.N, args.H, lane);
    }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kSoftmaxRegs));
        // ---------------- softmax, O rescaling and output: one query row per thread ----------------
        const int g = warp >> 2;                         // query tile of this warpgroup
        const int q = warp & 3;                          // tensor-memory lane quadrant of this warp
        const uint32_t lane_addr = tmem_base + ((uint32_t)(q * 32) << 16);
        const uint32_t s_addr = lane_addr + kSCol + g * BKV, p_addr = lane_addr + kPCol + g * (BKV / 2),
                       o_addr = lane_addr + kOCol + g * DH;
        const float sl = args.scale_log2;
        uint32_t cnt = 0;                                // key tiles this warpgroup has walked through
        // A wait that runs out ends the issuing threads and is reported through the status word; these warps walk on to the end
        // of their items, whose results are void then, so that no lane ever leaves a collective access to the others.
        auto wait = [&](uint64_t* bar, uint32_t parity) {
            mbar_wait<false, true>(bar, parity, abort_flag);
            __syncwarp();
            tc_fence_after();
        };
        auto arrive = [&](uint64_t* bar) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar);
        };
        // what last read the P columns, and wrote O: P V of the previous key tile (before the first one the barrier lets the
        // parity of its last phase through at once)
        auto wait_o = [&]() { wait(&o_done[g], (cnt - 1) & 1u); };
        // The key tiles of one query tile: nkv of them, the first nfull whole, the last one of valid_last keys otherwise.  Leaves the
        // running maximum (times scale * log2 e) and sum of this thread's row.
        // gap1: the gap of the second key tile.  two_first: the running maximum starts as that of the first two key tiles, both whole.
        // What rounding the weights to bf16 costs is decided by the largest ones.  The weight at the running maximum is 1 and exact; so up to 128 keys
        // the maximum is the true one, and of more it starts as that of the first 128, as with key tiles of 128.  Where the true maximum `top` lies
        // above the running one all the same, its weight goes into the sum as it was rounded: numerator and denominator then err together, and of
        // a weight that outweighs the rest nothing remains of its error.  Error against 64 bits, 1e-3, scores of standard deviation 1 / 4: from the first 64
        // keys' maximum, from 128, with the top weight as rounded: 64 x 12 x 197 2.272 / 2.104, 2.224 / 1.952, 2.217 / 1.786; 16 x 12 x 1569
        // 2.335 / 2.098, 2.330 / 2.149, 2.328 / 1.886.  Time: 25.0 -> 27.3 us and 159 -> 161 (the wait for the second key tile's S, 1000 cycles an item).
        // Keys cut in three have three running maxima, each exact for a part of the keys, and need neither (1 x 12 x 197: from 128 keys 2.262 / 1.954, cut 2.215 / 1.923).
        // lowest: what the running maximum is at least.  +infinity for rows past a sample's own count: their weights are zeros then and they have
        // no say in which piece of code a key tile goes through, so that a row's bits are those of its sample's tokens alone.
        auto walk = [&](int nkv, int nfull, int valid_last, float gap1, bool two_first, float lowest, float& m_l2, float& l_run) {
            float top = -INFINITY;                       // (not scaled)
            m_l2 = lowest;
            l_run = 0.f;
            int j = 0;
            if (two_first) {
                // S of the first key tile is handed back once it is in registers; of the second's, which stays where it is, only
                // the maximum is taken before the first's exponentials.
                uint32_t r[BKV];
                wait(&s_full[g], cnt & 1u);
                tmem_ld_32x32(s_addr, r);
                tmem_ld_32x32(s_addr + 32, r + 32);
                tmem_wait_ld();
                arrive(&s_free[g]);
                float mx = row_max<BKV>(r);
                wait(&s_full[g], (cnt + 1) & 1u);
#pragma unroll
                for (int c = 0; c < BKV; c += 32) {
                    uint32_t s[32];
                    tmem_ld_32x32(s_addr + c, s);
                    tmem_wait_ld();
                    mx = fmaxf(mx, row_max<32>(s));
                }
                top = mx;
                m_l2 = fmaxf(mx * sl, lowest);
                uint32_t unused[1];
                l_run = exp_pass<0, BKV, false>(r, unused, sl, -m_l2);
                wait_o();
                tmem_st_32x32(p_addr, r);
                tmem_wait_st();
                arrive(&p_ready[g]);
                ++j, ++cnt;
            }
            for (; j < nkv; ++j, ++cnt) {
                // Whole key tiles whose maximum stays within 2^kRescaleGap of the running one: nearly all of them.
                bool have_s = false;
                for (; j < nfull; ++j, ++cnt) {
                    wait(&s_full[g], cnt & 1u);
                    uint32_t r[BKV], lo[SPLIT ? BKV / 2 : 1];
                    tmem_ld_32x32(s_addr, r);
                    tmem_ld_32x32(s_addr + 32, r + 32);
                    tmem_wait_ld();
                    const float mx = row_max<BKV>(r), mx_l2 = mx * sl;
                    if (j == 0) m_l2 = fmaxf(mx_l2, lowest);
                    have_s = __any_sync(0xffffffffu, mx_l2 > m_l2 + kRescaleGap);
                    if (have_s) break;
                    if (!SPLIT) top = fmaxf(top, mx);
                    float l_tile = exp_pass<0, BKV / 2, SPLIT>(r, lo, sl, -m_l2);
                    if (!SPLIT) arrive(&s_free[g]);      // the next Q K^T may overwrite S
                    l_tile += exp_pass<BKV / 2, BKV / 2, SPLIT>(r, lo, sl, -m_l2);
                    l_run += l_tile;
                    if constexpr (SPLIT) tmem_st_32x32(s_addr, lo);      // (S was complete after P V of the key tile before)
                    else wait_o();
                    tmem_st_32x32(p_addr, r);
                    tmem_wait_st();
                    arrive(&p_ready[g]);
                }
                if (j == nkv) break;
                // A key tile that raises the maximum, or the last one with fewer keys than columns: 16 columns at a time from
                // tensor memory, in little code.
                if (!have_s) wait(&s_full[g], cnt & 1u);
                const int valid = j < nfull ? BKV : valid_last;
                auto load16 = [&](int c, uint32_t (&s)[16]) {
                    tmem_ld_32x16(s_addr + c, s);
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < 16; ++i) s[i] = c + i < valid ? s[i] : 0xff800000u;      // past the keys: -infinity, a weight of 0
                };
                float mx = -INFINITY;
#pragma unroll 1
                for (int c = 0; c < valid; c += 16) {
                    uint32_t s[16];
                    load16(c, s);
#pragma unroll
                    for (int i = 0; i < 16; i += 2) mx = max3(mx, __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
                }
                const float mx_l2 = mx * sl;
                if (!SPLIT) top = fmaxf(top, mx);
                wait_o();
                if (j == 0) {
                    m_l2 = fmaxf(mx_l2, lowest);
                } else if (__any_sync(0xffffffffu, mx_l2 > m_l2 + (j == 1 ? gap1 : kRescaleGap))) {
                    const bool raise = mx_l2 > m_l2 + (j == 1 ? gap1 : kRescaleGap);
                    const float alpha = raise ? ex2(m_l2 - mx_l2) : 1.f;
                    if (raise) m_l2 = mx_l2;
                    l_run *= alpha;
#pragma unroll 1
                    for (int c = 0; c < DH; c += 16) {
                        uint32_t o[16];
                        tmem_ld_32x16(o_addr + c, o);
                        tmem_wait_ld();
#pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st_32x16(o_addr + c, o);
                    }
                }
#pragma unroll 1
                for (int c = 0; c < valid; c += 16) {
                    uint32_t s[16], low[8];
                    load16(c, s);
#pragma unroll
                    for (int i = 0; i < 16; i += 2) {
                        const float p0 = ex2(fmaf(__uint_as_float(s[i]), sl, -m_l2)), p1 = ex2(fmaf(__uint_as_float(s[i + 1]), sl, -m_l2));
                        const uint32_t h = pack_bf16(p0, p1);
                        if (SPLIT) low[i >> 1] = pack_bf16(p0 - __uint_as_float(h << 16), p1 - __uint_as_float(h & 0xffff0000u));
                        l_run += p0 + p1;
                        s[i >> 1] = h;
                    }
                    tmem_st_32x8(p_addr + (c >> 1), s);
                    if (SPLIT) tmem_st_32x8(s_addr + (c >> 1), low);     // (columns already read)
                }
                tmem_wait_st();
                arrive(&p_ready[g]);
                if (!SPLIT && lane == 0) mbar_arrive(&s_free[g]);        // (every lane's reads of S are complete at the arrival above)
            }
            if (two_first) {                             // (a top that raised the running maximum has a weight of 1)
                const float p = ex2(fmaf(top, sl, -m_l2));
                l_run += __uint_as_float(pack_bf16(p, 0.f) << 16) - p;
            }
        };
        // O / l -> bf16 -> global.  The warp's 32 rows x 64 values go to its own slab of shared memory (128-byte rows, 16-byte
        // pieces XOR-swizzled like the tensor map's box) and leave with one TMA store, which drops the rows past N.
        uint8_t* const warp_slab = smem + OFF_OST + (g * 4 + q) * 4096;
        uint8_t* const slab = warp_slab + (lane >> 3) * 1024 + (lane & 7) * 128;
        auto store = [&](const Item3& it, int tile) {        // `tile` of the item
            fence_async_smem();
            __syncwarp();
            const int sm = it.stream(tile), row0 = (it.q + tile - sm * it.nt) * BQ + q * 32;
            if (lane == 0 && row0 < it.n) {
                int h = it.h + sm, b = it.b;
                while (h >= args.H) { h -= args.H; ++b; }    // past the last head: of the next sample (or the one after)
                tma_store_4d(&tmO, warp_slab, 0, h, row0, b);
                tma_store_commit();
            }
        };
        auto first_gap = [](int nkv) { return !SPLIT && (RAGGED || !FIRST) && nkv == 2 ? 0.f : kRescaleGap; };
        auto two_first = [](int nkv) { return FIRST && (!RAGGED || nkv > 2); };
        // Whole key tiles.  The second of two counts as one with 64 keys: nearly all of them raise the maximum.
        auto whole_tiles = [](int n) { return !SPLIT && n <= 2 * BKV ? n >= BKV : n / BKV; };
        const int nkv_all = (args.N + BKV - 1) / BKV, nfull_all = whole_tiles(args.N), valid_all = args.N - nfull_all * BKV;
        const int whole = CUT ? args.n_whole : n_items;
        int w = blockIdx.x;
        for (; WHOLE && w < whole; w += gridDim.x) {
            const Item3 it = decode_item3<RAGGED, CUT>(args, samples, w);
            if (g >= it.ng) continue;
            const bool in_use = !RAGGED || (it.q + g - it.stream(g) * it.nt) * BQ + q * 32 + lane < it.n;
            float m_l2, l_run;
            if constexpr (RAGGED) walk(it.nkv, whole_tiles(it.n), it.n - whole_tiles(it.n) * BKV, first_gap(it.nkv), two_first(it.nkv), in_use ? kLowest : INFINITY, m_l2, l_run);
            else walk(nkv_all, nfull_all, valid_all, first_gap(nkv_all), two_first(nkv_all), kLowest, m_l2, l_run);
            wait_o();
            if (lane == 0) tma_store_wait_read<0>();     // the slab's previous store has read it
            __syncwarp();
            const float inv = 1.f / l_run;
#pragma unroll 1
            for (int c = 0; c < DH; c += 32) {
                uint32_t o[32];
                tmem_ld_32x32(o_addr + c, o);
                tmem_wait_ld();
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    uint32_t wv[4];
#pragma unroll
                    for (int i = 0; i < 4; ++i) wv[i] = pack_bf16(__uint_as_float(o[8 * e + 2 * i]) * inv, __uint_as_float(o[8 * e + 2 * i + 1]) * inv);
                    if (!in_use) wv[0] = wv[1] = wv[2] = wv[3] = 0u;
                    *reinterpret_cast<uint4*>(slab + ((((c >> 3) + e) ^ (lane & 7)) << 4)) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
                }
            }
            store(it, g);
        }
        // Keys cut in three.  (A loop of its own, with its own copy of the walk: with both kinds of items in one, the walk of the
        // others took 5 to 8 % longer.)
        if constexpr (CUT) {
            for (; w < n_items; w += gridDim.x) {
                const Item3 it = decode_item3<RAGGED, CUT>(args, samples, w);
                const int first = g * it.third, n = min(max(it.nkv - first, 0), it.third);
                float m_l2, l_run;
                walk(n, min(n, nfull_all - first), valid_all, kRescaleGap, false, kLowest, m_l2, l_run);
                wait_o();
                if (lane == 0) tma_store_wait_read<0>();
                __syncwarp();
                if (g) *reinterpret_cast<float2*>(warp_slab + lane * 8) = make_float2(m_l2, l_run);
                tc_fence_before();
                named_barrier(1, 4 * NG * 32);       // (no warp of these ever leaves early)
                tc_fence_after();
                if (g == 0) {
                    const float2 a = *reinterpret_cast<const float2*>(warp_slab + 4 * 4096 + lane * 8), b = *reinterpret_cast<const float2*>(warp_slab + 8 * 4096 + lane * 8);
                    const float m = fmaxf(m_l2, fmaxf(a.x, b.x));
                    float f[NG] = {ex2(m_l2 - m), ex2(a.x - m), ex2(b.x - m)};
                    const float inv = 1.f / (f[0] * l_run + f[1] * a.y + f[2] * b.y);
#pragma unroll
                    for (int i = 0; i < NG; ++i) f[i] *= inv;
                    const bool third = it.nkv > 2 * it.third;    // (else nothing was written there; the second part is never empty: nkv >= 2)
#pragma unroll 1
                    for (int c = 0; c < DH; c += 8) {
                        uint32_t o[NG][8];
                        tmem_ld_32x8(o_addr + c, o[0]);
                        tmem_ld_32x8(o_addr + DH + c, o[1]);
                        tmem_ld_32x8(o_addr + 2 * DH + c, o[2]);
                        tmem_wait_ld();
                        uint32_t wv[4];
#pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            float u[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e) {
                                u[e] = fmaf(__uint_as_float(o[1][2 * i + e]), f[1], __uint_as_float(o[0][2 * i + e]) * f[0]);
                                if (third) u[e] = fmaf(__uint_as_float(o[2][2 * i + e]), f[2], u[e]);
                            }
                            wv[i] = pack_bf16(u[0], u[1]);
                        }
                        *reinterpret_cast<uint4*>(slab + (((c >> 3) ^ (lane & 7)) << 4)) = make_uint4(wv[0], wv[1], wv[2], wv[3]);
                    }
                    store(it, 0);
                }
                tc_fence_before();
                named_barrier(2, 4 * NG * 32);       // the others' O and slabs may be used again
            }
        }
        if (lane == 0) tma_store_wait<0>();              // every output row written before the CTA exits
    }

    tc_fence_before();
    __syncthreads();
    if (*abort_flag && threadIdx.x == 0) atomicExch(args.status, RS_DEV_TIMEOUT);
    if (warp == 13) {
        __syncwarp();
        tc_fence_after();
        tmem_dealloc(tmem_base, kTmemCols);
    }
}

// The bounded waits by themselves: every warp waits n times, as the softmax warps do, for a barrier that nothing arrives at.
__global__ void __launch_bounds__(128) wait_check_kernel(int n, int* status) {
    __shared__ uint64_t bar;
    __shared__ volatile int abort_flag;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        abort_flag = 0;
        mbar_fence_init();
    }
    __syncthreads();
    for (int i = 0; i < n; ++i) {
        mbar_wait<false, true>(&bar, 0, &abort_flag);
        __syncwarp();
    }
    __syncthreads();
    if (abort_flag && threadIdx.x == 0) atomicExch(status, RS_DEV_TIMEOUT);
}

}  // namespace

cudaError_t launch_wait_check(rs_ctx* ctx, int n, cudaStream_t st) {
    wait_check_kernel<<<1, 128, 0, st>>>(n, ctx->d_status);
    return cudaGetLastError();
}

int attn_tc3_max_samples() { return kMaxSamples; }
// Tiles and items are counted in ints, with room for a stride of the grid past the last.
long long attn_tc3_max_tiles() { return (1ll << 31) - (1 << 20); }

// How many query tiles of every head are taken with the keys cut in three: the count with the shortest longest CTA.  An item of one, two
// or three query tiles takes 0.62, 0.80 or 1.03 us per key tile and 1.3, one with the keys cut 1.03 per key tile of a third and 1.4;
// those follow the others, on the CTAs first that the last round leaves out.
// Chosen where that is 6 % better: the kernel with both kinds of items takes 3 to 4 % longer at the others.  With none cut / as chosen, us:
// 1 x 12 x 197 5.7 / 5.6 (both tiles), 1 x 16 x 577 9.6 / 8.2 (all), 1 x 12 x 785 11.6 / 9.3 (all), 1 x 16 x 4097 110.8 / 99.3 (6 of 33),
// 2 x 12 x 2353 66.8 / 60.3 (1 of 19), 4 x 16 x 1729 80.4 / 77.2 (1 of 14).
int attn_tc3_cut(long long BH, int N, int G) {
    const int nt = (N + BQ - 1) / BQ, nkv = (N + BKV - 1) / BKV;
    if (nkv < 3) return 0;                               // (nothing to cut)
    const double per_tile[NG + 1] = {0, 0.62, 0.80, 1.03}, t_cut = 1.03 * ((nkv + NG - 1) / NG) + 1.4;
    int best = 0;
    double best_t = 0;
    for (int cut = 0; cut <= nt; ++cut) {
        const long long tiles = BH * (nt - cut), left = tiles % (NG * (long long)G), cuts = BH * cut;
        const long long rest = left ? (left + G - 1) / G : 0, n_left = left ? (left + rest - 1) / rest : 0;
        const double t_rest = left ? per_tile[rest] * nkv + 1.3 : 0;
        auto on = [&](long long place) { return cuts > place ? (double)((cuts - 1 - place) / G + 1) : 0.0; };     // items of that CTA, counted from the first idle one
        const double idle = n_left < G ? on(0) * t_cut : 0, busy = n_left ? t_rest + on(G - n_left) * t_cut : 0;
        const double t = (double)((tiles - left) / (NG * (long long)G)) * (per_tile[NG] * nkv + 1.3) + (idle > busy ? idle : busy);
        if (cut == 0 || t < (best ? 1.0 : 0.94) * best_t) { best_t = t; best = cut; }
    }
    return best;
}

// tmK, tmV: boxes of 64 rows; tmQ: 128 rows; tmO: 32 rows.
cudaError_t launch_attn_tc3(rs_ctx* ctx, const rs_attn_desc& d, const CUtensorMap& tmQ, const CUtensorMap& tmK,
                            const CUtensorMap& tmV, const CUtensorMap& tmO, void* padded_out, const int32_t* lens, bool split, cudaStream_t st) {
    static PerDeviceOnce attr_once;   // the attribute belongs to the device current at the call
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    e = (cudaError_t)attr_once.run(dev, [] {
        cudaError_t a = cudaSuccess;
        for (const void* f : {(const void*)attn_tc3_kernel<false, false, false, false>, (const void*)attn_tc3_kernel<false, false, false, true>, (const void*)attn_tc3_kernel<false, false, true, false>,
                              (const void*)attn_tc3_kernel<false, false, true, true>, (const void*)attn_tc3_kernel<false, true, false, true>, (const void*)attn_tc3_kernel<true, false, false, false>,
                              (const void*)attn_tc3_kernel<true, false, true, false>})
            if (a == cudaSuccess) a = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        return (int)a;
    });
    if (e != cudaSuccess) return e;
    Attn3Args args;
    args.N = d.N; args.H = d.H; args.B = d.B;
    const int G = ctx->sm_count;
    const long long BH = (long long)d.B * d.H;
    const int nt = (d.N + BQ - 1) / BQ;
    if (BH * nt >= attn_tc3_max_tiles()) return cudaErrorInvalidValue;
    args.cut = lens ? 0 : attn_tc3_cut(BH, d.N, G);
    args.nt = nt - args.cut;
    const long long tiles = BH * args.nt, left = tiles % (NG * (long long)G);
    args.tiles = (int)tiles;
    auto reciprocal = [](int v) { return v <= 1 ? 0xffffffffu : (uint32_t)((1ull << 32) / (unsigned)v); };
    args.by_nt = reciprocal(args.nt);
    args.by_h = reciprocal(d.H);
    args.by_cut = reciprocal(args.cut);
    args.full = (int)((tiles - left) / NG);
    // a last round of at most 2 G tiles: two to an item on twice the CTAs instead of three, 8 x 16 x 577 27.7 -> 25.0 us, 16 x 12 x 1569 165.8 -> 159.7
    args.rest = left ? (int)((left + G - 1) / G) : 1;
    args.n_whole = args.full + (int)((left + args.rest - 1) / args.rest);
    args.n_items = args.n_whole + (int)(BH * args.cut);
    args.lens = lens;
    args.out = (__nv_bfloat16*)padded_out;
    const float scale = d.scale != 0.f ? d.scale : 0.125f;
    args.scale_log2 = scale * 1.4426950408889634f;
    args.status = ctx->d_status;
    const long long most = lens ? BH * nt : args.n_items;
    const int grid = most < G ? (int)most : G;
    auto run = [&](auto kernel) { return launch_pdl(kernel, dim3(grid), dim3(kThreads), kSmem, st, tmQ, tmK, tmV, tmO, args); };
    if (lens) return run(attn_tc3_kernel<false, true, false, true>);
    if (split) return args.cut ? run(attn_tc3_kernel<true, false, true, false>) : run(attn_tc3_kernel<true, false, false, false>);
    // Short sequences, and those with all query tiles cut by keys, run without the code that only the others need.
    if (args.cut) return args.nt ? run(attn_tc3_kernel<false, false, true, true>) : run(attn_tc3_kernel<false, false, true, false>);
    return d.N > 2 * BKV ? run(attn_tc3_kernel<false, false, false, true>) : run(attn_tc3_kernel<false, false, false, false>);
}

}  // namespace rs
