// Small device helpers shared by the attention kernels.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace rs {
namespace attn {

constexpr float kLowest = -3.402823466e38f;      // stands for a maximum of -infinity, below which no finite one is: such scores are weights of 0

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// Packed fp32 pairs (two lanes of arithmetic per instruction on sm_100).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t ffma2(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t fadd2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

__device__ __forceinline__ uint64_t fmul2(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

// The larger of the two; NaN if either is (fmaxf drops a NaN).
__device__ __forceinline__ float max_nan(float a, float b) {
    float r;
    asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
    return r;
}

// 2^x for a pair on the FMA pipes instead of the special-function unit: round to nearest by adding 1.5 * 2^23 (whose
// low mantissa bits then hold the integer n), a degree-5 polynomial for 2^(x - n) on [-1/2, 1/2] (csrc/fit_ex2.py: relative
// error 2.2e-7 in fp32 arithmetic -- ex2.approx has 2 ulp), and a product with 2^n.  x up to about 120.  Values that are
// not finite come out as ex2.approx gives them: NaN stays NaN (max.NaN keeps it, and 2^n is multiplied in, not added to the
// exponent bits, which would make a number of it), and x below -126.5 gives 0.
__device__ __forceinline__ void ex2_pair_fma(uint64_t x2, float& p0, float& p1) {
    float x0, x1;
    unpack2(x2, x0, x1);
    x2 = pack2(max_nan(x0, -127.f), max_nan(x1, -127.f));
    const uint64_t t = fadd2(x2, pack2(12582912.f, 12582912.f));
    const uint64_t f = ffma2(fadd2(t, pack2(-12582912.f, -12582912.f)), pack2(-1.f, -1.f), x2);
    uint64_t q = ffma2(f, pack2(0.001327644451521337f, 0.001327644451521337f), pack2(0.00967553723603487f, 0.00967553723603487f));
    q = ffma2(f, q, pack2(0.05550713464617729f, 0.05550713464617729f));
    q = ffma2(f, q, pack2(0.24022120237350464f, 0.24022120237350464f));
    q = ffma2(f, q, pack2(0.6931469440460205f, 0.6931469440460205f));
    q = ffma2(f, q, pack2(1.0000001192092896f, 1.0000001192092896f));
    float t0, t1;
    unpack2(t, t0, t1);
    const uint64_t scale = pack2(__uint_as_float((__float_as_uint(t0) << 23) + 0x3f800000u),     // 2^n; n = -127: 0
                                 __uint_as_float((__float_as_uint(t1) << 23) + 0x3f800000u));
    unpack2(ffma2(q, scale, 0ull), p0, p1);
}

// Zeros in the rows of out ([B, N, H, 64]) that no query tile writes: every box of 32 rows that lies past its sample's count (lens, clamped
// to 1 .. N).  One warp per CTA, idle otherwise; eight rows at a time, so that few samples are spread over the CTAs too, and a lane
// to look up whether they are to be written.
__device__ __forceinline__ void zero_padding(__nv_bfloat16* out, const int* lens, int B, int N, int H, int lane) {
    const int parts = (N + 7) / 8, all = B * parts;          // (B * N rows of 128 bytes fit a GPU)
    for (int first = blockIdx.x; first < all; first += 32 * gridDim.x) {
        const int i = first + lane * gridDim.x, b = i / parts, row0 = (i - b * parts) * 8;
        uint32_t left = __ballot_sync(0xffffffffu, i < all && (row0 & ~31) >= min(max(__ldg(lens + min(b, B - 1)), 1), N));
        for (; left; left &= left - 1) {
            const int src = __ffs(left) - 1, fb = __shfl_sync(0xffffffffu, b, src), fr = __shfl_sync(0xffffffffu, row0, src);
            uint4* p = reinterpret_cast<uint4*>(out + ((long long)fb * N + fr) * H * 64);
            for (int e = lane, n = min(8, N - fr) * H * 8; e < n; e += 32) p[e] = make_uint4(0u, 0u, 0u, 0u);
        }
    }
}

}  // namespace attn
}  // namespace rs
