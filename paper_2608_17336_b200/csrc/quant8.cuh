// Arithmetic of the blockwise symmetric INT8 quantiser (App. C, "Blockwise INT8 Quantization"), shared by
// the quantise-once kernel and the attention kernel's on-chip quantiser: xhat = round(x / delta) with an
// IEEE FP32 quotient and round-half-to-even, clamped to [-127, 127].
#pragma once

#include <cuda_fp16.h>
#include <stdint.h>

namespace tilemix {

__device__ __forceinline__ uint32_t habs2_bits(uint32_t v) { return v & 0x7fff7fffu; }

// Larger magnitude of two packed pairs of binary16 values in one instruction; the sign bits of the result mean
// nothing (habs2_bits when the last one is in).  For the on-chip quantiser, which is bound by its instructions.
__device__ __forceinline__ uint32_t hmaxabs2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("max.NaN.xorsign.abs.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// max of two packed pairs of non-negative binary16 values: for non-negative finite halves the
// bit patterns order like unsigned integers.
__device__ __forceinline__ uint32_t umax2(uint32_t a, uint32_t b) { return __vmaxu2(a, b); }

// Scale of a block and what its codes are made with.  The definition is RN_int(RN(x / delta)), delta = RN(amax / 127);
// the codes are taken from ONE fused multiply-add, x * r + 1.5 * 2^23 (round-to-nearest-even puts the integer in the low
// mantissa bits, so the low byte of the sum IS the two's-complement INT8 code), which rounds x * r to the nearest
// integer exactly.  The two can only differ where the quotient is within ~2^-23 of a half-integer.  127 x / amax is a
// ratio of 11-bit integers and a power of two, so apart from exact half-integers it keeps a relative distance of at
// least 1 / (255 * 2048) from them.  Exact half-integers: 254 x = (2k + 1) amax, that is x = +-amax / 2 (k = 63), or 127
// divides amax's mantissa.
//  - x = amax / 2: the definition gives 64 if RN(x / delta) >= 63.5, else 63; r = RN(1 / delta) is moved by one unit in
//    the last place where x * r falls on the other side of 63.5;
//  - 127 divides the mantissa (then delta is exact; 8 of 1024 mantissas): `refine`, the quotient itself -- q0 = x * r,
//    then q0 + (x - delta * q0) * r with the residual exact in one FMA (P. Markstein, "Computation of elementary functions
//    on the IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990) -- before the rounding.
// Both forms equal the definition for every binary16 amax and every |x| <= amax (tests/test_quant_codes.py compares the
// arithmetic over all of them, tests/test_gpu_quant_exact.py the kernels next to the half-integers).
// amax = inf or NaN: r = 0 or NaN, `refine` stays off.
struct QuantScale {
    float delta, r;
    bool refine;
};
__device__ __forceinline__ QuantScale quant_scale(float amax) {
    QuantScale s;
    s.delta = __fdiv_rn(amax, 127.0f);
    s.r = __frcp_rn(s.delta);
    const float half = 0.5f * amax;
    // RN(half / delta) >= 63.5, from the exact residual: the quotient is at most half a unit (2^-19) below 63.5
    const bool up = __fmaf_rn(-63.5f, s.delta, half) >= -1.9073486328125e-6f * s.delta;
    const float side = __fmaf_rn(half, s.r, -63.5f);
    if (up && side < 0.f) s.r = __uint_as_float(__float_as_uint(s.r) + 1u);
    if (!up && side >= 0.f) s.r = __uint_as_float(__float_as_uint(s.r) - 1u);
    s.refine = __fmaf_rn(127.f, s.delta, -amax) == 0.f || (__fmaf_rn(half, s.r, -63.5f) >= 0.f) != up;
    return s;
}

// Eight elements, packed FP32x2 arithmetic.
template <bool REFINE>
__device__ __forceinline__ uint2 quant8(const uint4& v, const QuantScale& s) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const float2 r2 = make_float2(s.r, s.r), nd2 = make_float2(-s.delta, -s.delta);
    const float2 magic = make_float2(12582912.f, 12582912.f);
    float2 y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
        if constexpr (REFINE) {
            float2 q = __fmul2_rn(x, r2);
            q = __ffma2_rn(__ffma2_rn(nd2, q, x), r2, q);
            y[i] = __fadd2_rn(q, magic);
        } else {
            y[i] = __ffma2_rn(x, r2, magic);
        }
    }
    // low bytes of the eight sums -> two words
    const uint32_t p0 = __byte_perm(__float_as_uint(y[0].x), __float_as_uint(y[0].y), 0x0040);
    const uint32_t p1 = __byte_perm(__float_as_uint(y[1].x), __float_as_uint(y[1].y), 0x0040);
    const uint32_t p2 = __byte_perm(__float_as_uint(y[2].x), __float_as_uint(y[2].y), 0x0040);
    const uint32_t p3 = __byte_perm(__float_as_uint(y[3].x), __float_as_uint(y[3].y), 0x0040);
    return make_uint2(__byte_perm(p0, p1, 0x5410), __byte_perm(p2, p3, 0x5410));
}
__device__ __forceinline__ uint2 quant8(const uint4& v, const QuantScale& s) {
    return s.refine ? quant8<true>(v, s) : quant8<false>(v, s);
}

}  // namespace tilemix
