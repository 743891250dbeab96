// Dequantisation arithmetic shared by the GEMM kernels: packed 8-bit / 4-bit codes times an fp32 scale, rounded once
// (nearest even) to bf16, two weights per packed instruction.
#pragma once
#include <cuda_bf16.h>
#include <stdint.h>

namespace qg {

__device__ __forceinline__ uint32_t bf16x2(float lo, float hi) {
    const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&b);
}

// 8-bit codes.  A code byte c (0..255) dropped into byte 1 of 0x43000000 reads as the float 128 + c / 256, so
// q * s = fma(f, 256 s, -(32768 + 128) s) for the sign-flipped int8 byte: both constants and the result are exact in fp32,
// one rounding (to bf16) follows.
// Per weight: one byte permute builds f from a code byte and the magic word, half a packed two-float fused
// multiply-add (fma.rn.f32x2, each lane IEEE-exact as fmaf) converts, half a packed conversion rounds to bf16x2.
__device__ __forceinline__ uint32_t fma2_bf16x2(uint32_t a0, uint32_t a1, uint64_t m, uint64_t c) {
    uint32_t r;     // bf16(a0 * m.lo + c.lo) | bf16(a1 * m.hi + c.hi) << 16
    asm("{\n\t.reg .b64 t;\n\t.reg .b32 lo, hi;\n\t"
        "mov.b64 t, {%1, %2};\n\t"
        "fma.rn.f32x2 t, t, %3, %4;\n\t"
        "mov.b64 {lo, hi}, t;\n\t"
        "cvt.rn.bf16x2.f32 %0, hi, lo;\n\t}"
        : "=r"(r) : "r"(a0), "r"(a1), "l"(m), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
    return static_cast<uint64_t>(__float_as_uint(lo)) | (static_cast<uint64_t>(__float_as_uint(hi)) << 32);
}
template <int BYTE>
__device__ __forceinline__ uint32_t code_byte_to_float(uint32_t x, uint32_t magic) {   // bits of 128 + byte BYTE of x / 256
    return __byte_perm(x, magic, 0x7404 + (BYTE << 4));
}

// 4 int8 codes (one word) -> 4 bf16 = q * scale.  m2 = {256 s, 256 s}, c2 = {-32896 s, -32896 s}.
__device__ __forceinline__ void dq8_word(uint32_t x, uint64_t m2, uint64_t c2, uint32_t magic, uint32_t& o0, uint32_t& o1) {
    x ^= 0x80808080u;                            // byte = q + 128
    o0 = fma2_bf16x2(code_byte_to_float<0>(x, magic), code_byte_to_float<1>(x, magic), m2, c2);
    o1 = fma2_bf16x2(code_byte_to_float<2>(x, magic), code_byte_to_float<3>(x, magic), m2, c2);
}

// 8 4-bit codes (one word, nibble i = weight i, code u = q + 8) -> 8 bf16, in bf16 arithmetic.  A byte permute puts the word's
// byte j below and byte j of the word shifted right by one above, so that weight 2 j sits in bits 0-3 of the low half and
// weight 2 j + 1 in bits 3-6 of the high half; masked and under the exponents of 2^7 and 2^4 they read as 128 + u and 16 + u.
// Minus (136, 24) that is q, exactly.  The scale, 11 significant bits, is the sum of two bf16 numbers, its rounding to 8 bits
// (hi) and the rest, at most 3 bits (lo): q lo has 7 bits at most and is exact, and fma(q, hi, q lo) rounds the exact q * scale
// once, as the fp32 chain of the 8-bit codes does (equal bit for bit over all codes and finite scales).  9 instructions of the
// integer pipe and 12 of the FMA pipe per word, where permutes to fp32, packed fma and conversion were 17 (conversions
// included) and 4, and the integer pipe runs at half rate: the limit of a converting warp's arithmetic.
__device__ __forceinline__ void dq4_word(uint32_t x, uint32_t hi2, uint32_t lo2, uint32_t* o) {
    const uint32_t x1 = x >> 1;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t v = (__byte_perm(x, x1, 0x4400 + 0x1111 * j) & 0x0078000Fu) | 0x41804300u;
        asm("{\n\t.reg .b32 q, t;\n\t"
            "add.rn.bf16x2 q, %1, %2;\n\t"
            "mul.rn.bf16x2 t, q, %4;\n\t"
            "fma.rn.bf16x2 %0, q, %3, t;\n\t}"
            : "=r"(o[j]) : "r"(v), "r"(0xC1C0C308u), "r"(hi2), "r"(lo2));
    }
}
// The two parts of a scale, each in both halves.
__device__ __forceinline__ void dq4_consts(float s, uint32_t& hi2, uint32_t& lo2) {
    hi2 = bf16x2(s, s);
    const float lo = s - __uint_as_float(hi2 << 16);
    lo2 = bf16x2(lo, lo);
}

constexpr uint32_t DQ_MAGIC = 0x43000000u;

// Packed constants of 8-bit codes for one scale s: m2 = {256 s, 256 s}, c2 = {-32896 s, -32896 s}.
__device__ __forceinline__ void dq8_consts(float s, uint64_t& m2, uint64_t& c2) {
    const float m1 = 256.f * s, c1 = -32896.f * s;
    m2 = pack_f32x2(m1, m1);
    c2 = pack_f32x2(c1, c1);
}

}  // namespace qg
