// Warp-level pieces of the weight-streaming kernels: mma.sync with the weights as the 16-row operand, codes as bf16
// integers.
#pragma once
#include <stdint.h>

namespace qg {

__device__ __forceinline__ uint4 lds_u4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds_u1(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint2 lds_u2(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts_u4(uint32_t addr, const uint4& v) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint32_t sub_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}
__device__ __forceinline__ void mma_w16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// the same with a zero addend
__device__ __forceinline__ void mma_w16_first(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
                 "{%10, %10, %10, %10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
// eight nibbles (nibble i = code i) -> four bf16 pairs of integers code - 8: (0, 2), (4, 6), (1, 3), (5, 7).  The even
// and the odd nibbles become bytes, a byte permute puts the 0x43 of the bf16 number 128 + code above each.
__device__ __forceinline__ void q4_spread(uint32_t w, uint32_t (&p)[4]) {
    constexpr uint32_t HIGH = 0x43434343u, ZERO = 0x43084308u;   // 136
    const uint32_t e = w & 0x0F0F0F0Fu, o = (w >> 4) & 0x0F0F0F0Fu;
    p[0] = sub_bf16x2(__byte_perm(e, HIGH, 0x5140), ZERO);
    p[1] = sub_bf16x2(__byte_perm(e, HIGH, 0x7362), ZERO);
    p[2] = sub_bf16x2(__byte_perm(o, HIGH, 0x5140), ZERO);
    p[3] = sub_bf16x2(__byte_perm(o, HIGH, 0x7362), ZERO);
}

// four int8 codes (one word) -> two bf16 pairs of the same integers: (0, 2), (1, 3).  The low seven bits above 0x43 are the
// bf16 number 128 + bits, the sign bit above 0x43 is 128 or 256: their difference is exact.
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t mask, uint32_t base) {     // one LOP3 (two when written with operators)
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(mask), "r"(base));
    return r;
}
__device__ __forceinline__ void q8_spread(uint32_t w, uint32_t& p02, uint32_t& p13) {
    constexpr uint32_t LOW = 0x007F007Fu, SIGN = 0x00800080u, BASE = 0x43004300u;
    const uint32_t v = w >> 8;
    p02 = sub_bf16x2(and_or(w, LOW, BASE), and_or(w, SIGN, BASE));
    p13 = sub_bf16x2(and_or(v, LOW, BASE), and_or(v, SIGN, BASE));
}

}  // namespace qg
