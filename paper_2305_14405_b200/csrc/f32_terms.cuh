// fp32 products on the bf16 tensor cores: every fp32 operand is the sum of three bf16 terms.
//
//   a = h + m 2^-16 + l 2^-32,   h = bf16(a), m = bf16(2^16 (a - h)), l = 2^16 (m's remainder): 8 + 8 + 8 bits, exact
//   a w = h h' + 2^-16 (h m' + m h') + 2^-32 (m m' + h l' + l h') + terms of about 2^-26 of a w, of either sign, left out
//
// Six bf16 products instead of one fp32 product, at 26 times the rate.  The terms are exact for every a, and finite below 2^112:
// the kernels go back to FMAs where they are not.  (Below 2^-126, where a itself is subnormal, h has fewer bits and what is left
// out grows, to 2^-18 of a w at most; that is less than such an operand's own unit.)
// What needs care is the tensor core's sum, which is truncated, not rounded, at every step of 16 k: 1.55e-8 of the sum for each,
// where a chain of FMAs is off by 7.4e-9 sqrt(k).  So an accumulator of h h' takes four steps only and several of them are added
// up in fp32; the five small products have accumulators of their own, in which such an error is 2^-8 of that.  With operands of one
// sign the truncations do not average out: 8e-8 of the result from K = 64 on, 7e-8 of it the truncations (two steps: 5.5e-8, at a tenth
// more time); one chain of FMAs is off by 6e-8 at K = 16, 1.2e-7 at 64, 4e-7 at 768, 8e-7 at 3072.
#pragma once
#include "nm_common.cuh"

// Two fp32 numbers as three times two bf16 numbers.
__device__ __forceinline__ void nm_f32_terms2(float x, float y, uint32_t& h, uint32_t& m, uint32_t& l)
{
    const uint64_t minus = nm_pack2(-1.f, -1.f), up = nm_pack2(65536.f, 65536.f);
    uint64_t r = nm_pack2(x, y);
    auto term = [&](uint32_t& o) {   // o = bf16(r), r = what is left, 2^16-fold
        float a, b;
        nm_unpack2(r, a, b);
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(o) : "f"(b), "f"(a));
        const uint64_t t = nm_pack2(__uint_as_float(o << 16), __uint_as_float(o & 0xffff0000u));
        asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(r) : "l"(t), "l"(minus));
        asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(r) : "l"(up));
    };
    term(h);
    term(m);
    float a, b;
    nm_unpack2(r, a, b);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(b), "f"(a));
}
// Four as three times four.
__device__ __forceinline__ void nm_f32_terms4(const float4& v, uint2& h, uint2& m, uint2& l)
{
    nm_f32_terms2(v.x, v.y, h.x, m.x, l.x);
    nm_f32_terms2(v.z, v.w, h.y, m.y, l.y);
}
// The sum of the three kinds of products.
__device__ __forceinline__ float nm_f32_sum(float hh, uint32_t mid, uint32_t low)
{
    return __fmaf_rn(__fmaf_rn(__uint_as_float(low), 0x1p-16f, __uint_as_float(mid)), 0x1p-16f, hh);
}
