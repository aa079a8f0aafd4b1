// int4 -> fp16 tensor-core fragments shared by the batch-1 and the grouped kernels.
//
// A 32-bit word holds 8 codes k0..k7 of one row.  w & 0x000F000F holds the pair (k0, k4), w & 0x00F000F0 the pair (k1, k5) four bits
// higher, and the same on w >> 8 gives (k2, k6) and (k3, k7).  Three forms make fp16 of them: the masked words as the subnormals they are
// (dequant_word_s), under the exponents of 1024 and 64 (dequant_word_b), or q - z by one HFMA2 per pair (dequant_word_x).  The
// k slots of the m16n8k16 MMA are therefore used in the order (k0,k4 | k1,k5) for the first k-step of a 32-code
// chunk and (k2,k6 | k3,k7) for the second, lane t of a quad owning word t of the chunk; the
// activation operand is arranged in the same order (permute8), so a B fragment of a chunk is four
// consecutive 32-bit registers.
#pragma once

#include "edg_common.cuh"

namespace edg {

__device__ __forceinline__ uint32_t lop3_and_or(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t d;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}
__device__ __forceinline__ uint32_t h2_as_u32(__half2 v) { return *reinterpret_cast<uint32_t*>(&v); }
__device__ __forceinline__ __half2 u32_as_h2(uint32_t v) { return *reinterpret_cast<__half2*>(&v); }

// d = a . b  (fresh accumulator)
__device__ __forceinline__ void mma16816_zero(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
                 : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma16816_bf16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// 8 fp32 values as words of two bf16, part by part: 8 of their 24 bits each, three parts are the value
template <int PARTS>
__device__ __forceinline__ void bf16_parts(const float (&w)[8], uint32_t (&out)[PARTS][4]) {
    float r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = w[i];
#pragma unroll
    for (int q = 0; q < PARTS; ++q)
#pragma unroll
        for (int i = 0; i < 8; i += 2) {
            const uint32_t a = __float_as_uint(r[i]) & 0xFFFF0000u, b = __float_as_uint(r[i + 1]) & 0xFFFF0000u;
            out[q][i / 2] = (a >> 16) | b;
            r[i] -= __uint_as_float(a);
            r[i + 1] -= __uint_as_float(b);
        }
}

// 8 consecutive fp32 activations -> the fp16 residuals v - fp16(v), same k-slot order
__device__ __forceinline__ uint4 permute8_lo(const float (&v)[8]) {
    float r[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) r[i] = v[i] - __half2float(__float2half_rn(v[i]));
    uint4 o;
    o.x = h2_as_u32(__floats2half2_rn(r[0], r[4]));
    o.y = h2_as_u32(__floats2half2_rn(r[1], r[5]));
    o.z = h2_as_u32(__floats2half2_rn(r[2], r[6]));
    o.w = h2_as_u32(__floats2half2_rn(r[3], r[7]));
    return o;
}

// 8 consecutive activations -> fp16 in the k-slot order of the fragments: (x0,x4,x1,x5,x2,x6,x3,x7)
__device__ __forceinline__ uint4 permute8(const float (&v)[8]) {
    uint4 r;
    r.x = h2_as_u32(__floats2half2_rn(v[0], v[4]));
    r.y = h2_as_u32(__floats2half2_rn(v[1], v[5]));
    r.z = h2_as_u32(__floats2half2_rn(v[2], v[6]));
    r.w = h2_as_u32(__floats2half2_rn(v[3], v[7]));
    return r;
}

// 16 bytes of bf16 -> 8 fp16 (exact in the normal range), in the k-slot order of the fragments and in their own
__device__ __forceinline__ uint4 bf16x8_permute8(uint4 v) {
    const float f[8] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y), bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w)};
    return permute8(f);
}
__device__ __forceinline__ uint4 bf16x8_to_f16(uint4 v) {
    uint4 o;
    o.x = h2_as_u32(__floats2half2_rn(bf16_lo(v.x), bf16_hi(v.x)));
    o.y = h2_as_u32(__floats2half2_rn(bf16_lo(v.y), bf16_hi(v.y)));
    o.z = h2_as_u32(__floats2half2_rn(bf16_lo(v.z), bf16_hi(v.z)));
    o.w = h2_as_u32(__floats2half2_rn(bf16_lo(v.w), bf16_hi(v.w)));
    return o;
}

// The cheapest form: the code words masked straight into fp16 subnormals -- codes 0, 2, 4, 6 of a word are q * 2^-24, codes 1, 3,
// 5, 7 (their nibble sits four bits higher) q * 2^-20 -- five instructions a word and nothing to remove: the tensor cores take
// subnormal operands exactly.  The activations at odd positions carry the missing 2^-4 (permute8_s), sums of products come
// out as 2^-24 of the dot product with the codes, in which unit the caller removes the zero point
// (fma(-z, 2^-24 * sum of the activations, c)); kUnscaleS brings the end result back.
// fp16 would round small activations to multiples of 2^-25, and those at odd positions to 2^-21.  So a vector of them (the state, a
// quarter of an expert's h) is brought to a largest magnitude of 2^13 .. 2^14 first, by a power of two whose inverse goes into the
// factor of the end result: what is lost is 2^-34 of the largest, whatever the magnitude.
constexpr float kScaleS = 5.9604644775390625e-8f;      // 2^-24
constexpr float kUnscaleS = 16777216.f;                // 2^24
__device__ __forceinline__ void dequant_word_s(uint32_t w, uint32_t (&out)[4]) {
    const uint32_t w2 = w >> 8;
    out[0] = w & 0x000F000Fu;
    out[1] = w & 0x00F000F0u;
    out[2] = w2 & 0x000F000Fu;
    out[3] = w2 & 0x00F000F0u;
}
// the power of two for a vector whose largest magnitude has the bits m (2^126 at most; infinities stay what they are), and its inverse
__device__ __forceinline__ float vector_scale(uint32_t m) { return __uint_as_float(min(267u - (m >> 23), 253u) << 23); }
__device__ __forceinline__ float vector_unscale(float s) { return __uint_as_float((254u << 23) - __float_as_uint(s)); }
__device__ __forceinline__ uint32_t abs_max8(const float (&v)[8]) {
    uint32_t m = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) m = max(m, __float_as_uint(v[i]) & 0x7FFFFFFFu);
    return m;
}
// permute8 and permute8_lo of the activations times the vector's power of two, those at odd positions times 2^-4 more
__device__ __forceinline__ uint4 permute8_s(const float (&v)[8], float s) {
    const float o = s * 0.0625f, f[8] = {v[0] * s, v[1] * o, v[2] * s, v[3] * o, v[4] * s, v[5] * o, v[6] * s, v[7] * o};
    return permute8(f);
}
__device__ __forceinline__ uint4 permute8_lo_s(const float (&v)[8], float s) {
    const float o = s * 0.0625f, f[8] = {v[0] * s, v[1] * o, v[2] * s, v[3] * o, v[4] * s, v[5] * o, v[6] * s, v[7] * o};
    return permute8_lo(f);
}
// The biased form: codes 0, 2, 4, 6 of a word as 1024 + q, codes 1, 3, 5, 7 as 64 + q, five instructions a word too.  The dot
// product then carries 1024 * (sum of the activations at even positions) + 64 * (sum at odd positions), which the caller
// subtracts per scaled block along with the zero-point term.  Its fp32 sums of 10^4-sized terms cost 2e-5 relative on a
// layer's output; it stays for chains of dependent steps, whose state is rounded to bf16 and fed back: there another
// rounding can tip a near-tie of the routing further on, and a chain is to reproduce what it produced before.
__device__ __forceinline__ void dequant_word_b(uint32_t w, uint32_t (&out)[4]) {
    const uint32_t w2 = w >> 8;
    out[0] = lop3_and_or(w, 0x000F000Fu, 0x64006400u);
    out[1] = lop3_and_or(w, 0x00F000F0u, 0x54005400u);
    out[2] = lop3_and_or(w2, 0x000F000Fu, 0x64006400u);
    out[3] = lop3_and_or(w2, 0x00F000F0u, 0x54005400u);
}
// EX: the subnormal form, else the biased one
template <bool EX> __device__ __forceinline__ void dequant_code_word(uint32_t w, uint32_t (&o)[4]) {
    if (EX) dequant_word_s(w, o);
    else dequant_word_b(w, o);
}

// The exact form: (w & 0x000F000F) read as fp16 is the subnormal q * 2^-24, (w & 0x00F000F0) is q * 2^-20, so one HFMA2
// per pair of codes gives (q - z) * 2^-9 without rounding (subnormal inputs are exact numbers to it; zero points are
// multiples of 1/128) -- nine instructions a word, and no bias or zero point to remove afterwards.
// mz = neg_zero_x of the row's (scale, zero) pair; sums of products are scaled back by kUnscaleX.
constexpr float kUnscaleX = 512.f;
__device__ __forceinline__ __half2 neg_zero_x(__half2 sz) { return __hmul2(__high2half2(sz), u32_as_h2(0x98009800u)); }   // -z * 2^-9
__device__ __forceinline__ void dequant_word_x(uint32_t w, __half2 mz, uint32_t (&out)[4]) {
    const __half2 e15 = u32_as_h2(0x78007800u), e11 = u32_as_h2(0x68006800u);      // 2^15, 2^11
    const uint32_t w2 = w >> 8;
    out[0] = h2_as_u32(__hfma2(u32_as_h2(w & 0x000F000Fu), e15, mz));
    out[1] = h2_as_u32(__hfma2(u32_as_h2(w & 0x00F000F0u), e11, mz));
    out[2] = h2_as_u32(__hfma2(u32_as_h2(w2 & 0x000F000Fu), e15, mz));
    out[3] = h2_as_u32(__hfma2(u32_as_h2(w2 & 0x00F000F0u), e11, mz));
}
// a += s * c, two values in one instruction
__device__ __forceinline__ void fma2(float& a0, float& a1, float s, float c0, float c1) {
    asm("{\n.reg .b64 a, s, c;\nmov.b64 a, {%0, %1};\nmov.b64 s, {%2, %2};\nmov.b64 c, {%3, %4};\nfma.rn.f32x2 a, s, c, a;\nmov.b64 {%0, %1}, a;\n}"
        : "+f"(a0), "+f"(a1) : "f"(s), "f"(c0), "f"(c1));
}

}  // namespace edg
