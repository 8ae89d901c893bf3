// Register-level int4 -> bf16 dequantisation shared by every kernel of the
// library (the exported dequant, the GEMM and the small-M path), so that the
// GEMM's weights are w4a16_dequant's output, value for value (only the sign of
// a zero may differ).
//
// A packed 32-bit word holds eight consecutive codes q_0..q_7 of one row
// (q_i in bits 4i..4i+3: byte j carries the even k in its low nibble and the
// odd k in its high nibble).  For each pair (q_2j, q_2j+1) the word is turned
// into a bf16x2 without any int->float conversion:
//   - PRMT puts byte j of w in byte 0 and byte j of (w >> 4) in byte 2;
//   - masking to bits 0..3 / 16..19 and OR-ing 0x4300 into each half gives
//     the bf16 pattern 0x430q, whose value is 128 + q (bf16 spacing on
//     [128, 256) is exactly 1);
//   - a bf16x2 subtraction of 136 gives q - 8 exactly (|q - 8| <= 8);
//   - a bf16x2 multiply by the scale rounds the exact product once, to
//     nearest even -- the definition wd = RNE_bf16((q - 8) * s).
#pragma once

#include <cstdint>

namespace w4a16 {

__device__ __forceinline__ uint32_t prmt_b32(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

__device__ __forceinline__ uint32_t bf16x2_sub(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("sub.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

__device__ __forceinline__ uint32_t bf16x2_mul(uint32_t a, uint32_t b) {
    uint32_t r;
    asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
    return r;
}

// 8 codes -> 4 bf16x2 words; out[j] = (wd(k=2j) low half, wd(k=2j+1) high half).
// s2 holds the row's bf16 scale in both halves.
__device__ __forceinline__ void dequant_word(uint32_t w, uint32_t s2, uint32_t* out) {
    const uint32_t w4 = w >> 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t t = prmt_b32(w, w4, static_cast<uint32_t>(j | ((4 + j) << 8)));
        t = (t & 0x000F000Fu) | 0x43004300u;               // (128 + q_2j, 128 + q_2j+1)
        out[j] = bf16x2_mul(bf16x2_sub(t, 0x43084308u), s2);  // (q - 8) * s, one rounding
    }
}

// The same values with one rounding step per pair: RNE_bf16(q s - 8 s) as a
// single bf16x2 FMA.  Bits 0..7 of a bf16 with the other bits zero are the
// integer times 2^-133 (the subnormals and the first binade are one linear
// range), so a masked nibble is already a number: the even code moved to bits
// 3..6 of its byte is 8 q 2^-133, the odd code left in bits 4..7 is
// 16 q 2^-133, and the FMA's multiplier takes the power of two back.
// Exact before its one rounding for |s| < 2^-2 (the multiplier s 2^130 has to
// be finite); scale_is_wide marks the others, which take dequant_word.  A zero
// (q = 8) is always +0 here.
struct ScaleFma {
    uint32_t mul;  // (s 2^130, s 2^129): for the even, the odd code of a pair
    uint32_t add;  // (-8 s, -8 s)
};

__device__ __forceinline__ bool scale_is_wide(uint16_t s) { return (s & 0x7FFFu) >= 0x3E80u; }

__device__ __forceinline__ uint32_t bf16x2_fma(uint32_t a, uint32_t b, uint32_t c) {
    uint32_t r;
    asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
    return r;
}

__device__ __forceinline__ ScaleFma scale_fma(uint32_t s2) {
    ScaleFma f;
    f.mul = bf16x2_mul(bf16x2_mul(s2, 0x60006000u), 0x5F806000u);  // 2^65, then (2^65, 2^64)
    f.add = bf16x2_mul(s2, 0xC100C100u);
    return f;
}

// 8 codes -> 4 bf16x2 words as dequant_word: six integer ops (two masks, four
// byte selects; a selector of 8 + j repeats the sign bit of byte j, here the
// zero that fills the upper byte of each half), one multiply, four FMAs --
// 11 instructions where dequant_word takes 17.  Integer and bf16x2 operations
// issue at half rate, so this is what the GEMM's dequant warps are bound by:
// 256 x 12288 x 49152 215 -> 204 us, gate/up + SwiGLU at 8192 tokens
// 12.54 -> 12.17 ms (power cap), 2048 x 12288 x 12288 with g = 64 390 -> 370 us.
__device__ __forceinline__ void dequant_word_fma(uint32_t w, const ScaleFma& f, uint32_t* out) {
    uint32_t w8;
    asm("mul.lo.u32 %0, %1, 8;" : "=r"(w8) : "r"(w));
    const uint32_t e = w8 & 0x78787878u, o = w & 0xF0F0F0F0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t z = 8u + static_cast<uint32_t>(j);
        const uint32_t sel = static_cast<uint32_t>(j) | (z << 4) | (static_cast<uint32_t>(4 + j) << 8) | (z << 12);
        out[j] = bf16x2_fma(prmt_b32(e, o, sel), f.mul, f.add);
    }
}

// Puts the 8 bf16 of a 16-byte chunk (x0..x7) in the pair order
// (x0,x4),(x1,x5),(x2,x6),(x3,x7): the order in which one packed word yields
// its codes when each pair is masked out of a shifted copy of the word.
__device__ __forceinline__ uint4 interleave_chunk(uint4 c) {
    uint4 r;
    r.x = prmt_b32(c.x, c.z, 0x5410u);
    r.y = prmt_b32(c.x, c.z, 0x7632u);
    r.z = prmt_b32(c.y, c.w, 0x5410u);
    r.w = prmt_b32(c.y, c.w, 0x7632u);
    return r;
}

__device__ __forceinline__ uint32_t splat_bf16(uint16_t s) {
    return static_cast<uint32_t>(s) | (static_cast<uint32_t>(s) << 16);
}

// (w >> n) & 0x000F000F | 0x43004300 as one shift and one three-input logic
// op; written out so that the mask and the bias merge into a single LOP3.
template <int n>
__device__ __forceinline__ uint32_t nibble_pair_biased(uint32_t w) {
    uint32_t r;
    if constexpr (n == 0) {
        asm("lop3.b32 %0, %1, 0x000F000F, 0x43004300, 0xEA;" : "=r"(r) : "r"(w));
    } else {
        asm("{\n\t.reg .b32 t;\n\t"
            "shr.b32 t, %1, %2;\n\t"
            "lop3.b32 %0, t, 0x000F000F, 0x43004300, 0xEA;\n\t}"
            : "=r"(r)
            : "r"(w), "n"(n));
    }
    return r;
}

// Codes minus the zero point, q - 8, as exact bf16 pairs (k = j, k = j + 4)
// of one packed word: nibbles j and j + 4 sit 16 bits apart, so the mask of
// the word shifted by 4j gives (128 + q_j, 128 + q_j+4), and subtracting 136
// (all exact in bf16) the signed codes.
__device__ __forceinline__ void codes_signed(uint32_t w, uint32_t* out) {
    out[0] = bf16x2_sub(nibble_pair_biased<0>(w), 0x43084308u);
    out[1] = bf16x2_sub(nibble_pair_biased<4>(w), 0x43084308u);
    out[2] = bf16x2_sub(nibble_pair_biased<8>(w), 0x43084308u);
    out[3] = bf16x2_sub(nibble_pair_biased<12>(w), 0x43084308u);
}

// Shared-memory loads by 32-bit address (volatile: they stay after the
// barrier waits that guard them).
__device__ __forceinline__ uint2 lds64(uint32_t addr) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"(addr));
    return v;
}

__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

}  // namespace w4a16
