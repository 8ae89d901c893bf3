// Element math of the fused epilogue (operator fusion of what follows a
// linear layer, Sec. 5): z = acc + bias; SwiGLU h = silu(z_gate) * z_up with
// silu(t) = t / (1 + e^-t); GELU h = z * Phi(z) = z/2 (1 + erf(z / sqrt 2));
// out = h + residual.  fp32 throughout, one bf16 rounding at the store.
#pragma once

#include "internal.h"

#include <cstdint>

namespace w4a16 {

enum : int { kActNone = 0, kActSwiGLU = 1, kActGELU = 2 };

__device__ __forceinline__ float bf16_to_f32(uint16_t h) {
    return __uint_as_float(static_cast<uint32_t>(h) << 16);
}

__device__ __forceinline__ float silu_f32(float t) { return t / (1.0f + expf(-t)); }

__device__ __forceinline__ float gelu_f32(float t) {
    return 0.5f * t * (1.0f + erff(t * 0.70710678118654752f));
}

__device__ __forceinline__ uint16_t f32_to_bf16_rn(float f) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %1;" : "=r"(r) : "f"(f));
    return static_cast<uint16_t>(r & 0xFFFFu);
}

// bf16 pair (lo, hi) of two fp32 values.
__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

// Output of CNT consecutive tokens m0 .. of one weight row n per lane, from the
// finished sums v; lane and n have the same parity, and tokens from m_end on and
// lanes that are not `ok` store nothing (all lanes of the warp call).
// Neighbouring lanes swap values: the even one finishes the even tokens, the odd
// one the odd tokens, and each store (and residual load) is a 32-bit word of two
// columns; SwiGLU pairs rows (n, n ^ 1) = (gate, up) of one column, whose values
// meet the same way.  The residuals are read before anything is stored: they may be
// the output, and read one by one after the stores they are a chain of memory latencies
// (333 x 12288 x 12288 on the same buffers call after call, with a residual: 117 us one by
// one in 16-bit loads, 88 read first, 70 in pairs; with SwiGLU 79 us at 16 bits and no
// swap, 70 so).
template <int ACT, int CNT, bool PLAIN = false>
__device__ __forceinline__ void store_tokens_act(const Epilogue& e, uint16_t* out,
                                                 const float (&v)[CNT], int m0, int m_end, int n,
                                                 bool ok, float bias, int lane) {
    static_assert(CNT % 2 == 0, "token pairs");
    constexpr int H = CNT / 2;
    const bool odd = (lane & 1) != 0;
    if constexpr (ACT != kActSwiGLU) {
        if ((e.n_out & 1) != 0) {  // rows of odd width: columns cannot pair up
            if constexpr (PLAIN) {
                // addresses that advance: with a 64-bit product per store 16384 x 64 x 12289
                // takes 208 us against 125, 1000 x 64 x 36865 45.5 against 30 (fused they gain 10%
                // in a GEMM with GELU and cost 10 to 25% with a residual and where K is split)
                const int count = ok ? m_end - m0 : 0;  // tokens to store
                uint16_t* dst = out + static_cast<int64_t>(m0) * e.n_out + n;
#pragma unroll
                for (int j = 0; j < CNT; ++j, dst += e.n_out)
                    if (j < count) *dst = f32_to_bf16_rn(v[j]);
            } else {
                float r[CNT];
#pragma unroll
                for (int j = 0; j < CNT; ++j)
                    r[j] = e.residual != nullptr && ok && m0 + j < m_end
                               ? bf16_to_f32(e.residual[static_cast<int64_t>(m0 + j) * e.n_out + n])
                               : 0.0f;
#pragma unroll
                for (int j = 0; j < CNT; ++j) {
                    const float z = v[j] + bias;
                    const float h = (ACT == kActGELU ? gelu_f32(z) : z) + r[j];
                    if (ok && m0 + j < m_end)
                        out[static_cast<int64_t>(m0 + j) * e.n_out + n] = f32_to_bf16_rn(h);
                }
            }
            return;
        }
    }
    // this lane's tokens m0 + odd, + 2, ...; its column(s)
    const int col = ACT == kActSwiGLU ? n >> 1 : n & ~1;
    const int first = m0 + (odd ? 1 : 0);
    const int64_t at = static_cast<int64_t>(first) * e.n_out + col;
    const int64_t step = 2 * static_cast<int64_t>(e.n_out);
    const int count = ok ? (m_end - first + 1) / 2 : 0;  // of its tokens, those to store
    uint32_t res[H];
#pragma unroll
    for (int j = 0; j < H; ++j) res[j] = 0;
    if (e.residual != nullptr) {
        const uint16_t* src = e.residual + at;
#pragma unroll
        for (int j = 0; j < H; ++j, src += step) {
            if (j < count)
                res[j] = ACT == kActSwiGLU ? static_cast<uint32_t>(*src)
                                           : *reinterpret_cast<const uint32_t*>(src);
        }
    }
    uint16_t* dst = out + at;
#pragma unroll
    for (int j = 0; j < H; ++j, dst += step) {
        float a = v[2 * j] + bias, b = v[2 * j + 1] + bias;  // tokens 2j, 2j + 1 of row n
        if constexpr (ACT == kActGELU) {
            a = gelu_f32(a);
            b = gelu_f32(b);
        }
        const float other = __shfl_xor_sync(0xffffffffu, odd ? a : b, 1);
        const float lo = odd ? other : a, hi = odd ? b : other;  // rows n & ~1, n | 1
        if constexpr (ACT == kActSwiGLU) {
            const float h = silu_f32(lo) * hi + __uint_as_float(res[j] << 16);
            if (j < count) *dst = f32_to_bf16_rn(h);
        } else {
            const uint32_t w = pack_bf16x2(lo + __uint_as_float(res[j] << 16),
                                           hi + __uint_as_float(res[j] & 0xFFFF0000u));
            if (j < count) *reinterpret_cast<uint32_t*>(dst) = w;
        }
    }
}

// FUSED = false: no bias, activation or residual (none of their code or registers).
template <bool FUSED, int CNT>
__device__ __forceinline__ void store_tokens(const Epilogue& e, uint16_t* out,
                                             const float (&v)[CNT], int m0, int m_end, int n,
                                             bool ok, float bias, int lane) {
    if constexpr (!FUSED) {
        const Epilogue plain{nullptr, nullptr, kActNone, e.n_out};
        store_tokens_act<kActNone, CNT, true>(plain, out, v, m0, m_end, n, ok, 0.0f, lane);
    } else if (e.act == kActSwiGLU) {
        store_tokens_act<kActSwiGLU, CNT>(e, out, v, m0, m_end, n, ok, bias, lane);
    } else if (e.act == kActGELU) {
        store_tokens_act<kActGELU, CNT>(e, out, v, m0, m_end, n, ok, bias, lane);
    } else {
        store_tokens_act<kActNone, CNT>(e, out, v, m0, m_end, n, ok, bias, lane);
    }
}

}  // namespace w4a16
