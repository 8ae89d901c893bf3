// Element-wise kernels: the exported dequant (bit-exact test hook) and the
// weight quantiser (weight preparation).  Both are HBM-bound streams.
#include "dequant.cuh"
#include "internal.h"

#include <cuda_bf16.h>

namespace w4a16 {

// One thread per packed 32-bit word: 8 codes of one row -> 16 bytes of bf16.
// Rows and groups lie back to back in every buffer (K is a multiple of g), so
// word i belongs to scale group i / (g / 8) whatever the row.  SHIFT: log2(g / 8)
// where g is a power of two (the 64-bit divisions of the general form, SHIFT < 0,
// cost more than the dequantisation: 12288 x 12288 93.8 us with them, 57 without,
// 6.7 TB/s, the copy bandwidth), four words in flight per thread.  Streaming
// loads and stores: nothing is read twice.
template <int SHIFT>
__global__ void __launch_bounds__(256) dequant_kernel(const uint32_t* __restrict__ w,
                                                      const uint16_t* __restrict__ scales,
                                                      uint4* __restrict__ wd, int64_t total,
                                                      int64_t words_per_group) {
    constexpr int U = 4;
    const int64_t step = static_cast<int64_t>(gridDim.x) * (256 * U);
    for (int64_t i0 = blockIdx.x * static_cast<int64_t>(256 * U) + threadIdx.x; i0 < total;
         i0 += step) {
        uint32_t q[U];
        uint16_t s[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * 256;
            if (i < total) {
                q[u] = __ldcs(w + i);
                s[u] = __ldg(scales + (SHIFT >= 0 ? i >> (SHIFT >= 0 ? SHIFT : 0) : i / words_per_group));
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * 256;
            if (i < total) {
                uint32_t v[4];
                dequant_word(q[u], splat_bf16(s[u]), v);
                __stcs(wd + i, make_uint4(v[0], v[1], v[2], v[3]));
            }
        }
    }
}

cudaError_t launch_dequant(const uint8_t* w, const uint16_t* scales, uint16_t* wd, int64_t N,
                           int64_t K, int64_t g, cudaStream_t stream) {
    const int64_t total = N * (K / 8);
    int64_t blocks = (total + 1023) / 1024;
    if (blocks > 152 * 64) blocks = 152 * 64;
    auto kern = g == 64    ? dequant_kernel<3>
                : g == 128 ? dequant_kernel<4>
                : g == 256 ? dequant_kernel<5>
                           : dequant_kernel<-1>;
    kern<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(reinterpret_cast<const uint32_t*>(w),
                                                            scales, reinterpret_cast<uint4*>(wd),
                                                            total, g / 8);
    return cudaGetLastError();
}

// The code of element v for scale s, as the format defines it.
__device__ __forceinline__ uint32_t quantize_code(float v, float s) {
    if (s == 0.0f) return 8u;
    const float r = fminf(fmaxf(rintf(__fdiv_rn(v, s)), -8.0f), 7.0f);
    return static_cast<uint32_t>(static_cast<int>(r) + 8);
}

// g = 64, 128 or 256: LANES = g / 8 lanes per group, 8 consecutive elements per
// lane (two 16-byte loads), four packed bytes out, so that a warp reads 1 KB and
// writes 128 contiguous bytes; every element is read once.  Bound by HBM:
// 12288 x 12288 277 us before (4-byte loads 16 bytes apart, each element read
// twice and divided), 106 us so, 6.4 TB/s.
// The quotient is v (1 / s) first: within 2 ulp of v / s, so its rounding to an
// integer is that of the correctly rounded quotient unless it lies within
// 2^-12 of a tie (|v / s| < 8.1, so 2 ulp are at most 2^-19); a lane with such an
// element, a non-finite one, or a scale outside [2^-100, 2^100] divides.  Rounding
// adds 1.5 2^23 + 8 (round to nearest even; the low bits are then the code), and
// the eight codes are packed by multiply-adds on the raw bits.
template <int LANES>
__global__ void __launch_bounds__(256) quantize_lanes_kernel(const float4* __restrict__ w,
                                                             uint32_t* __restrict__ packed,
                                                             uint16_t* __restrict__ scales,
                                                             int64_t total) {
    constexpr int U = 2;  // 8-element blocks in flight per lane
    const int64_t step = static_cast<int64_t>(gridDim.x) * (256 * U);
    for (int64_t i0 = blockIdx.x * static_cast<int64_t>(256 * U) + threadIdx.x;
         i0 - threadIdx.x < total; i0 += step) {
        float v[U][8];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * 256;
            float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
            if (i < total) {
                a = __ldcs(w + 2 * i);
                b = __ldcs(w + 2 * i + 1);
            }
            v[u][0] = a.x, v[u][1] = a.y, v[u][2] = a.z, v[u][3] = a.w;
            v[u][4] = b.x, v[u][5] = b.y, v[u][6] = b.z, v[u][7] = b.w;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int64_t i = i0 + u * 256;
            float amax = 0.0f;
#pragma unroll
            for (int e = 0; e < 8; ++e) amax = fmaxf(amax, fabsf(v[u][e]));
#pragma unroll
            for (int off = LANES / 2; off > 0; off >>= 1)
                amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
            const __nv_bfloat16 sb = __float2bfloat16_rn(__fdiv_rn(amax, 7.0f));
            const float s = __bfloat162float(sb);
            const float inv = __frcp_rn(s);
            constexpr float kMagic = 12582912.0f + 8.0f;
            bool plain = s >= 7.9e-31f && s <= 1.2e30f;
            uint32_t word = 0;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float t = v[u][e] * inv;
                const float r = t + kMagic;
                plain = plain && fabsf(t - (r - kMagic)) < 0.49975f;
                word += __float_as_uint(r) << (4 * e);
            }
            // every term carries 0x4B400000, the bits of 1.5 2^23
            word -= 0x4B400000u + (0x4B400000u << 4) + (0x4B400000u << 8);
            if (!plain) {
                word = 0;
#pragma unroll
                for (int e = 0; e < 8; ++e) word |= quantize_code(v[u][e], s) << (4 * e);
            }
            if (i < total) {
                __stcs(packed + i, word);
                if (threadIdx.x % LANES == 0) scales[i / LANES] = __bfloat16_as_ushort(sb);
            }
        }
    }
}

// Any other g: one warp per (row, group).  Lane l owns the g/32 consecutive elements
// starting at l*g/32 (an even count, so whole bytes).
__global__ void __launch_bounds__(256) quantize_kernel(const float* __restrict__ w,
                                                       uint8_t* __restrict__ packed,
                                                       uint16_t* __restrict__ scales, int64_t N,
                                                       int64_t K, int64_t g) {
    const int64_t KG = K / g;
    const int64_t groups = N * KG;
    const int lane = threadIdx.x & 31;
    const int per_lane = static_cast<int>(g / 32);
    const int64_t warps_total = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
    for (int64_t gi = (blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x) >> 5;
         gi < groups; gi += warps_total) {
        const int64_t n = gi / KG;
        const int64_t j = gi - n * KG;
        const float* src = w + n * K + j * g + static_cast<int64_t>(lane) * per_lane;
        float amax = 0.0f;
        for (int e = 0; e < per_lane; ++e) amax = fmaxf(amax, fabsf(src[e]));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        const __nv_bfloat16 sb = __float2bfloat16_rn(__fdiv_rn(amax, 7.0f));
        const float s = __bfloat162float(sb);
        if (lane == 0) scales[gi] = __bfloat16_as_ushort(sb);
        uint8_t* dst = packed + n * (K / 2) + (j * g + static_cast<int64_t>(lane) * per_lane) / 2;
        for (int e = 0; e < per_lane; e += 2) {
            dst[e / 2] = static_cast<uint8_t>(quantize_code(src[e], s) |
                                              (quantize_code(src[e + 1], s) << 4));
        }
    }
}

cudaError_t launch_quantize(const float* w, uint8_t* packed, uint16_t* scales, int64_t N,
                            int64_t K, int64_t g, cudaStream_t stream) {
    const int64_t groups = N * (K / g);
    if (g == 64 || g == 128 || g == 256) {
        const int64_t total = N * (K / 8);
        int64_t blocks = (total + 511) / 512;
        if (blocks > 152 * 64) blocks = 152 * 64;
        auto kern = g == 64    ? quantize_lanes_kernel<8>
                    : g == 128 ? quantize_lanes_kernel<16>
                               : quantize_lanes_kernel<32>;
        kern<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(
            reinterpret_cast<const float4*>(w), reinterpret_cast<uint32_t*>(packed), scales, total);
        return cudaGetLastError();
    }
    int64_t blocks = (groups * 32 + 255) / 256;
    if (blocks > 152 * 64) blocks = 152 * 64;
    quantize_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(w, packed, scales, N, K,
                                                                       g);
    return cudaGetLastError();
}

}  // namespace w4a16
