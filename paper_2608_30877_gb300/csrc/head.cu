// Linear layers of very few weight rows (N <= 8: the affinity head) for sm_103a.
//
// A 128-row MMA tile would be nearly empty and one cluster would walk K alone; here
// the tokens are split over the CTAs, and K over the threads: a thread takes 8
// consecutive k at a time, dequantises the rows' codes (wd, the format's definition)
// and accumulates in fp32 on the FMA pipe.  Per CTA the partial sums meet by shuffles
// and shared memory in a fixed order; TM tokens per CTA share one dequantisation.
// Bound by latency for few tokens (64 x 12288 x 2: 68 us as one 128-row tile, 4.8 here),
// by reading x for one or two rows (65536 tokens x 2 316 -> 241 us, 6.7 TB/s), by the
// FMAs for eight.
#include "dequant.cuh"
#include "epilogue.cuh"
#include "internal.h"

namespace w4a16 {

namespace {

constexpr int kThreads = 256;

template <int TM, int NR>
__global__ void __launch_bounds__(kThreads)
    w4a16_head_kernel(const uint4* __restrict__ x, const uint32_t* __restrict__ w,
                      const HeadParams p) {
    __shared__ float part[kThreads / 32][TM * NR];
    const int words = p.K / 8, KG = p.K / p.g, wpg = p.g / 8;
    const int m0 = blockIdx.x * TM;
    float acc[TM][NR];
#pragma unroll
    for (int t = 0; t < TM; ++t)
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[t][r] = 0.0f;
#pragma unroll 2
    for (int i = threadIdx.x; i < words; i += kThreads) {
        uint4 xv[TM];
#pragma unroll
        for (int t = 0; t < TM; ++t)
            xv[t] = m0 + t < p.M ? __ldg(x + static_cast<int64_t>(m0 + t) * words + i)
                                 : make_uint4(0, 0, 0, 0);
        uint32_t q[NR];
        uint16_t s[NR];
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            q[r] = 0x88888888u;
            s[r] = 0;
            if (r < p.N) {
                q[r] = __ldg(w + static_cast<int64_t>(r) * words + i);
                s[r] = __ldg(p.scales + static_cast<int64_t>(r) * KG + i / wpg);
            }
        }
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            uint32_t v[4];
            dequant_word(q[r], splat_bf16(s[r]), v);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float w0 = __uint_as_float(v[j] << 16);
                const float w1 = __uint_as_float(v[j] & 0xFFFF0000u);
#pragma unroll
                for (int t = 0; t < TM; ++t) {
                    const uint32_t xw = j == 0 ? xv[t].x : j == 1 ? xv[t].y : j == 2 ? xv[t].z : xv[t].w;
                    acc[t][r] = fmaf(__uint_as_float(xw << 16), w0, acc[t][r]);
                    acc[t][r] = fmaf(__uint_as_float(xw & 0xFFFF0000u), w1, acc[t][r]);
                }
            }
        }
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int t = 0; t < TM; ++t)
#pragma unroll
        for (int r = 0; r < NR; ++r) {
            float a = acc[t][r];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) part[warp][t * NR + r] = a;
        }
    __syncthreads();
    const Epilogue& e = p.epi;
    for (int i = threadIdx.x; i < TM * e.n_out; i += kThreads) {
        const int t = i / e.n_out, c = i - t * e.n_out, m = m0 + t;
        if (m >= p.M) break;
        auto z = [&](int r) {
            float a = 0.0f;
#pragma unroll
            for (int k = 0; k < kThreads / 32; ++k) a += part[k][t * NR + r];
            return e.bias != nullptr ? a + bf16_to_f32(e.bias[r]) : a;
        };
        const int64_t o = static_cast<int64_t>(m) * e.n_out + c;
        float h = e.act == kActSwiGLU ? silu_f32(z(2 * c)) * z(2 * c + 1)
                  : e.act == kActGELU ? gelu_f32(z(c))
                                      : z(c);
        if (e.residual != nullptr) h += bf16_to_f32(e.residual[o]);
        p.out[o] = f32_to_bf16_rn(h);
    }
}

template <int TM>
cudaError_t launch_tokens(const void* x, const void* w, const HeadParams& p, cudaStream_t stream) {
    auto kern = p.N <= 1   ? w4a16_head_kernel<TM, 1>
                : p.N <= 2 ? w4a16_head_kernel<TM, 2>
                : p.N <= 4 ? w4a16_head_kernel<TM, 4>
                           : w4a16_head_kernel<TM, 8>;
    kern<<<(p.M + TM - 1) / TM, kThreads, 0, stream>>>(static_cast<const uint4*>(x),
                                                       static_cast<const uint32_t*>(w), p);
    return cudaGetLastError();
}

}  // namespace

double head_cost_us(int64_t M, int64_t N, int64_t K) {
    // the FMAs behind the sums over the CTA's threads (65536 tokens, K = 64: 23 us for one row,
    // 36 for two, 60 for three or four, 16384 tokens 34 for eight; 8000 x 12288 x 4 56 us),
    // or reading x with half of the sums next to it (65536 x 12288 x 2 241 us)
    const double m = static_cast<double>(M), mk = m * static_cast<double>(K);
    const double nr = N <= 1 ? 1 : N <= 2 ? 2 : N <= 4 ? 4 : 8;  // rows the kernel computes
    const double sums = m * (1.0e-4 + 2.3e-4 * nr);
    const double fma = sums + mk * 0.64e-7 * (nr + static_cast<double>(N));
    const double read = 0.5 * sums + mk * 2.65e-7;
    return 1.7 + (read > fma ? read : fma);
}

cudaError_t launch_head(const void* x, const void* w, const HeadParams& p, int sm_count,
                        cudaStream_t stream) {
    // one token per CTA until that gives every SM four, then four
    if (p.M <= 4 * sm_count) return launch_tokens<1>(x, w, p, stream);
    return launch_tokens<4>(x, w, p, stream);
}

}  // namespace w4a16
