// Scoring readout for sm_103a: the last two modules of the screening pipeline
// (Sec. 3.3) -- the affinity head reads one hidden state per pair, and the
// predicted affinities are sorted for export.
//
//   gather_rows   dst[p, :] = src[idx[p], :] (bf16 rows, 16-byte copies);
//   topk_smallest the k smallest scores (best binders: lowest free energy),
//                 ascending by IEEE totalOrder with NaN last, ties by index.
//
// Top-k, GB300-first: one thread-block cluster of 8 CTAs (1024 threads each; 16 CTAs
// beyond 320000 scores) reads the scores once and does a radix select, most
// significant digit first, over (order-preserving 32-bit key, index) pairs.  Each CTA
// keeps the keys of its contiguous slice in shared memory (up to 40000; longer slices
// are read again) and histograms them, the first digit into four copies by
// lane, as most scores share a few exponents.  Every CTA adds up all histograms
// through distributed shared memory and finds the digit itself: one cluster
// barrier a digit of 11 bits.  The search ends with the first bin that is wanted
// whole; the digits of the index only matter where equal keys straddle the k-th.
// The selected pairs are gathered by every CTA, which ranks its share of them by
// counting smaller pairs, and stores them.  Nothing goes through global memory.
// Bound by latency (about five cluster barriers) and the first digit's atomics:
// 200000 scores, k = 1000 56 -> 21 us; 10000, k = 100 27.7 -> 11.3; 2000000, k = 1024
// 295 -> 89 (before: seven passes over the scores by scalar loads, a digit search by one
// thread and 55 sorting steps on one CTA).
#include "internal.h"

#include <atomic>
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <cstdint>
#include <utility>

namespace cg = cooperative_groups;

namespace w4a16 {

namespace {

constexpr int kTopkThreads = 1024;
constexpr int kTopkWarps = kTopkThreads / 32;
constexpr int kTopkBins = 2048;         // 11-bit digits
constexpr int kTopkCopies = 4;          // histograms of the first digit, by lane
constexpr int kTopkCache = 40 * 1000;   // keys a CTA keeps in shared memory

// Keys whose unsigned order is totalOrder on the scores; every NaN maps to
// the largest key.
__device__ __forceinline__ uint32_t order_key_f32(float f) {
    const uint32_t u = __float_as_uint(f);
    if ((u & 0x7F800000u) == 0x7F800000u && (u & 0x007FFFFFu) != 0u) return 0xFFFFFFFFu;
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

struct TopkShared {
    uint32_t keys[kTopkCache];
    // (the copies of one bin lie on different banks)
    uint32_t priv[kTopkCopies][kTopkBins + 32 / kTopkCopies];
    // this CTA's histogram of a pass, read by the other CTAs; a pass's buffer
    // is written again two passes on, two cluster barriers after the last read
    uint32_t hist[2][kTopkBins];
    unsigned long long list[kTopkMaxK];   // this CTA's selected (key << 32 | index)
    unsigned long long all[kTopkMaxK];    // every CTA's
    uint32_t warp_sum[kTopkWarps];
    uint32_t digit, before, bin;          // of the current pass
    uint32_t count;
};

// Scores are fp32, or bf16 (widened exactly: its bits are the top half of
// the fp32's).
template <bool BF16>
__device__ __forceinline__ float score_at(const void* scores, int64_t i) {
    if constexpr (BF16)
        return __uint_as_float(static_cast<uint32_t>(static_cast<const uint16_t*>(scores)[i]) << 16);
    else
        return static_cast<const float*>(scores)[i];
}

template <bool BF16>
__device__ __forceinline__ uint32_t order_key(const void* scores, int64_t i) {
    return order_key_f32(score_at<BF16>(scores, i));
}

template <bool BF16, int kTopkCtas>
__global__ void __launch_bounds__(kTopkThreads, 1)
    topk_smallest_kernel(const void* __restrict__ scores, int64_t n, int k,
                         int32_t* __restrict__ out_idx, float* __restrict__ out_val) {
    extern __shared__ __align__(16) uint8_t topk_smem[];
    TopkShared& sh = *reinterpret_cast<TopkShared*>(topk_smem);
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = static_cast<int>(cluster.block_rank());
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

    // the CTA's slice, starting on a 16-byte boundary of the scores
    constexpr int V = BF16 ? 8 : 4;
    const int64_t per = (n + kTopkCtas * V - 1) / (kTopkCtas * V) * V;
    const int64_t lo = per * rank < n ? per * rank : n;
    const int count = static_cast<int>((lo + per < n ? lo + per : n) - lo);
    const bool cached = per <= kTopkCache;

    for (int i = tid; i < static_cast<int>(sizeof(sh.priv) / 4); i += kTopkThreads)
        (&sh.priv[0][0])[i] = 0;
    if (tid == 0) sh.count = 0;
    __syncthreads();
    // ---- one read of the scores: keys, and the histogram of their first digit
    uint32_t* mine = sh.priv[lane % kTopkCopies];
    auto first = [&](int i, uint32_t key) {
        if (cached) sh.keys[i] = key;
        atomicAdd(&mine[key >> 21], 1u);
    };
    const int whole = count / V * V;
    constexpr int kLoads = 4;  // 16-byte loads in flight per thread
    for (int i0 = tid * V; i0 < whole; i0 += kLoads * kTopkThreads * V) {
        uint4 c[kLoads];
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
            const int i = i0 + u * kTopkThreads * V;
            if (i < whole)
                c[u] = __ldg(reinterpret_cast<const uint4*>(static_cast<const uint8_t*>(scores) +
                                                            (lo + i) * (BF16 ? 2 : 4)));
        }
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
            const int i = i0 + u * kTopkThreads * V;
            if (i >= whole) break;
            const uint32_t h[4] = {c[u].x, c[u].y, c[u].z, c[u].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if constexpr (BF16) {
                    first(i + 2 * e, order_key_f32(__uint_as_float(h[e] << 16)));
                    first(i + 2 * e + 1, order_key_f32(__uint_as_float(h[e] & 0xFFFF0000u)));
                } else {
                    first(i + e, order_key_f32(__uint_as_float(h[e])));
                }
            }
        }
    }
    for (int i = whole + tid; i < count; i += kTopkThreads) first(i, order_key<BF16>(scores, lo + i));
    __syncthreads();
    auto key_at = [&](int i) { return cached ? sh.keys[i] : order_key<BF16>(scores, lo + i); };

    // ---- radix select over (key, index): the k-th smallest pair, 11 bits at a
    // time, the digits of the index only where equal keys straddle the k-th (2000 equal
    // scores, k = 1: 20.5 us with all 32 bits of it, 15.2 with those of n).  A
    // pass ends the search as soon as a whole bin is wanted.  `top` holds the
    // digits found, `low` the bits below them.
    unsigned long long top = 0;
    int low = 64;
    uint32_t need = static_cast<uint32_t>(k);
    for (int pass = 0;; ++pass) {
        if (pass == 3) {  // on to the index: no pass over bits that none below n has
            low = 32 - __clz(static_cast<int>(n) - 1);
            top <<= 32 - low;
        }
        const int bits = pass == 2 ? 10 : low < 11 ? low : 11;
        uint32_t* hist = sh.hist[pass & 1];
        const int b0 = 2 * tid;  // this thread's bins
        if (pass == 0) {
            uint32_t s0 = 0, s1 = 0;
#pragma unroll
            for (int c = 0; c < kTopkCopies; ++c) {
                s0 += sh.priv[c][b0];
                s1 += sh.priv[c][b0 + 1];
            }
            hist[b0] = s0;
            hist[b0 + 1] = s1;
        } else {
            hist[b0] = hist[b0 + 1] = 0;
            __syncthreads();
            for (int i = tid; i < count; i += kTopkThreads) {
                const unsigned long long pair =
                    (static_cast<unsigned long long>(key_at(i)) << 32) | static_cast<uint32_t>(lo + i);
                if (pair >> low == top)
                    atomicAdd(&hist[static_cast<uint32_t>(pair >> (low - bits)) & ((1u << bits) - 1u)], 1u);
            }
        }
        cluster.sync();
        // every CTA adds up all histograms and finds the digit for itself
        uint32_t t0 = 0, t1 = 0;
#pragma unroll
        for (int r = 0; r < kTopkCtas; ++r) {
            const uint2 h = *reinterpret_cast<const uint2*>(
                &cluster.map_shared_rank(&sh, r)->hist[pass & 1][b0]);
            t0 += h.x;
            t1 += h.y;
        }
        uint32_t incl = t0 + t1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) sh.warp_sum[warp] = incl;
        __syncthreads();
        uint32_t before = sh.warp_sum[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, before, o);
            if (lane >= o) before += v;
        }
        before = __shfl_sync(0xffffffffu, before, warp > 0 ? warp - 1 : 0);
        before = (warp > 0 ? before : 0u) + incl - (t0 + t1);  // of all bins before b0
        if (before < need && need <= before + t0) {
            sh.digit = b0;
            sh.before = before;
            sh.bin = t0;
        } else if (before + t0 < need && need <= before + t0 + t1) {
            sh.digit = b0 + 1;
            sh.before = before + t0;
            sh.bin = t1;
        }
        __syncthreads();
        top = (top << bits) | sh.digit;
        low -= bits;
        need -= sh.before;
        if (need == sh.bin) break;
    }

    // ---- the CTA's pairs up to the bin, in any order; exactly k in the cluster
    for (int i = tid; i < count; i += kTopkThreads) {
        const unsigned long long pair =
            (static_cast<unsigned long long>(key_at(i)) << 32) | static_cast<uint32_t>(lo + i);
        if (pair >> low <= top) sh.list[atomicAdd(&sh.count, 1u)] = pair;
    }
    cluster.sync();
    // ---- every CTA gathers all k and ranks its share of them
    if (tid < k) {
        uint32_t at = tid;
        int r = 0;
        for (; r < kTopkCtas - 1; ++r) {
            const uint32_t c = cluster.map_shared_rank(&sh, r)->count;
            if (at < c) break;
            at -= c;
        }
        sh.all[tid] = cluster.map_shared_rank(&sh, r)->list[at];
    }
    auto done = cluster.barrier_arrive();  // this CTA has read the others' lists
    __syncthreads();
    constexpr int kLanes = 8;  // threads per ranked pair
    const int e0 = k * rank / kTopkCtas, e1 = k * (rank + 1) / kTopkCtas;
    for (int e = e0 + tid / kLanes; e - tid / kLanes < e1; e += kTopkThreads / kLanes) {
        const unsigned long long p = e < e1 ? sh.all[e] : 0ull;
        uint32_t pos = 0;
        for (int j = tid % kLanes; j < k; j += kLanes) pos += sh.all[j] < p;
#pragma unroll
        for (int o = 1; o < kLanes; o <<= 1) pos += __shfl_xor_sync(0xffffffffu, pos, o);
        if (e < e1 && tid % kLanes == 0) {
            const uint32_t idx = static_cast<uint32_t>(p);
            out_idx[pos] = static_cast<int32_t>(idx);
            out_val[pos] = score_at<BF16>(scores, idx);
        }
    }
    cluster.barrier_wait(std::move(done));
}

// A CTA copies one kGatherChunk-element piece of a row at a time (blockIdx.y
// and on), in 16-byte units where rows have whole ones: 64 rows of 24 KB on one CTA each
// were a serial chain of six loads and stores per thread.  Else element by element, all
// of a thread's eight read before any is stored (5000 rows of 12289: 72 us by whole rows, 123
// in pieces one element after the other, 52 so).
constexpr int kGatherThreads = 256;
constexpr int kGatherChunk = 8 * kGatherThreads;

template <bool WHOLE>
__global__ void __launch_bounds__(kGatherThreads)
    gather_rows_kernel(const uint16_t* __restrict__ src, int64_t src_rows, int64_t D,
                       const int32_t* __restrict__ idx, int64_t P, uint16_t* __restrict__ dst,
                       int* status) {
    const int64_t j_step = static_cast<int64_t>(gridDim.y) * kGatherChunk;
    for (int64_t p = blockIdx.x; p < P; p += gridDim.x) {
        const int32_t r = idx[p];
        const bool ok = r >= 0 && r < src_rows;
        if (!ok && threadIdx.x == 0 && blockIdx.y == 0)
            atomicCAS(status, 0, 1 /* W4A16_ERR_INVALID_ARG; the first error is kept */);
        const uint16_t* s = src + (ok ? static_cast<int64_t>(r) : 0) * D;
        uint16_t* d = dst + p * D;
        for (int64_t j0 = static_cast<int64_t>(blockIdx.y) * kGatherChunk; j0 < D; j0 += j_step) {
            if constexpr (WHOLE) {
                // (two pieces in flight)
                const int64_t j = j0 + 8 * threadIdx.x, k = j + j_step;
                uint4 a = make_uint4(0, 0, 0, 0), b = a;
                if (ok && j < D) a = __ldg(reinterpret_cast<const uint4*>(s + j));
                if (ok && k < D) b = __ldg(reinterpret_cast<const uint4*>(s + k));
                if (j < D) *reinterpret_cast<uint4*>(d + j) = a;
                if (k < D) *reinterpret_cast<uint4*>(d + k) = b;
                j0 += j_step;
            } else {
                const int left = static_cast<int>(D - j0 < kGatherChunk ? D - j0 : kGatherChunk);
                const uint16_t* sj = s + j0 + threadIdx.x;
                uint16_t* dj = d + j0 + threadIdx.x;
                uint16_t v[8];
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    v[u] = ok && static_cast<int>(threadIdx.x) + u * kGatherThreads < left
                               ? __ldg(sj + u * kGatherThreads) : static_cast<uint16_t>(0);
#pragma unroll
                for (int u = 0; u < 8; ++u)
                    if (static_cast<int>(threadIdx.x) + u * kGatherThreads < left)
                        dj[u * kGatherThreads] = v[u];
            }
        }
    }
}

// Rows of fewer units (uint4, or pairs of elements) than a CTA has threads: the units of all rows
// in one run over the threads, kGatherUnits in flight each (100000 rows of 100 elements: a
// row per CTA 51 us, 72 in pieces as above, 20 so; of 128: 55, 57, 6.4; of 1: 39, 56, 2.7).
// Index: 32 bits where that counts the units.
constexpr int kGatherUnits = 4;

template <typename Unit, typename Index>
__global__ void __launch_bounds__(kGatherThreads)
    gather_units_kernel(const Unit* __restrict__ src, int64_t src_rows, Index per_row,
                        const int32_t* __restrict__ idx, Index total, Unit* __restrict__ dst,
                        int* status) {
    constexpr Index kBlock = kGatherThreads * kGatherUnits;
    const Index step = static_cast<Index>(gridDim.x) * kBlock;
    for (Index i0 = static_cast<Index>(blockIdx.x) * kBlock; i0 < total;
         i0 = total - i0 > step ? i0 + step : total) {  // (no overflow past total)
        Unit v[kGatherUnits];
#pragma unroll
        for (int u = 0; u < kGatherUnits; ++u) {
            const Index at = static_cast<Index>(threadIdx.x + u * kGatherThreads);
            if (at >= total - i0) continue;
            const Index p = (i0 + at) / per_row, j = i0 + at - p * per_row;
            const int32_t r = __ldg(idx + p);
            const bool ok = r >= 0 && r < src_rows;
            if (!ok && j == 0) atomicCAS(status, 0, 1 /* W4A16_ERR_INVALID_ARG */);
            v[u] = Unit{};
            if (ok) v[u] = __ldg(src + static_cast<int64_t>(r) * per_row + j);
        }
#pragma unroll
        for (int u = 0; u < kGatherUnits; ++u) {
            const Index at = static_cast<Index>(threadIdx.x + u * kGatherThreads);
            if (at < total - i0) dst[i0 + at] = v[u];
        }
    }
}

template <typename Unit>
void launch_gather_units(const uint16_t* src, int64_t src_rows, int64_t per_row, const int32_t* idx,
                         int64_t P, uint16_t* dst, int* status, int sm_count, cudaStream_t stream) {
    const int64_t total = P * per_row, block = kGatherThreads * kGatherUnits;
    const int64_t need = (total + block - 1) / block, most = 8 * static_cast<int64_t>(sm_count);
    const unsigned grid = static_cast<unsigned>(need < most ? need : most);
    const Unit* s = reinterpret_cast<const Unit*>(src);
    Unit* d = reinterpret_cast<Unit*>(dst);
    if (total < (int64_t{1} << 32) - block)
        gather_units_kernel<Unit, uint32_t><<<grid, kGatherThreads, 0, stream>>>(
            s, src_rows, static_cast<uint32_t>(per_row), idx, static_cast<uint32_t>(total), d, status);
    else
        gather_units_kernel<Unit, uint64_t><<<grid, kGatherThreads, 0, stream>>>(
            s, src_rows, static_cast<uint64_t>(per_row), idx, static_cast<uint64_t>(total), d, status);
}

template <bool BF16, int CTAS>
cudaError_t topk_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) {
    auto kern = topk_smallest_kernel<BF16, CTAS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         sizeof(TopkShared));
    if (e == cudaSuccess && CTAS > 8)
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = CTAS;
    attr->val.clusterDim.y = 1;
    attr->val.clusterDim.z = 1;
    cfg->gridDim = dim3(CTAS);
    cfg->blockDim = dim3(kTopkThreads);
    cfg->dynamicSmemBytes = sizeof(TopkShared);
    cfg->attrs = attr;
    cfg->numAttrs = 1;
    return e;
}

template <bool BF16, int CTAS>
cudaError_t launch_topk(const void* scores, int64_t n, int k, int32_t* out_idx, float* out_val,
                        cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cudaError_t e = topk_config<BF16, CTAS>(&cfg, attr);
    if (e != cudaSuccess) return e;
    cfg.stream = stream;
    e = cudaLaunchKernelEx(&cfg, topk_smallest_kernel<BF16, CTAS>, scores, n, k, out_idx, out_val);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

// Whether the device can place a cluster of 16 of these CTAs; asked once per device.
bool wide_cluster_fits() {
    constexpr int kMaxDev = 64;
    static std::atomic<int> cache[kMaxDev] = {};  // 0: not asked, 1: yes, 2: no
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return false;
    int v = cache[dev].load(std::memory_order_relaxed);
    if (v == 0) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        int clusters = 0;
        v = topk_config<false, 16>(&cfg, attr) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&clusters, topk_smallest_kernel<false, 16>, &cfg) ==
                        cudaSuccess &&
                    clusters > 0
                ? 1
                : 2;
        cudaGetLastError();  // a failed query leaves no sticky error for the next launch
        cache[dev].store(v, std::memory_order_relaxed);
    }
    return v == 1;
}

}  // namespace

cudaError_t launch_topk_smallest(const void* scores, bool bf16, int64_t n, int k,
                                 int32_t* out_idx, float* out_val, cudaStream_t stream) {
    // 16 CTAs (a cluster size beyond the portable 8) where 8 cannot keep their keys in
    // shared memory and the GPU can place them: 2000000 scores 89 us against 127.
    // Below that their longer barriers cost more (200000: 28 against 21).
    const bool wide = n > 8 * kTopkCache && wide_cluster_fits();
    return bf16 ? (wide ? launch_topk<true, 16>(scores, n, k, out_idx, out_val, stream)
                        : launch_topk<true, 8>(scores, n, k, out_idx, out_val, stream))
                : (wide ? launch_topk<false, 16>(scores, n, k, out_idx, out_val, stream)
                        : launch_topk<false, 8>(scores, n, k, out_idx, out_val, stream));
}

cudaError_t launch_gather_rows(const uint16_t* src, int64_t src_rows, int64_t D,
                               const int32_t* idx, int64_t P, uint16_t* dst, int* status,
                               int sm_count, cudaStream_t stream) {
    const bool whole = (D & 7) == 0;  // rows of 16-byte units (bases are 16-byte aligned)
    if ((whole ? D / 8 : D / 2) < kGatherThreads) {
        if (whole)
            launch_gather_units<uint4>(src, src_rows, D / 8, idx, P, dst, status, sm_count, stream);
        else
            launch_gather_units<uint16_t>(src, src_rows, D, idx, P, dst, status, sm_count, stream);
        return cudaGetLastError();
    }
    // pieces of rows until the CTAs fill the SMs eight times over
    const int64_t pieces = (D + kGatherChunk - 1) / kGatherChunk;
    const int64_t want = 8 * static_cast<int64_t>(sm_count);
    const int64_t bx = P < want ? P : want;
    const int64_t by = pieces < (want + bx - 1) / bx ? pieces : (want + bx - 1) / bx;
    auto kern = whole ? gather_rows_kernel<true> : gather_rows_kernel<false>;
    kern<<<dim3(static_cast<unsigned>(bx), static_cast<unsigned>(by)), kGatherThreads, 0, stream>>>(
        src, src_rows, D, idx, P, dst, status);
    return cudaGetLastError();
}

}  // namespace w4a16
