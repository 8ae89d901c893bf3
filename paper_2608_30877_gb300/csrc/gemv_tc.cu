// Streaming int4-dequant + matmul on the 5th-generation tensor core for few
// tokens (M <= 128, every group size, and more tokens in 128-token tiles
// where the GEMM's CTA pairs would leave SMs idle): the regime where the whole
// packed weight matrix streams from HBM about once per call.
//
// out[m, n] = sum_k x[m, k] * wd[n, k],   wd = RNE_bf16((q[n, k] - 8) * s[n, k / g])
//
// (the same weights as w4a16_dequant and the large-M GEMM: the result differs
// from theirs only in the fp32 summation order).
//
// Per CTA (persistent, one per SM): a contiguous range of RB <= 384 weight
// rows as up to three MMA tiles of 128 rows, each with one fp32 accumulator of
// NTOK = 32 to 128 token columns in tensor memory for the whole K walk.
// Per stage of 128 k:
//   warp 0      TMA: two 64-k boxes of x (NTOK token rows, 128-byte swizzle,
//               rows >= M zero-filled) and two boxes of RB/2 rows x 64 B of
//               packed weights (64-byte swizzle) into a ring of S stages;
//   warps 4..   dequant: thread = one weight row of one tile (its TMEM lane);
//               wd as bf16 pairs in k order (one FMA per pair, dequant.cuh) ->
//               tcgen05.st into the tile's ring of SA A stages of AK k; after the last
//               stage, the epilogue: tcgen05.ld of the row's accumulators in slices
//               of 32 tokens, each slice's (fused) epilogue from registers;
//   warps 1..3  one per tile: D_t[128 x NTOK] += A_t[128 x 16] x B[NTOK x 16]^T (A
//               from tensor memory, B = x in shared memory).  One commit frees
//               the A stage, one the TMA stage (x by the MMAs, the weights by the
//               row warps before them).
// Narrow layers split K: `split` CTAs of a cluster share one chunk of rows, each
// walks its slice of K, and the partial sums meet in distributed shared memory, 32
// tokens at a time, each CTA finishing its share of them in the order of the
// ranks (deterministic).  12288 rows on 152 SMs are 82 rows, one 128-row tile, per
// CTA without a split, and a lone tile runs at the latency of its four row
// warps (0.47 us per stage whatever M): K = 49152 at M = 100 with bias and residual,
// L2 flushed, 398 us (before) -> 120 us (clusters of 4, 342 rows each); 12288 x 12288 at M =
// 24 56 -> 23 us.
//
// What bounds it (K = 12288, 152 SMs): the row warps' latency and issue slots, not the
// tensor pipe: a stage costs 0.39-0.50, 0.51-0.71, 0.62-1.05 us for one, two, three
// tiles (N = 49152, one launch after another: 61 us at M <= 32, 77 at 64, 85 at 96, 111 at
// 112, 112 at 128; 63, 78, 84, 103 and 104 where these stages were fitted).  In order,
// what brought it there from 92, 103, 137, 137 and 139: weights dequantised in k order,
// with no x reorder warp, through one FMA, operands in uniform registers, addresses that
// only advance (72, 80, 86, -, 110); then, from stamps of a row warp, whose 1540 clocks
// per stage were two barrier polls of 190-230 that found their barriers long complete,
// 310 to read the codes and dequantise half, 340 for the other half, 110 for the stores and 360
// of scales and votes: the two polls under way together, and the next stage's scales
// prepared during the stores where a stage is one A stage (in more, smaller A stages that
// is slower: 64 tokens 82 against 79 us).
// tcgen05.mma with A in tensor memory runs at 18 / 32 / 64 clocks for 32 / 64 /
// 128 columns with three independent accumulators, 44 with one (measured alone), so
// the MMAs need 0.22-0.8 us of a stage.  From 97 tokens on three tiles leave the A ring
// only two or three slots of a quarter stage.  Token columns: whole output slices of 32, and
// 112, which leave the ring a third slot there and cost less of a stage (M = 112 with 112 columns
// and 128 with 128: 111 and 112 us at N = 49152, 74 and 80 at 36864, 45 and 46 at 19456); 48 and 80
// have not been tried.
// A stage in which a row of the warp has a scale of 2^-2 or more takes the general dequantisation
// (dequant.cuh): if all do, M = 8 to 32 95 us at N = 49152, 80 at 36864, where the warp-level
// kernel takes 65 and 52 up to 8 tokens (W4A16_SMALL_M=mma keeps a model of such scales on
// it; those of weights N(0, 0.02) are near 2^-7).  Constants shifted for such rows were measured: the
// ordinary call then takes 2 to 4% more, whichever way the second walk is kept out of the
// first one's code.
// Measured and not kept (M <= 32): two groups of row warps per tile (99 us: the A ring is
// too short for them), the next stage's codes read before this one's stores end (71) or
// after (66), one issuing warp for all tiles (92), a rolled dequant loop (78), 16 token
// columns for M <= 16 (67).
//
// Every wait is bounded (ptx.cuh); on a timeout the kernel records
// W4A16_ERR_TIMEOUT, drains its copies and MMAs, frees tensor memory and
// returns.
#include "dequant.cuh"
#include "epilogue.cuh"
#include "internal.h"
#include "ptx.cuh"

#include <atomic>

namespace w4a16 {

namespace {


constexpr int kTilesMax = 3;      // MMA tiles of 128 rows per CTA, at most
constexpr int kGroupK = 128;      // k per TMA stage
constexpr int kFirstRowWarp = 4;  // warps 1..3 issue the MMAs of tiles 0..2

// 32 lanes x 16 columns of 32 bits (see tmem_st_32x32b_x32).
__device__ __forceinline__ void tmem_st_32x32b_x16(uint32_t taddr, const uint32_t* v) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
        "r"(v[15])
        : "memory");
}

// TILES: MMA tiles of 128 rows a CTA holds (2 or 3); NTOK: token columns.
template <int NTOK, int TILES_>
struct TLayout {
    static_assert(NTOK % 16 == 0 && NTOK <= 128, "MMA N for M = 128");
    static constexpr int TILES = TILES_;
    static constexpr int ROWS_MAX = 128 * TILES;                     // rows per CTA chunk
    static constexpr int X_BOX = NTOK * 128;                         // 64 k x NTOK tokens
    static constexpr int X_BYTES = 2 * X_BOX;
    static constexpr int W_HALF = (ROWS_MAX / 2) * (kGroupK / 2);    // ROWS_MAX / 2 rows x 64 B
    static constexpr int W_BYTES = 2 * W_HALF;
    static constexpr int STAGE = X_BYTES + W_BYTES;                  // x, then the weights
    // TMA slots: what 224 KB hold, at most 7
    static constexpr int S_FIT = (222 * 1024) / STAGE;
    static constexpr int S = S_FIT < 7 ? S_FIT : 7;
    // tensor memory: the accumulators (TILES x NTOK columns), then SA A stages
    // of AK k (TILES x AK / 2 columns each)
    static constexpr int D_COLS = TILES * NTOK;
    static constexpr int A_FREE = 512 - D_COLS;
    static constexpr int AK = A_FREE / (TILES * 64) >= 2 ? 128 : A_FREE / (TILES * 32) >= 2 ? 64 : 32;
    static constexpr int SA = A_FREE / (TILES * (AK / 2));
    static constexpr int SUB = kGroupK / AK;   // A stages per TMA stage
    static constexpr int CHUNKS = AK / 32;     // 16-byte chunks (32 codes) per row and A stage
    static constexpr int A_COL = 512 - SA * TILES * (AK / 2);
    static constexpr int A_COLS = TILES * (AK / 2);
    static constexpr int TMEM_COLS = 512;
    static constexpr int ROW_WARPS = 4 * TILES;
    static constexpr int THREADS = 32 * (kFirstRowWarp + ROW_WARPS);
    // full_tma[S], empty_smem[S], then per tile: full_a[SA], empty_a[SA],
    // d_full, d_empty, drain
    static constexpr int BAR_OFF = S * STAGE;
    static constexpr int TILE_BARS = 2 * SA + 3;
    static constexpr int NBARS = 2 * S + TILES * TILE_BARS;
    static constexpr int MISC_OFF = BAR_OFF + NBARS * 8;
    static constexpr int SMEM_BYTES = MISC_OFF + 16 + 1024;          // + 1024-B alignment slack
    // split K: partial sums of a slice of EC tokens, double-buffered, over the
    // stages once they are consumed
    static constexpr int EC = 32;  // (reduce_slice)
    static constexpr int PART = ROWS_MAX * EC * 4;
    static_assert(2 * PART <= S * STAGE, "partial sums fit the stages");
    static_assert(SA >= 2 && D_COLS <= A_COL, "tensor memory holds 512 columns");
    static_assert(X_BOX % 1024 == 0 && W_HALF % 1024 == 0 && STAGE % 1024 == 0,
                  "swizzled boxes keep 1024-byte alignment");
    static_assert(S >= 2 && SMEM_BYTES <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ float ld_shared_cluster_f32(uint32_t addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
    return v;
}

// Sums of one row over the SP CTAs of the cluster, in the order of the ranks,
// and their output: the tokens [rank 32 / SP, ..) of a slice of 32.  All the
// remote loads are issued before the first sum (one round trip per slice).
template <int SP, bool FUSED>
__device__ __forceinline__ void reduce_slice(const GemvParams& p, uint32_t part, int pitch, int rank,
                                             int r, float bias, int m, int m_end, int n, bool valid,
                                             int lane) {
    constexpr int PER = 32 / SP;
    float v[SP][PER];
#pragma unroll
    for (int c = 0; c < SP; ++c) {
        const uint32_t at = mapa_shared(part + 4u * (rank * PER * pitch + r), c);
#pragma unroll
        for (int j = 0; j < PER; ++j) v[c][j] = ld_shared_cluster_f32(at + 4u * j * pitch);
    }
    float sum[PER];
#pragma unroll
    for (int j = 0; j < PER; ++j) {
        sum[j] = v[0][j];
#pragma unroll
        for (int c = 1; c < SP; ++c) sum[j] += v[c][j];
    }
    store_tokens<FUSED, PER>(p.epi, p.out, sum, m + rank * PER, m_end, n, valid, bias, lane);
}

template <int NTOK, int TILES, bool FUSED, bool SPLIT>
__global__ void __launch_bounds__(TLayout<NTOK, TILES>::THREADS, 1)
    w4a16_gemv_tc_kernel(const __grid_constant__ CUtensorMap tmap_x,
                         const __grid_constant__ CUtensorMap tmap_w, const GemvParams p) {
    using L = TLayout<NTOK, TILES>;
    constexpr int S = L::S, SA = L::SA, SUB = L::SUB;
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t* smem = smem_raw + (sbase - raw);

    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int RB = p.rows_per_cta;

    const uint32_t bars = sbase + L::BAR_OFF;
    auto full_tma = [&](int s) { return bars + 8u * s; };
    auto empty_smem = [&](int s) { return bars + 8u * (S + s); };
    auto tile_bar = [&](int t, int i) { return bars + 8u * (2 * S + t * L::TILE_BARS + i); };
    auto full_a = [&](int t, int a) { return tile_bar(t, a); };
    auto empty_a = [&](int t, int a) { return tile_bar(t, SA + a); };
    auto d_full = [&](int t) { return tile_bar(t, 2 * SA); };
    auto d_empty = [&](int t) { return tile_bar(t, 2 * SA + 1); };
    auto drain = [&](int t) { return tile_bar(t, 2 * SA + 2); };
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::MISC_OFF);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::MISC_OFF + 4);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(full_tma(s), 1);
            mbar_init(empty_smem(s), p.nt);  // every tile's MMAs
        }
        for (int t = 0; t < p.nt; ++t) {
            const int warps = (RB - 128 * t + 31) / 32 < 4 ? (RB - 128 * t + 31) / 32 : 4;
            for (int a = 0; a < SA; ++a) {
                mbar_init(full_a(t, a), warps);  // the row warps of the stage's group
                mbar_init(empty_a(t, a), 1);
            }
            mbar_init(d_full(t), 1);
            mbar_init(d_empty(t), warps);
            mbar_init(drain(t), 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
        prefetch_tmap(&tmap_x);
        prefetch_tmap(&tmap_w);
    }
    if (warp == 1) {
        tmem_alloc(smem_u32(tmem_slot), L::TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_launch_dependents();
    grid_wait();

    // The CTA's stages: all of K, or its slice of it among the CTAs of the
    // cluster; walked from a starting point of its own, so that the CTAs read
    // different x slices from L2 at any moment.
    const int KS = (p.K + kGroupK - 1) / kGroupK;
    const int rank = SPLIT ? static_cast<int>(cluster_ctarank()) : 0;
    const int k_first = SPLIT ? static_cast<int>(static_cast<int64_t>(KS) * rank / p.split) : 0;
    const int k_count =
        (SPLIT ? static_cast<int>(static_cast<int64_t>(KS) * (rank + 1) / p.split) : KS) - k_first;
    const int chunk0 = SPLIT ? static_cast<int>(blockIdx.x) / p.split : static_cast<int>(blockIdx.x);
    const int chunk_step = SPLIT ? p.num_chunks : static_cast<int>(gridDim.x);
    const int rot = k_first + static_cast<int>(static_cast<int64_t>(chunk0) * k_count / chunk_step);
    const int k_end = k_first + k_count;

    const int row_tile = (warp - kFirstRowWarp) >> 2;             // row warps: MMA tile
    // warps wholly past the chunk's rows do nothing
    const bool row_warp = warp >= kFirstRowWarp && row_tile * 128 + (warp & 3) * 32 < RB;
    const int sub = warp & 3;                                     // TMEM sub-partition
    const int r = row_tile * 128 + sub * 32 + lane;               // local row
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(sub * 32) << 16);
    bool ok = true;

    if (warp == 0) {
        // ------------------------------------------------------------ TMA producer
        if (lane == 0) {
            const uint32_t tx = L::X_BYTES + static_cast<uint32_t>(RB) * (kGroupK / 2);
            uint32_t it = 0;
            for (int chunk = chunk0; ok && chunk < p.num_chunks; chunk += chunk_step) {
                const int tt = chunk / p.row_chunks;
                const int row0 = (chunk - tt * p.row_chunks) * RB, m0 = tt * NTOK;
                int kk = rot;
                for (int g = 0; g < k_count; ++g, ++it) {
                    const int s = it % S;
                    if (!wait_one<false, 64>(empty_smem(s), ((it / S) & 1u) ^ 1u, abort_flag,
                                             p.status, p.wait_ns)) {
                        ok = false;
                        break;
                    }
                    mbar_arrive_expect_tx(full_tma(s), tx);
                    const uint32_t st = sbase + s * L::STAGE;
                    const uint32_t end = sbase + L::BAR_OFF;
                    if (dbg_check(tma_box_ok(st, L::X_BOX, 1024, sbase, end, kk * kGroupK, 2) &&
                                      tma_box_ok(st + L::X_BOX, L::X_BOX, 1024, sbase, end,
                                                 kk * kGroupK + 64, 2),
                                  p.status)) {
                        tma_load_2d(st, &tmap_x, full_tma(s), kk * kGroupK, m0);
                        tma_load_2d(st + L::X_BOX, &tmap_x, full_tma(s), kk * kGroupK + 64, m0);
                    }
                    const uint32_t wbox = static_cast<uint32_t>(RB / 2) * (kGroupK / 2);
                    if (dbg_check(wbox <= L::W_HALF &&
                                      tma_box_ok(st + L::X_BYTES, wbox, 1024, sbase, end,
                                                 kk * (kGroupK / 2), 1) &&
                                      tma_box_ok(st + L::X_BYTES + L::W_HALF, wbox, 1024, sbase,
                                                 end, kk * (kGroupK / 2), 1),
                                  p.status)) {
                        tma_load_2d(st + L::X_BYTES, &tmap_w, full_tma(s), kk * (kGroupK / 2),
                                    row0);
                        tma_load_2d(st + L::X_BYTES + L::W_HALF, &tmap_w, full_tma(s),
                                    kk * (kGroupK / 2), row0 + RB / 2);
                    }
                    if (it == 0 &&
                        !short_limit_ok(full_tma(0), 0, abort_flag, p.status, p.wait_ns)) {
                        ok = false;
                        ++it;
                        break;
                    }
                    if (++kk == k_end) kk = k_first;
                }
            }
            // every load this thread issued has landed before exit
            const uint32_t last = it < static_cast<uint32_t>(S) ? it : S;
            for (uint32_t i = it - last; i < it; ++i) settle(full_tma(i % S), (i / S) & 1u);
        }
    } else if (warp < kFirstRowWarp) {
        // ------------------------------------------------------------ MMA issuers
        // one thread per tile; tiles past the chunk's rows, t >= p.nt, are not computed
        // (whole warps run the loops, so that the operands stay in uniform registers)
        const int t = warp - 1;
        if (t < p.nt) {
            constexpr uint32_t idesc = idesc_bf16_f32(128, NTOK);
            int s = 0, a = 0;
            uint32_t pa = 0, nchunk = 0;
            bool issued = false;
            for (int chunk = chunk0; ok && chunk < p.num_chunks; chunk += chunk_step, ++nchunk) {
                // the epilogue has read the previous chunk's accumulators
                if (nchunk > 0 &&
                    !wait_warp(d_empty(t), (nchunk - 1u) & 1u, abort_flag, p.status, p.wait_ns)) {
                    ok = false;
                    break;
                }
                for (int g = 0; ok && g < k_count; ++g) {
                    const uint64_t bdesc = sdesc_kmajor_sw128(sbase + s * L::STAGE);
#pragma unroll
                    for (int h = 0; h < SUB; ++h) {

                        // the A stage is written; its row warps waited for the
                        // stage's copies, so x has landed too
                        if (!wait_warp(full_a(t, a), pa, abort_flag, p.status, p.wait_ns)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint32_t a_tm = tmem + L::A_COL + a * L::A_COLS + t * (L::AK / 2);
                        if (elect_one()) {
#pragma unroll
                            for (int ks = 0; ks < L::AK / 16; ++ks) {
                                // k offset in the group -> x box (64 k) and 32-byte step
                                // in it; the descriptor's start address is in 16-byte units
                                const int kg = h * L::AK + ks * 16;
                                tc_mma_ts(tmem + t * NTOK, a_tm + ks * 8,
                                          bdesc + static_cast<uint64_t>(
                                                      ((kg >> 6) * L::X_BOX + (kg & 63) * 2) >> 4),
                                          idesc, (g | h | ks) != 0);
                            }
                            tc_commit(empty_a(t, a));
                            // the stage's x and, before it, its weights are read
                            if (h == SUB - 1) tc_commit(empty_smem(s));
                        }
                        __syncwarp();
                        issued = true;
                        if (++a == SA) a = 0, pa ^= 1u;
                    }
                    if (++s == S) s = 0;
                }
                if (!ok) break;
                if (elect_one()) tc_commit(d_full(t));  // the chunk's accumulators of tile t are final
                __syncwarp();
            }
            if (issued) {
                // every MMA issued has completed before tensor memory is freed
                if (elect_one()) {
                    tc_commit(drain(t));
                    settle(drain(t), 0);
                }
                __syncwarp();
            }
        }
    } else if (row_warp) {
        // ------------------------------------------------------------ dequant + epilogue
        const int t = row_tile;
        // the row's four 16-byte chunks in a stage (64-byte swizzle: chunk j of row rr
        // sits at j ^ ((rr >> 1) & 3))
        const bool in_range = r < RB;
        const int bx = r >= RB / 2 ? 1 : 0;
        const int rr = in_range ? r - bx * (RB / 2) : 0;
        const uint32_t w_first = sbase + L::X_BYTES + bx * L::W_HALF + rr * (kGroupK / 2);
        uint32_t c_off[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) c_off[i] = 16u * (static_cast<uint32_t>(i) ^ ((rr >> 1) & 3));
        const int KG = p.K / p.g;      // scales per row
        const int upg = p.g >> 6;      // 64-k halves of a stage per scale group
        // running stage and A slots (addresses that advance by a constant and wrap)
        uint32_t w_at = w_first, full_at = full_tma(0), ph = 0;
        uint32_t empty_at = empty_a(t, 0), a_at = lane_base + L::A_COL + t * (L::AK / 2), pa = 1;
        uint32_t nchunk = 0;
        for (int chunk = chunk0; ok && chunk < p.num_chunks; chunk += chunk_step, ++nchunk) {
            const int tt = chunk / p.row_chunks;
            const int n = (chunk - tt * p.row_chunks) * RB + r;
            const bool valid = in_range && n < p.N;
            // the row's scales of a stage's two 64-k halves (equal when g is a
            // multiple of 128), loaded a stage ahead; rows past the range
            // compute on other rows' data, their sums are never stored
            const uint16_t* srow = p.scales + static_cast<int64_t>(valid ? n : 0) * KG;
            int kk = rot;
            uint16_t n_lo, n_hi;
            auto load_scales = [&]() {
                if (upg == 2) {
                    n_lo = __ldg(srow + kk);
                } else {
                    const int lo = 2 * kk / upg, hi = (2 * kk + 1) / upg;
                    n_lo = __ldg(srow + lo);
                    // K ends in the middle of the stage: its second half is zero
                    n_hi = hi < KG ? __ldg(srow + hi) : static_cast<uint16_t>(0);
                }
                if (++kk == k_end) kk = k_first;
            };
            // the scales of the next stage to dequantise, and the load for the one after:
            // with one A stage per stage, while its last stores are under way
            uint32_t s2_lo = 0, s2_hi = 0;
            ScaleFma f_lo{}, f_hi{};
            bool wide = false;
            auto next_scales = [&]() {
                s2_lo = s2_hi = splat_bf16(n_lo);
                f_lo = f_hi = scale_fma(s2_lo);
                bool w_scale = scale_is_wide(n_lo);
                if (upg != 2) {
                    s2_hi = splat_bf16(n_hi);
                    f_hi = scale_fma(s2_hi);
                    w_scale = w_scale || scale_is_wide(n_hi);
                }
                load_scales();
                wide = __any_sync(0xffffffffu, w_scale);
            };
            load_scales();
            if (SUB == 1) next_scales();
            for (int left = k_count; left > 0; --left) {
                if (SUB > 1) next_scales();
                // the stage has landed, and the previous MMAs of its first A slot are done
                if (!wait_warp2(full_at, ph, empty_at, pa, abort_flag, p.status, p.wait_ns)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
#pragma unroll
                for (int h = 0; h < SUB; ++h) {
                    uint4 c[L::CHUNKS];
#pragma unroll
                    for (int i = 0; i < L::CHUNKS; ++i) c[i] = lds128(w_at + c_off[L::CHUNKS * h + i]);
                    const bool st_ok = dbg_check(
                        (a_at & 0xFFFFu) + L::AK / 2 <= (tmem & 0xFFFFu) + L::TMEM_COLS, p.status);
                    // wd = RNE_bf16((q - 8) * s), as bf16 pairs of the row's lane
                    constexpr int CS = L::CHUNKS == 1 ? 1 : 2;  // chunks per store
#pragma unroll
                    for (int i = 0; i < L::CHUNKS; i += CS) {
                        const bool hi_half = L::CHUNKS * h + i >= 2;
                        const ScaleFma& f = hi_half ? f_hi : f_lo;
                        const uint32_t s2 = hi_half ? s2_hi : s2_lo;
                        uint32_t v[16 * CS];
                        if (!wide) {
#pragma unroll
                            for (int q = 0; q < CS; ++q) {
                                dequant_word_fma(c[i + q].x, f, v + 16 * q);
                                dequant_word_fma(c[i + q].y, f, v + 16 * q + 4);
                                dequant_word_fma(c[i + q].z, f, v + 16 * q + 8);
                                dequant_word_fma(c[i + q].w, f, v + 16 * q + 12);
                            }
                        } else {
#pragma unroll
                            for (int q = 0; q < CS; ++q) {
                                dequant_word(c[i + q].x, s2, v + 16 * q);
                                dequant_word(c[i + q].y, s2, v + 16 * q + 4);
                                dequant_word(c[i + q].z, s2, v + 16 * q + 8);
                                dequant_word(c[i + q].w, s2, v + 16 * q + 12);
                            }
                        }
                        if (h > 0 && i == 0) {
                            // the slot's previous MMAs are done
                            if (!wait_warp(empty_at, pa, abort_flag, p.status, p.wait_ns)) {
                                ok = false;
                                break;
                            }
                            tc_fence_after();
                        }
                        if (st_ok) {
                            if constexpr (CS == 1)
                                tmem_st_32x32b_x16(a_at, v);
                            else
                                tmem_st_32x32b_x32(a_at + i * 16, v);
                        }
                    }
                    if (!ok) break;
                    if (SUB == 1 && h == SUB - 1) next_scales();
                    tmem_st_wait();
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(empty_at - 8u * SA);  // full_a of the slot
                    empty_at += 8u;
                    a_at += L::A_COLS;
                    if (empty_at == empty_a(t, SA)) {
                        empty_at -= 8u * SA;
                        a_at -= L::A_COLS * SA;
                        pa ^= 1u;
                    }
                }
                if (!ok) break;
                w_at += L::STAGE;
                full_at += 8u;
                if (full_at == full_tma(S)) {
                    full_at = full_tma(0);
                    w_at = w_first;
                    ph ^= 1u;
                }
            }
            if (!ok) break;
            // the row's NTOK accumulators
            if (!wait_warp(d_full(t), nchunk & 1u, abort_flag, p.status, p.wait_ns)) {
                ok = false;
                break;
            }
            tc_fence_after();
            if constexpr (!SPLIT) {
                const float bias = (FUSED && p.epi.bias != nullptr && valid)
                                       ? bf16_to_f32(p.epi.bias[n]) : 0.0f;
                const int mt = tt * NTOK, m_end = mt + NTOK < p.M ? mt + NTOK : p.M;
#pragma unroll 1
                for (int m0 = 0; mt + m0 < m_end; m0 += L::EC) {
                    uint32_t d[32];
                    float v[L::EC];
                    tmem_ld_32x32b_x32(lane_base + t * NTOK + m0, d);
                    tmem_ld_wait(d);
#pragma unroll
                    for (int j = 0; j < L::EC; ++j) v[j] = __uint_as_float(d[j]);
                    store_tokens<FUSED, L::EC>(p.epi, p.out, v, mt + m0, m_end, n, valid, bias, lane);
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(d_empty(t));  // the next chunk's MMAs may overwrite D
            }
        }
    }

    if constexpr (SPLIT) {
        // ------------------------------------------------------------ sum over the cluster
        // One chunk per cluster; each CTA holds its K slice's sums.  Per slice
        // of EC tokens every CTA writes its partial sums to shared memory
        // (over the consumed stages), and CTA `rank` adds up and finishes its
        // EC / split tokens, always in the order of the ranks.  The stages
        // are free once every role of the CTA is done with them.
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
        const int tt = chunk0 / p.row_chunks;
        const int n = (chunk0 - tt * p.row_chunks) * RB + r;
        const bool valid = row_warp && r < RB && n < p.N;
        const float bias =
            (FUSED && p.epi.bias != nullptr && valid) ? bf16_to_f32(p.epi.bias[n]) : 0.0f;
        const int mt = tt * NTOK, m_end = mt + NTOK < p.M ? mt + NTOK : p.M;
        uint32_t part = sbase;
#pragma unroll 1
        for (int m0 = 0; mt + m0 < m_end; m0 += L::EC) {
            // a CTA that gave up leaves the sums unwritten: its output is incomplete
            if (row_warp && ok) {
                uint32_t d[32];
                tmem_ld_32x32b_x32(lane_base + row_tile * NTOK + m0, d);
                tmem_ld_wait(d);
#pragma unroll
                for (int j = 0; j < L::EC; ++j)
                    asm volatile("st.shared.u32 [%0], %1;" ::"r"(part + 4u * (j * L::ROWS_MAX + r)),
                                 "r"(d[j]) : "memory");
            }
            __syncwarp();
            cluster_sync();
            if (row_warp && ok) {
                if (p.split == 2)
                    reduce_slice<2, FUSED>(p, part, L::ROWS_MAX, rank, r, bias, mt + m0, m_end, n,
                                           valid, lane);
                else if (p.split == 4)
                    reduce_slice<4, FUSED>(p, part, L::ROWS_MAX, rank, r, bias, mt + m0, m_end, n,
                                           valid, lane);
                else
                    reduce_slice<8, FUSED>(p, part, L::ROWS_MAX, rank, r, bias, mt + m0, m_end, n,
                                           valid, lane);
            }
            __syncwarp();
            part = part == sbase ? sbase + L::PART : sbase;
        }
        cluster_sync();  // no CTA leaves while another reads its sums
    }

    __syncwarp();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 1) tmem_dealloc(tmem, L::TMEM_COLS);
}

template <int NTOK, int TILES, bool SPLIT>
cudaError_t launch_tc_variant(const CUtensorMap* tx, const CUtensorMap* tw, const GemvParams& p,
                              int grid, cudaStream_t stream) {
    using L = TLayout<NTOK, TILES>;
    const bool fused =
        p.epi.bias != nullptr || p.epi.residual != nullptr || p.epi.act != kActNone;
    auto kern = fused ? w4a16_gemv_tc_kernel<NTOK, TILES, true, SPLIT>
                      : w4a16_gemv_tc_kernel<NTOK, TILES, false, SPLIT>;
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(L::THREADS);
    cfg.dynamicSmemBytes = L::SMEM_BYTES;
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // grid_wait
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if constexpr (SPLIT) {
        attr[1].id = cudaLaunchAttributeClusterDimension;
        attr[1].val.clusterDim.x = static_cast<unsigned>(p.split);
        attr[1].val.clusterDim.y = 1;
        attr[1].val.clusterDim.z = 1;
        cfg.numAttrs = 2;
    }
    e = cudaLaunchKernelEx(&cfg, kern, *tx, *tw, p);
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template <int NTOK, int TILES>
cudaError_t launch_tc_split(const CUtensorMap* tx, const CUtensorMap* tw, const GemvParams& p,
                            int sm_count, cudaStream_t stream) {
    if (p.split > 1)
        return launch_tc_variant<NTOK, TILES, true>(tx, tw, p, p.num_chunks * p.split, stream);
    const int grid = p.num_chunks < sm_count ? p.num_chunks : sm_count;
    return launch_tc_variant<NTOK, TILES, false>(tx, tw, p, grid, stream);
}

// Clusters of `split` CTAs that can be resident at once; cached per device.
int cluster_slots(int split, int sm_count) {
    if (split == 1) return sm_count;
    constexpr int kMaxDev = 64;
    static std::atomic<int> cache[kMaxDev][4] = {};
    const int slot = split == 2 ? 0 : split == 4 ? 1 : 2;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDev) return 0;
    int n = cache[dev][slot].load(std::memory_order_relaxed);
    if (n != 0) return n;
    using L = TLayout<128, 3>;
    auto kern = w4a16_gemv_tc_kernel<128, 3, false, true>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, L::SMEM_BYTES) ==
        cudaSuccess) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = static_cast<unsigned>(split);
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(static_cast<unsigned>(sm_count / split * split));
        cfg.blockDim = dim3(L::THREADS);
        cfg.dynamicSmemBytes = L::SMEM_BYTES;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) n = 0;
    }
    cudaGetLastError();  // a failed query leaves no sticky error for the next launch
    if (n <= 0) n = -1;  // none: no split
    cache[dev][slot].store(n, std::memory_order_relaxed);
    return n;
}

}  // namespace

GemvTcPlan gemv_tc_plan(int64_t M, int64_t N, int64_t K, int64_t g, const Epilogue& epi,
                        int sm_count) {
    // us per 128-k stage of a CTA that holds 1, 2 or 3 tiles of 128 rows, by token
    // columns 32, 64, 96, 112, 128 (K = 12288, N = 19000 without a split, 36864 and 49152,
    // less 4 us: 41.4 / 45.4 / 46.6 / 48.0 / 52.3, 52.6 / 58.3 / 64 / 67.3 / 72.5 and
    // 63.2 / 78.2 / 83.6 / 103.3 / 104.2 us in all)
    static constexpr double kStageUs[3][5] = {{0.39, 0.43, 0.44, 0.46, 0.50},
                                              {0.51, 0.57, 0.63, 0.66, 0.71},
                                              {0.62, 0.77, 0.83, 1.03, 1.05}};
    GemvTcPlan best{};
    // equal tiles of at most 128 tokens
    const int64_t tok_tiles = (M + 127) / 128;
    const int64_t per = (M + tok_tiles - 1) / tok_tiles;
    best.tokens = per <= 32 ? 32 : per <= 64 ? 64 : per <= 96 ? 96 : per <= 112 ? 112 : 128;
    const int tok = best.tokens == 32 ? 0 : best.tokens == 64 ? 1 : (best.tokens - 64) / 16;
    // What the choice between the splits leaves out and the one between the kernels needs:
    // up to 16 tokens, against the warp-level kernel, the same stages one launch after
    // another (39.1, 50.4 and 60.4 us in all; fused 53 and 64), a further wave (98304
    // rows, K = 128 6.5 us, half of them 4.0) and the fused output stage of a chunk (K = 256,
    // 49152 rows, M = 1: 5.4 us plain, 6.0 with a residual, 7.3 GELU, 8.8 SwiGLU); beyond, that
    // of odd widths (M = 128, K = 64: 4.1 plain, 20 with GELU) and a long walk's second
    // scales a stage where g is not 128 (M = 129, N = 36864, g = 64 150 us, 143 on the GEMM)
    const bool fused = epilogue_fused(epi);
    const double kFewTokensStageUs[3] = {0.38, fused ? 0.535 : 0.495, fused ? 0.64 : 0.60};
    const double output =
        M <= 16 ? (!fused ? 0.0 : epi.act == kActSwiGLU ? 2.8 : epi.act == kActGELU ? 1.9 : 0.6)
                : (epilogue_odd(epi) && epi.act == kActGELU ? 15.0 : 0.0);
    double chosen = 0.0;
    const int64_t KS = (K + kGroupK - 1) / kGroupK;
    for (int split = 1; split <= 8; split *= 2) {
        const int64_t slots = cluster_slots(split, sm_count);
        if (split > 1 && (slots < tok_tiles || split > KS)) continue;
        // rows: spread evenly over as few waves of the slots as hold them (a
        // cluster takes one chunk); even, SwiGLU pairs rows 2j, 2j + 1
        int64_t waves = (N * tok_tiles + slots * 128 * kTilesMax - 1) / (slots * 128 * kTilesMax);
        if (split > 1 && waves > 1) continue;
        int64_t rb = 0;
        for (;; ++waves) {
            const int64_t chunks = slots * waves / tok_tiles;
            if (chunks < 1) continue;
            rb = ((N + chunks - 1) / chunks + 1) / 2 * 2;
            if (rb <= 128 * kTilesMax || split > 1) break;
        }
        if (rb > 128 * kTilesMax) continue;
        const int nt = static_cast<int>((rb + 127) / 128);
        const double stages = static_cast<double>(waves) * static_cast<double>((KS + split - 1) / split);
        const double cost = 4.0 + stages * kStageUs[nt - 1][tok] +
                            (split > 1 ? 1.5 + 0.04 * best.tokens : 0.0);
        if (chosen == 0.0 || cost < chosen) {
            chosen = cost;
            best.cost_us = cost + static_cast<double>(waves) * output / split +
                           (g != 128 && best.tokens <= 96 && stages >= 64.0 ? 0.1 * stages : 0.0);
            if (M <= 16)
                best.cost_us += (static_cast<double>(waves) - 1.0) * 1.3 + 0.35 * (nt - 3) +
                                stages * (kFewTokensStageUs[nt - 1] - kStageUs[nt - 1][tok]);
            best.split = split;
            best.rows_per_cta = static_cast<int>(rb);
            best.row_chunks = static_cast<int>((N + rb - 1) / rb);
            best.num_chunks = static_cast<int>(best.row_chunks * tok_tiles);
        }
    }
    return best;
}

cudaError_t gemv_tc_launch(const CUtensorMap* tx, const CUtensorMap* tw, const GemvParams& p,
                           int tokens, int sm_count, cudaStream_t stream) {
    const bool two = p.nt <= 2;
    switch (tokens) {
        case 32:
            return two ? launch_tc_split<32, 2>(tx, tw, p, sm_count, stream)
                       : launch_tc_split<32, 3>(tx, tw, p, sm_count, stream);
        case 64:
            return two ? launch_tc_split<64, 2>(tx, tw, p, sm_count, stream)
                       : launch_tc_split<64, 3>(tx, tw, p, sm_count, stream);
        case 96:
            return two ? launch_tc_split<96, 2>(tx, tw, p, sm_count, stream)
                       : launch_tc_split<96, 3>(tx, tw, p, sm_count, stream);
        case 112:
            return two ? launch_tc_split<112, 2>(tx, tw, p, sm_count, stream)
                       : launch_tc_split<112, 3>(tx, tw, p, sm_count, stream);
        default:
            return two ? launch_tc_split<128, 2>(tx, tw, p, sm_count, stream)
                       : launch_tc_split<128, 3>(tx, tw, p, sm_count, stream);
    }
}

}  // namespace w4a16
