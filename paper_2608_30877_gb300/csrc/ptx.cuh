// Inline-PTX building blocks for sm_103a: mbarriers, TMA tensor loads and the
// tcgen05 (5th-generation tensor core / tensor memory) instructions.
#pragma once

#include <cuda.h>
#include <cstdint>

namespace w4a16 {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// One lane of a converged warp (the same one every time).
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(p));
    return p != 0;
}

// Programmatic launch: a kernel launched with cudaLaunchAttributeProgrammaticStream-
// Serialization may start when every CTA of the one before it in the stream has called
// grid_launch_dependents (or ended), and touches global memory only after grid_wait,
// which returns once that one has completed and its writes are visible.  Its launch, barriers
// and tensor memory are then under way as the SMs of the one before it fall idle: 0.5 us
// of a streaming kernel (12288 x 12288, M = 8 23.3 -> 22.8 us; 2048 x 2048, M = 1 7.1 ->
// 6.5; 36864 x 12288 with g = 64 after other work 66.0 -> 64.2).  A kernel calls
// grid_launch_dependents before its own grid_wait: the next one waits for all of it.
__device__ __forceinline__ void grid_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ void grid_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---------------------------------------------------------------- mbarrier

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// A thread whose phase has not completed may be suspended for up to
// kSuspendHintNs (it resumes as soon as the phase completes), so waiting
// warps do not take issue slots from the working ones.
constexpr uint32_t kSuspendHintNs = 0x20000;

// Whether the phase has completed, without suspending the thread (kCluster: see below).
template <bool kCluster = false>
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (kCluster) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
    }
    return ok != 0;
}

// kCluster: acquire at cluster scope, for barriers that threads or tensor-core
// commits of the other CTA of a pair arrive on.
template <bool kCluster = false>
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (kCluster) {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspendHintNs)
            : "memory");
    } else {
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity), "r"(kSuspendHintNs)
            : "memory");
    }
    return ok != 0;
}

// Records `code` in the device status word unless an earlier error is
// already there: the first error of a run is the one reported.
__device__ __forceinline__ void record_status(int* status, int code) {
    atomicCAS(status, 0, code);
}

// ---------------------------------------------------------------- debug checks
// Built with -DW4A16_DEBUG, the kernels check the indices they compute before
// each TMA copy, tensor-memory access and global store: a failed check records
// W4A16_ERR_INDEX (6) in the status word and the access is skipped (no trap,
// the context stays usable; a skipped copy makes the waits on it run out).
// Without the flag every check is the constant true and compiles away.
#ifdef W4A16_DEBUG
constexpr bool kDebugChecks = true;
#else
constexpr bool kDebugChecks = false;
#endif

__device__ __forceinline__ bool dbg_check(bool ok, int* status) {
    if constexpr (kDebugChecks) {
        if (!ok) atomicCAS(status, 0, 6 /* W4A16_ERR_INDEX */);
        return ok;
    }
    return true;
}

// A tiled TMA load into [dst, dst + box_bytes): the innermost coordinate times
// the element size a multiple of 16 bytes (else the copy is an illegal
// instruction), the destination aligned to `align` and inside the shared-memory
// region [lo, hi) that holds the CTA's staging buffers.
__device__ __forceinline__ bool tma_box_ok(uint32_t dst, uint32_t box_bytes, uint32_t align,
                                           uint32_t lo, uint32_t hi, int32_t c0,
                                           uint32_t elem_bytes) {
    return c0 >= 0 && ((static_cast<uint32_t>(c0) * elem_bytes) & 15u) == 0 &&
           (dst & (align - 1u)) == 0 && dst >= lo && dst + box_bytes <= hi;
}

// Every wait in the kernels is bounded: after limit_ns of global time (the
// launch's wait limit, kWaitLimitNs unless a test lowers it) or kWaitIterCap
// polls the waiter gives up, raises the CTA's abort flag and records a
// timeout in the device status word.  With the default limit the clock and
// the flag are checked every few polls, with a lowered one (a test of the
// abort path) after every failed poll.  A poll may suspend its thread until the
// phase completes, so a lowered limit does not by itself make a wait run out:
// each producer waits for its first copy with polls that do not suspend
// (short_limit_ok), and a debug build polls that way in every wait, so that there
// any role can be the first to give up.  The drains before a kernel exits (its
// own copies and MMAs in flight) always use kWaitLimitNs.
constexpr uint64_t kWaitLimitNs = 4000000000ull;  // 4 s
constexpr uint32_t kWaitIterCap = 1u << 26;

// The producers' check for a lowered limit.  Always true with the default one, and in a
// debug build.
__device__ __forceinline__ bool short_limit_ok(uint32_t bar, uint32_t parity,
                                               volatile int* abort_flag, int* status,
                                               uint64_t limit_ns) {
    if (kDebugChecks || limit_ns >= kWaitLimitNs) return true;
    const uint64_t t0 = global_timer_ns();
    while (!mbar_test_wait(bar, parity)) {
        if (global_timer_ns() - t0 > limit_ns) {
            *abort_flag = 1;
            record_status(status, 5 /* W4A16_ERR_TIMEOUT */);
            return false;
        }
    }
    return true;
}

// A poll of the waits below.
template <bool kCluster>
__device__ __forceinline__ bool mbar_poll(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
    if constexpr (kDebugChecks) {
        if (limit_ns < kWaitLimitNs) return mbar_test_wait<kCluster>(bar, parity);
    }
    return mbar_try_wait<kCluster>(bar, parity);
}

// Wait by one thread.  Returns false if the wait ran out or the CTA aborted.
// With SLEEP_NS the thread sleeps between polls, for waits that have stages in
// hand (a TMA producer with a full ring): its polls then take no issue slots
// from the warps doing the work.
template <bool kCluster = false, uint32_t SLEEP_NS = 0>
__device__ __forceinline__ bool wait_one(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                         int* status, uint64_t limit_ns) {
    if (mbar_poll<kCluster>(bar, parity, limit_ns)) return true;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1;; ++it) {
        if (SLEEP_NS > 0) __nanosleep(SLEEP_NS);
        if (mbar_poll<kCluster>(bar, parity, limit_ns)) return true;
        if ((it & 31u) == 0u || limit_ns < kWaitLimitNs) {
            if (*abort_flag) return false;
            if (it > kWaitIterCap || global_timer_ns() - t0 > limit_ns) {
                *abort_flag = 1;
                record_status(status, 5 /* W4A16_ERR_TIMEOUT */);
                return false;
            }
        }
    }
}

// Wait by a whole warp; every lane polls the barrier and the exit is
// warp-uniform (so that .sync.aligned instructions after it stay converged).
// SLEEP_NS as above: for long, latency-tolerant waits (an epilogue waiting for
// a whole tile's MMAs).
template <bool kCluster = false, uint32_t SLEEP_NS = 0>
__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, uint64_t limit_ns) {
    // (the timer is slow to read: only once a poll has failed)
    if (__all_sync(0xffffffffu, mbar_poll<kCluster>(bar, parity, limit_ns))) return true;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t t0 = global_timer_ns();
    for (uint32_t it = 1;; ++it) {
        if (SLEEP_NS > 0) __nanosleep(SLEEP_NS);
        const bool done = mbar_poll<kCluster>(bar, parity, limit_ns);
        if (__all_sync(0xffffffffu, done)) return true;
        if ((it & (SLEEP_NS > 0 ? 7u : 31u)) == 0u || limit_ns < kWaitLimitNs) {
            int give_up = 0;
            if (lane == 0) {
                if (*abort_flag) {
                    give_up = 1;
                } else if (it > kWaitIterCap || global_timer_ns() - t0 > limit_ns) {
                    *abort_flag = 1;
                    record_status(status, 5 /* W4A16_ERR_TIMEOUT */);
                    give_up = 1;
                }
            }
            if (__shfl_sync(0xffffffffu, give_up, 0)) return false;
        }
    }
}

// Wait by a whole warp for two barriers, their polls under way together.
__device__ __forceinline__ bool wait_warp2(uint32_t bar0, uint32_t parity0, uint32_t bar1,
                                           uint32_t parity1, volatile int* abort_flag, int* status,
                                           uint64_t limit_ns) {
    const bool d0 = mbar_poll<false>(bar0, parity0, limit_ns),
               d1 = mbar_poll<false>(bar1, parity1, limit_ns);
    if (__all_sync(0xffffffffu, d0 && d1)) return true;
    return wait_warp(bar0, parity0, abort_flag, status, limit_ns) &&
           wait_warp(bar1, parity1, abort_flag, status, limit_ns);
}

// Bounded wait used by the drains before exit: gives up silently after
// kWaitLimitNs (the copy or MMA it waits for was issued by this CTA and
// completes on its own).
template <bool kCluster = false>
__device__ __forceinline__ void settle(uint32_t bar, uint32_t parity) {
    const uint64_t t0 = global_timer_ns();
    while (!mbar_try_wait<kCluster>(bar, parity)) {
        if (global_timer_ns() - t0 > kWaitLimitNs) break;
    }
}

// ---------------------------------------------------------------- TMA

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// 2-D tiled load of one box into shared memory; completion is signalled on
// `bar` as transaction bytes.  c0 is the innermost coordinate.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                            int32_t c0, int32_t c1) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}

// All threads of all CTAs of the cluster.
__device__ __forceinline__ void cluster_sync() {
    asm volatile(
        "barrier.cluster.arrive.release.aligned;\n\t"
        "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

// Address in the shared::cluster window of the variable at shared::cta
// address `addr` in the cluster's CTA `rank`.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// One arrival without release semantics on an mbarrier of the cluster.  For
// hand-offs of tensor-memory data only: a tcgen05.wait::st / ::ld has already
// completed the stores or loads the arrival signals, and
// tcgen05.fence::before_thread_sync orders them before it.  A release at
// cluster scope here costs a cluster-wide memory fence per arrival (the CTA
// pair GEMM ran at 916 instead of 1463 TFLOP/s with it).
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_addr) {
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr)
                 : "memory");
}

__device__ __forceinline__ void st_shared_cluster_u32(uint32_t cluster_addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr), "r"(v) : "memory");
}

__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map,
                                                 uint32_t bar, int32_t c0, int32_t c1,
                                                 uint64_t policy) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
        " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
        : "memory");
}

__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// ---------------------------------------------------------------- tcgen05

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     dst_smem),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Arrive once on `bar` when every tcgen05 operation issued so far by this
// thread has completed.
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]^T, kind::f16 (bf16 inputs, fp32 accumulator).
__device__ __forceinline__ void tc_mma_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                          uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// ---- CTA pairs (cta_group::2): one MMA of M = 256 rows spans the tensor
// cores of two CTAs of a cluster; each CTA holds its 128 rows of A and D in
// its own tensor memory and N/2 rows of B in its own shared memory, at the
// same addresses.  Allocation, release and deallocation are done by one warp
// of each CTA; the MMAs and their commits by one thread of the even CTA.

__device__ __forceinline__ void tmem_alloc_pair(uint32_t dst_smem, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     dst_smem),
                 "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void tmem_relinquish_pair() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}

// Arrive once on the mbarrier at shared::cluster address `bar` (either CTA of
// the pair) when every pair MMA issued so far by this thread has completed.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
        : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]^T over the CTA pair, kind::f16.
__device__ __forceinline__ void tc_mma_ts_pair(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                               uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

// Instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, M rows x N columns.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int m, int n) {
    return (1u << 4)                              // D format: f32
           | (1u << 7)                            // A format: bf16
           | (1u << 10)                           // B format: bf16
           | (static_cast<uint32_t>(n >> 3) << 17)  // N / 8
           | (static_cast<uint32_t>(m >> 4) << 24); // M / 16
}

// Shared-memory matrix descriptor for a K-major operand stored with the
// 128-byte swizzle: rows of 128 bytes, 8-row (1024-byte) swizzle atoms
// stacked at a stride of 1024 bytes.  The tile base must be 1024-byte
// aligned; moving along K inside the atom adds to the start address.
__device__ __forceinline__ uint64_t sdesc_kmajor_sw128(uint32_t saddr) {
    uint64_t d = 0;
    d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);  // start address / 16
    d |= static_cast<uint64_t>(0) << 16;                  // leading byte offset (unused here)
    d |= static_cast<uint64_t>(1024 >> 4) << 32;          // stride byte offset / 16
    d |= static_cast<uint64_t>(1) << 46;                  // descriptor version (fixed 0b001)
    d |= static_cast<uint64_t>(2) << 61;                  // swizzle mode: 128 B
    return d;
}

// 32 lanes x 32 columns of 32 bits: thread i of the warp owns lane
// (warp's sub-partition base + i); registers map to consecutive columns.
__device__ __forceinline__ void tmem_st_32x32b_x32(uint32_t taddr, const uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(
            taddr),
        "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]),
        "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]),
        "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]),
        "r"(v[29]), "r"(v[30]), "r"(v[31])
        : "memory");
}

__device__ __forceinline__ void tmem_st_wait() {
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
        "[%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]),
          "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]),
          "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_ld_32x32b_x16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr)
        : "memory");
}

__device__ __forceinline__ void tmem_ld_wait_x16(uint32_t (&v)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                   "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                   "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15])
                 :
                 : "memory");
}

// Waits for this thread's tcgen05.ld; the registers are listed as operands so
// that no use of them can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&v)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                   "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                   "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]),
                   "+r"(v[17]), "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]),
                   "+r"(v[22]), "+r"(v[23]), "+r"(v[24]), "+r"(v[25]), "+r"(v[26]),
                   "+r"(v[27]), "+r"(v[28]), "+r"(v[29]), "+r"(v[30]), "+r"(v[31])
                 :
                 : "memory");
}

}  // namespace w4a16
