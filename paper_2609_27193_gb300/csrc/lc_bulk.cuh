// lc_bulk.cuh -- the bulk-copy engine pieces shared by the kernels that
// stream global memory through shared-memory rings (lc_copy.cu: the pack,
// commit and restore; lc_measure.cu: the Eq. 1 scan): mbarrier waits that
// give up after a bound, cp.async.bulk loads and stores, the fault word, and
// 16-byte windows at any even offset in staged bytes.
#pragma once

#include "lc_internal.cuh"

namespace lc {
namespace {

// A wait gives up after this long (a 32 KB load completes in microseconds);
// the iteration cap bounds it even if the timer were not advancing.
constexpr uint64_t kWaitNs = 1000000000ull;
constexpr uint64_t kDrainNs = 100000000ull;
constexpr uint32_t kWaitIters = 1u << 28;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// Waits for the phase with the given parity to complete, for at most
// `limit_ns` (and kWaitIters polls).  Returns false if it gave up.  A poll
// suspends the thread for a while in hardware; the timer is read on every
// kPollsPerTime-th one only.
constexpr uint32_t kPollsPerTime = 16;
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    uint64_t t0 = 0;
    for (uint32_t it = 1; it < kWaitIters; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if (it % kPollsPerTime) continue;
        const uint64_t t = global_ns();
        if (t0 == 0) t0 = t;
        else if (t - t0 > limit_ns) return false;
    }
    return false;
}

// A consumer warp's wait: its lanes poll together and take the outcome
// together.  True: the phase is complete and every lane's reads come after
// it.  (With lane 0 polling for the warp, unrelated code in the loop decided
// between two speeds of the whole kernel: the 8B measure took 4.28 or 4.79 ms,
// the fused step over 1.2 G parameters 5.22 or 6.66 ms.  This way it has been
// the faster one with every variant of that code.)
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    uint64_t t0 = 0;
    for (uint32_t it = 1; it < kWaitIters; ++it) {
        if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        if (it % kPollsPerTime) continue;
        const uint64_t t = __shfl_sync(0xffffffffu, global_ns(), 0);
        if (t0 == 0) t0 = t;
        else if (t - t0 > kWaitNs) return false;
    }
    return false;
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// One arrival for the warp, once all its lanes are done.  What the warp still
// does with registers alone comes after it (after_handback): the buffer's next
// load then starts before that work, not behind it.
__device__ __forceinline__ void mbar_arrive_warp(uint32_t bar, int lane) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
    __syncwarp();
}

// Keeps the use of x and y behind the hand-back that precedes it: arithmetic on
// registers may otherwise be scheduled ahead of it.
__device__ __forceinline__ void after_handback(float& x, float& y) { asm volatile("" : "+f"(x), "+f"(y)::"memory"); }

// global -> shared, completing `bytes` of the barrier's transaction count.
__device__ __forceinline__ void bulk_g2s(uint32_t dst_smem, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// shared -> global, in the thread's current bulk group.
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src_smem, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src_smem), "r"(bytes)
                 : "memory");
}

// Bytes [SH, SH + 16) of the 32 bytes of a and b (SH even).
template <int SH>
__device__ __forceinline__ uint4 window16(const uint4& a, const uint4& b) {
    const uint32_t x[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    constexpr int q = SH / 4;
    if constexpr (SH % 4 == 0) {
        return make_uint4(x[q], x[q + 1], x[q + 2], x[q + 3]);
    } else {
        return make_uint4(__funnelshift_r(x[q], x[q + 1], 16), __funnelshift_r(x[q + 1], x[q + 2], 16),
                          __funnelshift_r(x[q + 2], x[q + 3], 16), __funnelshift_r(x[q + 3], x[q + 4], 16));
    }
}

// Records that a bounded wait ran out: the host reads the word (host-mapped).
__device__ __forceinline__ void raise_fault(uint32_t* fault) {
    if (fault) {
        *reinterpret_cast<volatile uint32_t*>(fault) = 1u;
        __threadfence_system();
    }
}

}  // namespace
}  // namespace lc
