// bsp_ptx.h -- mbarriers, bulk copies and tcgen05 helpers shared by the
// tensor-core kernels.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bsp {
namespace {

constexpr long long WAIT_CYCLES = 1ll << 33;   // ~4 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// Has the phase of parity `parity` completed?  test_wait never blocks;
// try_wait may block for a short time set by the hardware.
__device__ __forceinline__ bool mbar_test(uint32_t addr, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    return done != 0;
}
__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    return done != 0;
}
// Wait for the phase of parity `parity` to complete; false once `limit` cycles
// have passed (~4 s by default).  After one plain try_wait, waits poll with a
// suspend-time hint: the waiting thread sleeps in the barrier until the phase
// completes (or ~2 us pass) instead of re-reading shared memory in a tight
// loop, which took shared-memory bandwidth from the copies, the pair products
// and the MMAs.  Under a short limit (< 2^20 cycles) the wait polls with
// test_wait instead, so that the limit holds to within a few hundred cycles.
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, long long limit = WAIT_CYCLES) {
    const uint32_t addr = smem_u32(b);
    const bool sleep = limit >= (1ll << 20);
    if (sleep ? mbar_try(addr, parity) : mbar_test(addr, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        uint32_t done;
        if (sleep)
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
                " selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(done)
                : "r"(addr), "r"(parity), "r"(2000u)
                : "memory");
        else
            done = mbar_test(addr, parity);
        if (done) return true;
        if (clock64() - t0 > limit) return false;
    }
}

// The whole warp waits for its lanes' barriers, each lane its own address and
// parity: one pass through the (busy) shared-memory pipe tests them all.  Tested
// one after another, three barriers that had long completed took 250 cycles each.
// The first SPIN tests poll, the rest sleep (a sleeping wait wakes some 300 cycles
// late: starting with one cost the contraction 20 %, even when the phase was complete).
// The same result in every lane: false once `limit` cycles have passed or *abort is set
// (abort may be null: a last wait that nothing else ends).
template <int SPIN>
__device__ __forceinline__ bool warp_wait(uint32_t addr, uint32_t parity, long long limit, const volatile int* abort) {
    bool done = mbar_test(addr, parity);
    if (__all_sync(0xffffffffu, done)) {
        __syncwarp();   // what one lane's barrier released is visible to all
        return true;
    }
    // (a phase that has completed cannot be followed by another before this warp moves on)
#pragma unroll 1
    for (int i = 1; i < SPIN; ++i) {
        done = mbar_test(addr, parity);
        if (__all_sync(0xffffffffu, done)) {
            __syncwarp();
            return true;
        }
    }
    const bool sleep = limit >= (1ll << 20);
    const long long t0 = clock64();
    // every lane tests again, also those whose phase is complete: with the sleeping test under a
    // branch (or a predicate) of `done`, a warp with one open barrier came apart here and its other lanes
    // left with true (tests/gpu_probes/warp_wait.cu); testing again costs nothing measurable
    while (true) {
        if (sleep) {
            uint32_t d;
            asm volatile(
                "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
                " selp.u32 %0, 1, 0, p;\n}\n"
                : "=r"(d)
                : "r"(addr), "r"(parity), "r"(2000u)
                : "memory");
            done = d != 0;
        } else {
            done = mbar_test(addr, parity);
        }
        if (__all_sync(0xffffffffu, done)) {
            __syncwarp();
            return true;
        }
        if (__any_sync(0xffffffffu, (abort != nullptr && *abort != 0) || clock64() - t0 > limit)) return false;
    }
}

// 1-D bulk copy global -> shared (16-byte aligned, size a multiple of 16), completing on bar.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ bool elect_one() {
    uint32_t e;
    asm volatile("{\n .reg .b32 r;\n .reg .pred p;\n elect.sync r|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
    return e != 0;
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     smem_u32(bar))
                 : "memory");
}

}  // namespace
}  // namespace bsp
