// The hardware's block scheduler as a work queue: the kernel is launched with
// one block per item, and a resident block that is done asks for the next
// block that has not started (clusterlaunchcontrol.try_cancel), takes over its
// index and keeps its own constants, buffers and prefetches.
//
// Against a fixed stride over the items (one block per slot): the blocks of an
// SM do not run at one speed (the scheduler prefers the older warps), so with
// equal shares the first ones leave and the SM ends with too few warps.
#pragma once

#include "common.cuh"
#include "tc.cuh"

namespace vl {

// All of it is one thread's work, which tells the others (init before a block
// barrier). A request is outstanding until take() returns its item, -1 when none
// is left: after that no further request may be made.
struct WorkQueue {
    static constexpr uint32_t kPolls = 1u << 20;  // bound of a wait (far beyond any real answer)
    ulonglong2 answer;
    uint64_t bar;

    __device__ __forceinline__ void init() { tc::mbar_init(&bar, 1); }
    __device__ __forceinline__ void request() {
        tc::fence_async_smem();  // the last answer was read before this one is written
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(tc::smem_addr(&bar)), "r"(16u)
                     : "memory");
        asm volatile(
            "clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];\n" ::"r"(
                tc::smem_addr(&answer)),
            "r"(tc::smem_addr(&bar))
            : "memory");
    }
    // the item of the i-th request (from 0)
    __device__ __forceinline__ int take(int i, unsigned long long* counters) {
        if (!tc::mbar_wait(&bar, (uint32_t)i & 1u, kPolls)) {
            atomicAdd(&counters[CNT_COPY_TIMEOUT], 1ull);
            return -1;
        }
        const ulonglong2 r = answer;
        uint32_t ok, x = 0;
        asm volatile(
            "{\n .reg .b128 h;\n .reg .pred p;\n mov.b128 h, {%1, %2};\n"
            " clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, h;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "l"(r.x), "l"(r.y));
        if (!ok) return -1;
        asm volatile(
            "{\n .reg .b128 h;\n mov.b128 h, {%1, %2};\n"
            " clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, h;\n}\n"
            : "=r"(x)
            : "l"(r.x), "l"(r.y));
        return (int)x;
    }
};

}  // namespace vl
