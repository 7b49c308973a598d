// mbarrier helpers shared by the warp-specialised kernels (tensor-core prefill kernels, streaming kernels):
// init / arrive / expect-tx / try-wait, and the BOUNDED wait every role uses.  A wait never spins without limit:
// after `budget` SM clock ticks it raises the CTA's abort flag and the sticky status EXMOE_ERR_TIMEOUT and returns
// false; every other waiter of the CTA sees the flag within 16 polls and returns false too, so that all roles
// leave their loops and the kernel ends with the context intact (exercised by exmoe_debug_wait_timeout).
#pragma once
#include <stdint.h>
#include <cuda_runtime.h>
#include "../../include/exmoe.h"

namespace exmoe {

constexpr long long kWaitBudget = 2000000000ll;   // clock64 ticks (~1 s) before a wait gives up

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// bounded wait; returns false when the CTA is aborting (and raises the abort on expiry)
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          long long budget = kWaitBudget) {
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    unsigned polls = 0;
    while (!mbar_try(bar, parity)) {
        if ((++polls & 15u) == 0) {                    // the bookkeeping of the bound is amortised over 16 polls
            if (*abort_flag) return false;
            if (clock64() - t0 > budget) {
                *abort_flag = 1;
                atomicExch(status, EXMOE_ERR_TIMEOUT);
                return false;
            }
        }
    }
    return true;
}

// The same by a whole warp, for barriers given by their shared-memory address: control flow that the compiler knows to be
// uniform (no divergence bookkeeping around the poll, and the code around it keeps its uniform registers), no address
// conversion per call.  The wait ends when EVERY lane has seen the phase complete: what the barrier guards is ordered only
// behind a lane's own successful wait.
__device__ __forceinline__ void mbar_arrive_at(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_at(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// A look that never blocks (try_wait suspends the thread until the phase completes or a time limit of the hardware's).
__device__ __forceinline__ bool mbar_look_at(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status) {
    if (__all_sync(0xffffffffu, mbar_try_at(bar, parity))) return true;
    const long long t0 = clock64();
    for (unsigned polls = 1;; ++polls) {
        if (__all_sync(0xffffffffu, mbar_try_at(bar, parity))) return true;
        if ((polls & 15u) == 0) {
            const bool late = clock64() - t0 > kWaitBudget;
            if (late) {
                *abort_flag = 1;
                atomicExch(status, EXMOE_ERR_TIMEOUT);
            }
            if (__any_sync(0xffffffffu, late || *abort_flag)) return false;
        }
    }
}
// one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
    uint32_t p;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
    return p != 0;
}
template <typename T>
__device__ __forceinline__ T warp_uniform(T v) { return __shfl_sync(0xffffffffu, v, 0); }

}  // namespace exmoe
