// Pieces shared by the tcgen05 kernels: bounded mbarrier waits, no-swizzle
// K-major shared-memory descriptors of 64-byte rows.
#pragma once

#include "qmc_internal.cuh"

namespace qmc {
namespace {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

constexpr unsigned kPSpin = 1u << 22;          // mbarrier polls before a wait gives up
constexpr uint32_t kPLBO = 128;                // K-adjacent core matrices
constexpr uint32_t kPSBO = 4 * 128;            // 8-row groups (64-byte rows)

__device__ __forceinline__ uint64_t psmem_desc(uint32_t saddr) {
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFFu);
    d |= (uint64_t)((kPLBO >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((kPSBO >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bounded wait for the completion of phase `parity`; false once the abort
// flag is set or after kPSpin polls (then the flag and kErrTimeout are set).
__device__ __forceinline__ bool pwait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned* err) {
    for (unsigned it = 0; it < kPSpin; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if ((it & 255) == 255 && *abort_flag) return false;
    }
    *abort_flag = 1;
    atomicOr(err, kErrTimeout);
    return false;
}
// The same wait without the abort flag (the final drains).
__device__ __forceinline__ void pdrain(uint32_t bar, uint32_t parity) {
    for (unsigned it = 0; it < kPSpin; ++it) {
        uint32_t ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return;
    }
}

}  // namespace
}  // namespace qmc
