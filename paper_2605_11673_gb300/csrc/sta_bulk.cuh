// Bulk copies (the tensor-memory-access unit's untiled cp.async.bulk) with mbarrier completion.
#pragma once

#include <stdint.h>

namespace sta {
namespace {

// Polls of a wait on a barrier at most: a wait that runs out is reported, never endless.
constexpr unsigned BAR_SPINS = 1u << 22;

__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void bar_init(uint64_t *bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
// after bar_init, before the CTA's barrier that publishes the initialised barriers
__device__ __forceinline__ void bar_init_fence() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t *bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
// arrival that also expects `bytes` of bulk copies before the phase completes
__device__ __forceinline__ void bar_arrive_expect(uint64_t *bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)),
                 "r"(bytes)
                 : "memory");
}
// whether the phase of the given parity has completed, within BAR_SPINS polls
__device__ __forceinline__ bool bar_wait(uint64_t *bar, unsigned parity) {
    const uint32_t a = smem_addr(bar);
    for (unsigned i = 0; i < BAR_SPINS; ++i) {
        unsigned ok;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(ok)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (ok) return true;
    }
    return false;
}
// 8 or 16 bytes by the calling thread; part of its open commit group
template <int N> __device__ __forceinline__ void cp_async(void *dst, const void *src) {
    static_assert(N == 8 || N == 16, "cp.async sizes used here");
    if constexpr (N == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
// bytes: a multiple of 16; both addresses 16-byte aligned
__device__ __forceinline__ void bulk_load(void *dst, const void *src, unsigned bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

}  // namespace
}  // namespace sta
