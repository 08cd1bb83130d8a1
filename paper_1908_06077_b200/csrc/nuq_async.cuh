// mbarriers and the bulk asynchronous copy.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace nuq {

// ---------------------------------------------------------------------------
// Bulk asynchronous copy (TMA, untiled form) and its mbarrier.  CTA-local barriers only.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory operands are addresses in shared memory, or pointers.
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) { mbar_init(smem_u32(bar), count); }

// Orders this thread's earlier accesses to shared memory before its later bulk copies.
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Announces `bytes` to the barrier and starts the copy global -> shared.  Both addresses
// 16-byte aligned, `bytes` a positive multiple of 16.  The fenced form orders earlier generic writes to dst first.
__device__ __forceinline__ void bulk_load_unfenced(uint32_t dst_smem, const void* src_gmem, uint32_t bytes, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst_smem),
                 "l"(src_gmem), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void* src_gmem, uint32_t bytes, uint32_t bar) {
    fence_async_proxy();
    bulk_load_unfenced(dst_smem, src_gmem, bytes, bar);
}
__device__ __forceinline__ void bulk_load(void* dst_smem, const void* src_gmem, uint32_t bytes, uint64_t* bar) {
    bulk_load(smem_u32(dst_smem), src_gmem, bytes, smem_u32(bar));
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Waits until the phase with the given parity has completed.  Bounded: false after ~tens of ms.
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity) {
    // the hardware parks the thread for up to the hinted time (ns), so a wait costs a handful of
    // instructions; the number of tries bounds the wait (a fraction of a second at most)
    for (uint32_t polls = 0; polls < (1u << 17); ++polls) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(addr), "r"(parity), "r"(2000u)
            : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) { return mbar_wait(smem_u32(bar), parity); }

}  // namespace nuq
