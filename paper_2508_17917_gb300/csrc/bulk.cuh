// bulk.cuh -- bulk copies into shared memory on an mbarrier, with bounded waits.
#pragma once
#include <cuda_runtime.h>

namespace dg {

// Waits (about 100 ns each, 1.7 s in all) for copies still in flight after a
// wait on them gave up: they land in the block's shared memory, so the block
// stays until they have, whatever limit the caller set for its waits.
constexpr unsigned kDrainWaits = 1u << 24;

// Bulk copies (the tensor memory accelerator's 1-D form) into shared memory,
// completing on an mbarrier: the warp's own tile and the operator table.
__device__ __forceinline__ void mbar_init1(unsigned bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// 16-byte aligned addresses, a multiple of 16 bytes
__device__ __forceinline__ void bulk_g2s(unsigned dst, const void *src, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// bounded wait for phase `parity` of an mbarrier; false if it gave up
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity, unsigned limit)
{
    for (unsigned it = 0;; ++it) {
        unsigned ok;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(ok)
            : "r"(bar), "r"(parity)
            : "memory");
        if (ok) return true;
        if (it >= limit) return false;
        __nanosleep(100);
    }
}

// orders this thread's ordinary reads and writes against bulk copies
__device__ __forceinline__ void fence_async()
{
    asm volatile("fence.proxy.async;" ::: "memory");
}

}  // namespace dg
