// mbarriers and asynchronous (TMA) copies into shared memory: copies complete on an mbarrier, and
// every wait on one has a limit.
#pragma once
#include <cuda.h>

#include "cbct_internal.cuh"

namespace cbct {

__device__ __forceinline__ void mbar_init(unsigned long long *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long *bar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// one try: suspends the thread for up to about a millisecond while the phase is incomplete
__device__ __forceinline__ bool mbar_try_wait(unsigned long long *bar, unsigned parity)
{
    unsigned ok;
    asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(ok)
                 : "r"(smem_u32(bar)), "r"(parity), "r"(1000000u)
                 : "memory");
    return ok != 0;
}
// Every wait ends: after WAIT_CYCLES (about two seconds), or once another warp of the
// block has given up, it returns false, and the block then ends with NaN results and bit 1
// of the iteration's status word instead of a hang. The verdict is the warp's: lanes may leave
// the loop for different reasons, and a warp that went on with some of them would wait at its
// next full-mask shuffle for the others. Called by whole warps.
constexpr long long WAIT_CYCLES = 4000000000ll;
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity, volatile int *give_up)
{
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) {
        const long long t0 = clock64();
        while (!(ok = mbar_try_wait(bar, parity)) && !*give_up)
            if (clock64() - t0 > WAIT_CYCLES) *give_up = 1;
    }
    return __all_sync(0xffffffffu, ok);
}
// generic accesses of this thread to shared memory before, bulk copies into it after
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }

// cuTensorMapEncodeTiled of the driver the runtime has loaded (no link to libcuda); nullptr if absent.
using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_tiled();

} // namespace cbct
