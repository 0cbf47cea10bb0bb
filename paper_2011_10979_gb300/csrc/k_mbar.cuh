// k_mbar.cuh -- mbarriers in shared memory that TMA copies complete on: set-up, the copies, and waits bounded
// in time.
//
// A wait that runs out sets the pair's timeout flag (the solve then reports OF_ETIMEOUT) and the launch ends
// without the missing data.  The bound is in nanoseconds of %globaltimer, as the persistent engine's: an attempt
// of mbarrier.try_wait may suspend the thread for a time of the hardware's choice, so a number of
// attempts is no known duration.  Once the flag is set, later waits of the solve give up after a millisecond: the
// launches that follow one that gave up end quickly too.
#pragma once
#include <cuda.h>

namespace tvl1 {

__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *b, unsigned n) {
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(n) : "memory");
}
// Makes the initialised mbarriers visible to copies and to the cluster.
__device__ __forceinline__ void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect(unsigned long long *b, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_load(void *dst, const CUtensorMap *map, int x, int y, unsigned long long *b) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
                 ::"r"(smem_u32(dst)), "l"(map), "r"(x), "r"(y), "r"(0), "r"(smem_u32(b))
                 : "memory");
}

// One attempt at the phase of parity ph.  CLUSTER: what arrives is sent by other CTAs of the cluster.
template <bool CLUSTER> __device__ __forceinline__ bool mbar_try(unsigned long long *b, unsigned ph) {
    unsigned ok;
    if (CLUSTER)
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
            : "=r"(ok)
            : "r"(smem_u32(b)), "r"(ph)
            : "memory");
    else
        asm volatile("{ .reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
                     : "=r"(ok)
                     : "r"(smem_u32(b)), "r"(ph)
                     : "memory");
    return ok;
}
// The rest of a wait that its first attempts did not end: at most ns nanoseconds, or one millisecond when *flag (may
// be NULL) is set; false when the time ran out.  Out of line, beside the registers and the code of the kernels.
template <bool CLUSTER> __device__ __noinline__ bool mbar_wait_timed(unsigned long long *b, unsigned ph, long long ns, const int *flag) {
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
        if (mbar_try<CLUSTER>(b, ph)) return true;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        const long long dt = (long long)(t - t0);
        if (dt > ns || (dt > 1000000 && flag && *(const volatile int *)flag)) return false;
    }
}
// Waits for the phase of parity ph (reading the timer takes longer than a wait usually does).
template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(unsigned long long *b, unsigned ph, long long ns, const int *flag) {
#pragma unroll 1
    for (int k = 0; k < 4096; ++k)
        if (mbar_try<CLUSTER>(b, ph)) return true;
    return mbar_wait_timed<CLUSTER>(b, ph, ns, flag);
}

}  // namespace tvl1
