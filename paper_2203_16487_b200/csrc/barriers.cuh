// Shared-memory addresses, mbarriers and the cluster barrier: what the kernels of every translation unit share.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace sd {

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok;
}
// Bounded wait: gives up after ~2e8 clocks, raises the CTA-wide abort flag and the global error word.  The warp that gives up then holds the
// CTA, and with it the shared memory that its copies in flight and its peers still write to, for about a millisecond longer: many times what
// a copy that was issued before the flag was up can take.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err_word,
                                          int code) {
    if (mbar_try_wait(bar, parity)) return true;      // fast path: no other shared-memory access
    if (*abort_flag) return false;
    const long long t0 = clock64();
    while (true) {
        if (mbar_try_wait(bar, parity)) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > 200000000LL) {
            *abort_flag = 1;
            atomicExch(err_word, code);
            while (clock64() - t0 < 202000000LL) {}
            return false;
        }
    }
}
// The same for a converged warp: every lane gets the same answer, as an elected instruction behind it needs all of them there.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err_word, int code) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, err_word, code));
}
// 16 consecutive bytes to the shared memory of CTA `rank` of this cluster, counted on its mbarrier.
__device__ __forceinline__ void st_peer16(uint32_t local_addr, uint32_t local_bar, uint32_t rank, uint4 v) {
    uint32_t ra, rb;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(local_addr), "r"(rank));
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(rb) : "r"(local_bar), "r"(rank));
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];"
                 ::"r"(ra), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(rb) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_cluster_sync() { cluster_arrive(); cluster_wait(); }

}  // namespace sd
