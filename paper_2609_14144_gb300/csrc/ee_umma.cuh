// tcgen05 (fifth-generation tensor core) and mbarrier helpers shared by the
// projections and the attention of the multi-position layer pass.
#ifndef EE_UMMA_CUH_
#define EE_UMMA_CUH_

#include <stdint.h>

#include "ee_internal.h"

namespace ee {

constexpr long long kUWaitCycles = 4000000000ll;   // bound of a wait: about 2 s

__device__ __forceinline__ uint32_t u_saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void u_mb_init(uint64_t* b, int n) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(u_saddr(b)), "r"(n) : "memory");
}
__device__ __forceinline__ bool u_mb_test(uint64_t* b, int parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(u_saddr(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Wait for the phase of parity `parity`; false after the bound, or (when
// `err` is given) once the error word carries kErrStall.
__device__ __forceinline__ bool u_mb_wait(uint64_t* b, int parity, const volatile int* err) {
    if (u_mb_test(b, parity)) return true;
    const long long t0 = clock64();
    for (unsigned it = 1;; ++it) {
        if (u_mb_test(b, parity)) return true;
        if ((it & 255) == 0) {
            if (clock64() - t0 > kUWaitCycles) return false;
            if (err && (*err & kErrStall)) return false;
        }
    }
}

__device__ __forceinline__ void u_mb_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(u_saddr(b)) : "memory");
}

// ---------------------------------------------------------------- tcgen05
// Shared-memory operand descriptor, no swizzle: start address and the byte
// offsets between core matrices (8 x 16 bytes, contiguous) along K (lbo) and
// along the rows M or N (sbo).  K-major: a core matrix is 8 rows of 8 K
// elements; N-major: 8 K indices of 8 rows.
__device__ __forceinline__ uint64_t u_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr >> 4) & 0x3fffu);
    d |= (uint64_t)((lbo >> 4) & 0x3fffu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3fffu) << 32;
    d |= (uint64_t)1 << 46;  // descriptor version of sm_100 and later
    return d;                // base offset 0, layout type 0 (no swizzle)
}
// Instruction descriptor of kind::f16: fp32 accumulator, bf16 A and B, A
// K-major, B K-major or (b_mn) with its N index contiguous, M = 128, N = n (a
// multiple of 16, 16 <= n <= 256).
__device__ __forceinline__ uint32_t u_idesc(int n, bool b_mn = false) {
    return (1u << 4) | (1u << 7) | (1u << 10) | (b_mn ? 1u << 16 : 0u) | ((uint32_t)(n >> 3) << 17) | (8u << 24);
}

__device__ __forceinline__ void u_mma(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{ .reg .pred p; setp.ne.u32 p, %4, 0; tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p; }" ::"r"(
            tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void u_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(u_saddr(bar))
                 : "memory");
}
__device__ __forceinline__ void u_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void u_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

// 16 consecutive fp32 columns of this thread's tensor-memory lane; the values
// are there after u_wait_ld().
__device__ __forceinline__ void u_ld16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void u_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

}  // namespace ee

#endif  // EE_UMMA_CUH_
