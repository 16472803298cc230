// Shared-memory mbarriers and bulk copies (cp.async.bulk, completed through an
// mbarrier's transaction count), used by the tensor-core kernels; programmatic
// dependent launch.  Every wait is bounded by kSpinLimit polls; the
// caller turns a timeout into an error flag.
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

namespace h2 {

constexpr uint32_t kSpinLimit = 1u << 25;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* b, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
// Non-blocking test of a phase (acquire semantics when it reports completion):
// a caller issues it ahead of the work it overlaps and reads the result later.
__device__ __forceinline__ bool mbar_test(uint64_t* b, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{ .reg .pred p; mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(ok)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity) {
    for (uint32_t i = 0; i < kSpinLimit; ++i)
        if (mbar_try(b, parity)) return true;
    return false;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// L2 policies for bulk copies: data streamed once (evict first) and data read again
// by later copies (evict last).
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
// Programmatic dependent launch: a kernel launched with launch_chained may start
// while its predecessor on the stream still runs.  Every thread of such a kernel
// calls chain_release(), after which the successor's CTAs may be scheduled (they take
// what this grid leaves free), and chain_wait(), after which everything that earlier
// kernels wrote is visible; only work on data that no kernel writes stands before it.
// Every kernel waits, so completion passes down the chain.  Such a kernel is alive while
// its predecessors write, so what they write (and the caller's blocks, which may be the
// output of the product before) is not read-only to it: __ldg and __restrict__, which
// promise that and let loads pass the wait, are for matrix data and index lists alone.
__device__ __forceinline__ void chain_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Byte offset of element (row r, column c) of a core-matrix tile whose rows hold
// kp values of es bytes (kp·es a multiple of 16): 8-row groups outermost, then
// 16-byte column chunks, then the 8 rows of 16 bytes of one core matrix.
__host__ __device__ __forceinline__ int64_t cm_off(int r, int c, int kp, int es) {
    const int per = 16 / es;
    return ((int64_t)(r >> 3) * (kp / per) + (c / per)) * 128 + (r & 7) * 16 + (c % per) * es;
}

}  // namespace h2
