// Device helpers shared by the walk engine's translation units: warp
// collectives, TMA bulk copies, mbarriers, bounded waits.
#pragma once

#include "fw_internal.cuh"

namespace fw {
namespace {

constexpr unsigned FULL = 0xffffffffu;
constexpr int INT_BIG = 0x7fffffff;

__device__ __forceinline__ unsigned long long global_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // bounded waits: 2 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned long long* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(unsigned long long* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(unsigned long long* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)  // let the thread sleep up to 20 us for the phase
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of an mbarrier; false after kWaitLimitNs (a copy
// that never lands means a bug: the caller then stops cleanly).
__device__ __forceinline__ bool mbar_wait_bounded(unsigned long long* bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_timer_ns();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_timer_ns() - t0 > kWaitLimitNs) return false;
    }
}

// The same for a whole warp: every lane learns whether all of them saw the phase.
__device__ __forceinline__ bool mbar_wait_warp(unsigned long long* bar, uint32_t parity) {
    if (__all_sync(FULL, mbar_try_wait(bar, parity))) return true;
    return __all_sync(FULL, mbar_wait_bounded(bar, parity));
}

// 1-D bulk copy global -> shared, completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_1d(void* dst, const void* src, uint32_t bytes, unsigned long long* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

// Start fetching `bytes` (a multiple of 16) from a 16-byte boundary into L2.
__device__ __forceinline__ void prefetch_l2(const void* src, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}

// Read-only loads under a predicate, as single instructions: the compiler
// neither turns them into branches, one waiting for the other, nor moves them
// down past later volatile ones to where their value is used.
__device__ __forceinline__ int ldg_if(const int32_t* p, bool ok, int other) {
    int v;
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\tmov.b32 %0, %3;\n\t@q ld.global.nc.b32 %0, [%1];\n\t}"
        : "=&r"(v)
        : "l"(p), "r"((int)ok), "r"(other));
    return v;
}
__device__ __forceinline__ float4 ldg_if(const float4* p, bool ok) {
    float4 v;
    asm volatile(
        "{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\t"
        "mov.b32 %3, 0;\n\t@q ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "=&f"(v.x), "=&f"(v.y), "=&f"(v.z), "=&f"(v.w)
        : "l"(p), "r"((int)ok));
    return v;
}

// Orders this thread's ordinary shared-memory stores before later bulk copies
// into the same bytes.
__device__ __forceinline__ void fence_proxy_async_cta() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ float unit_open(uint32_t w) {
    // strictly inside (0, 1): 23 random bits centred in their cell, so the
    // largest value is 1 - 2^-24 (exact in FP32) and -log(u) > 0 always
    return ((float)(w >> 9) + 0.5f) * (1.0f / 8388608.0f);
}

// First index i >= pos with B[i] >= x, or pd.  Warp-collective, uniform result.
__device__ __noinline__ int lower_bound_from(const int32_t* __restrict__ B, int pd, int pos, int x, int lane) {
    {
        const int idx = pos + lane;
        const int v = idx < pd ? __ldg(B + idx) : INT_BIG;
        const unsigned m = __ballot_sync(FULL, v < x);
        if (m != FULL) return pos + __popc(m);
    }
    int lo = pos + 32, hi = pd;  // the answer lies in [lo, hi]
    while (hi - lo > 32) {
        const int s = (hi - lo + 31) >> 5;
        const long long idx = (long long)lo + (long long)s * (lane + 1) - 1;
        const int v = idx < hi ? __ldg(B + idx) : INT_BIG;
        const int k = __popc(__ballot_sync(FULL, v < x));
        const int nlo = lo + s * k;
        const long long nhi = (long long)lo + (long long)s * (k + 1) - 1;
        lo = nlo;
        hi = nhi < hi ? (int)nhi : hi;
    }
    const int v = lo + lane < hi ? __ldg(B + lo + lane) : INT_BIG;
    return lo + __popc(__ballot_sync(FULL, v < x));
}

}  // namespace
}  // namespace fw
