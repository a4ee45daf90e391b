// L2 eviction-priority hints for the stream that meets itself in L2 within
// one iteration: the agent sweep writes q' (or u, consensus_from_q), which the
// consensus gather reads right after, while the amplitudes and the stack
// reads of the sweep are used once per iteration.  The stack the gather reads
// is stored evict-last, the single-use streams are marked evict-first, so
// more of it is still in L2 when the gather runs.  The evict-last hint is only
// given where the stack can mostly stay in L2 (no larger than twice the L2),
// else it is stored evict-normal.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace pmace {

__device__ __forceinline__ uint64_t l2_policy_evict_last() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_normal() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void st_l2_hint(float2* ptr, float2 v, uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(ptr), "f"(v.x), "f"(v.y), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ float2 ld_l2_hint(const float2* ptr, uint64_t pol) {
    float2 v;
    asm volatile("ld.global.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;" : "=f"(v.x), "=f"(v.y) : "l"(ptr), "l"(pol));
    return v;
}
__device__ __forceinline__ uint4 ld_nc_l2_hint(const uint4* ptr, uint64_t pol) {
    uint4 v;
    asm volatile("ld.global.nc.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr), "l"(pol));
    return v;
}

}  // namespace pmace
