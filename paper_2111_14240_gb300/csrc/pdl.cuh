// Programmatic dependent launch between the two kernels of an iteration: the
// next kernel's CTAs may start while the last ones of the kernel before it
// still run, load what does not depend on it (probe tables, window corners,
// gather lists) and wait.  Every kernel launched this way calls pdl_wait
// before it touches the stacks or images, and lets its own successor start
// only after that, so at most two kernels of a stream overlap.  In a launch
// without the attribute both calls do nothing.
//
// Only for iterations whose consensus leaves the GPU mostly empty
// (small_consensus): 169 windows of 32 x 32 14.3 -> 12.2 us an iteration, 81
// of 64 x 64 14.0 -> 12.2.  On larger ones the SMs go from one kernel to the
// next without a drain and so keep the sweep's split of their 256 KB, which
// leaves the gather little L1: 900 windows of 128 x 128 120 -> 131 us, 64009
// 6.72 -> 7.86 ms.
#pragma once

#include <cuda_runtime.h>

namespace pmace {

// Wait until the kernels before this one have finished and their writes are
// visible, then let the next one start.
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A load of what an earlier kernel of the stream wrote (the consensus image),
// for kernels that may be launched with the attribute: they are resident while
// that kernel still writes, which read-only loads (__ldg, ld.global.nc) do not
// allow, and the compiler may move those over pdl_wait.
__device__ __forceinline__ float2 ld_live(const float2* p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

inline cudaLaunchAttribute pdl_attribute() {
    cudaLaunchAttribute a = {};
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    return a;
}

// Launch fn<<<grid, block, smem, s>>>(args...), with the attribute if `on`.
template <typename... P, typename... A>
cudaError_t pdl_launch(bool on, void (*fn)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                       A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    cfg.attrs = attr;
    cfg.numAttrs = on ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, fn, args...);
}

}  // namespace pmace
