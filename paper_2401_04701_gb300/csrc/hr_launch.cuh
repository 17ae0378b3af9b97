// hr_launch.cuh - launches that overlap the end of the kernel before them.
//
// A check is a chain of 3 to 8 dependent launches of 2 to 500 us, and five of them find
// nothing to do when the pre-pass leaves a check to the per-wave checker.  With
// programmatic stream serialization a kernel's CTAs are placed, and fill their tables,
// while the kernel before it ends, instead of a launch latency after it.  Checks with no
// chosen variant (us, before and after): 262,144 records in one wave on 2^22 words 63 and
// 43 (40 without the binned kernels and with ordinary launches), 0.29M records in 32
// waves on 2^20 words 108 and 94, 4.7M on 2^22 words 156 and 143, 75.2M on 2^26 words
// 1,313 and 1,291.  No kernel lets its successor start early (launch_dependents): the
// successor's CTAs would hold their SMs against other streams' kernels meanwhile.
#pragma once

#include <cuda_runtime.h>

namespace {

// In every kernel that hr_launch launches, by every thread, before anything that a kernel
// before it writes is read and before anything is written: wait until the kernel before
// it in the stream has finished and its writes are visible.  As every thread does so, a
// kernel that has finished has its predecessors finished too.
__device__ __forceinline__ void hr_grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t hr_launch(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, A... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace
