// Launch helper of the single-grid step kernels.
#pragma once

#include <cuda_runtime.h>

namespace vss {

// ---------------------------------------------------------------------------
// Programmatic dependent launch.  The single-grid step kernels are launched
// with programmatic stream serialization allowed: each block first lets the next launch on the stream
// start (the next grid is launched once every block of this one has started
// or exited, so its blocks only take SM slots this grid no longer needs), then
// waits until the previous grid has completed and its memory is visible, and
// only then touches global memory.  The next step's launch latency is thereby
// hidden behind this step's tail.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... KArgs, typename... Args>
static cudaError_t launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block,
                              size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace vss
