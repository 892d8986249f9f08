#pragma once

#include <cuda_runtime.h>

namespace lmk {
namespace {

// Programmatic dependent launch: kernels that follow one another in
// small steps are launched with cudaLaunchAttributeProgrammaticStreamSerialization, so that
// each can be scheduled while its predecessor in the stream drains.  Every
// such kernel first waits for its predecessors to complete (griddepcontrol.
// wait: their memory operations are then visible), so the order of all
// memory accesses is that of plain stream order; only the launch latency
// overlaps.  It then allows its own dependent to be scheduled.  In a launch
// without the attribute both instructions return at once.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t dyn, cudaStream_t s, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = dyn;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace
}  // namespace lmk
