// Launches whose start-up overlaps the end of the kernel before them in the stream
// (programmatic dependent launch).  A kernel launched with pdl_launch may begin while its
// predecessor still runs, so every block calls pdl_wait before it touches global memory:
// the wait returns once the predecessor has completed and its writes are visible (and, as
// that one waited too, everything before it).  pdl_trigger lets the successor begin
// launching; after a plain launch both are no-ops.  The chains of a composition step are a
// few microseconds per kernel, of which launch latency and block start-up are a part (DRE
// n = 81: 47.6 -> 44.3 us a step).  Used for T3 and the FP64 products of few blocks only: in the
// chains of the tensor kernels the early blocks cost more than they saved (DRE n = 1024
// split, 64 steps: 11.8 -> 13.5 ms; DLE n = 256 FP64, 100 steps: 6.3 -> 6.8 ms).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace dme {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
cudaError_t pdl_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace dme
