// Launches that overlap the kernel before them in the stream (programmatic
// dependent launch): the later grid may start once every block of the earlier
// one has called launch_dependents (or left), and sees the earlier one's memory
// after wait_for_previous_grid, which returns when that grid is complete.  Both
// are no operations in a grid launched the plain way.
#pragma once
#include <cuda_runtime.h>

namespace oct {

__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... Params, class... Args>
cudaError_t launch_overlapped_smem(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, bool overlap,
                                   cudaStream_t st, const Args &...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1u : 0u;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

template <class... Params, class... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, bool overlap, cudaStream_t st,
                              const Args &...args) {
    return launch_overlapped_smem(kernel, grid, block, 0, overlap, st, args...);
}

}  // namespace oct
