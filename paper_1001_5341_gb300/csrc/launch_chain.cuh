// launch_chain.cuh -- kernels of a chain of launches whose prologues overlap the
// end of the launch before them (programmatic dependent launch).
#pragma once

#include <cuda_runtime.h>

namespace fdtd {

// the next launch's blocks may start once every block of this one has
__device__ __forceinline__ void release_next_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// the launch before this one is complete and its writes are visible; nothing that
// it reads or writes is touched before this
__device__ __forceinline__ void after_last_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// a launch that may begin before the one in front of it ends where `early`; the
// kernel calls after_last_launch
template <typename... P, typename... A>
inline void launch_after(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);   // errors: the caller's cudaGetLastError
}

}  // namespace fdtd
