// vlb_chain.cuh -- launches whose set-up overlaps the end of the kernel before them.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace vlb {

// Launches in a chain (programmatic dependent launch): a kernel that calls chain_begin() before
// its first access to memory, and is launched by launch_chained, is set up while its
// predecessor in the stream drains; chain_begin waits until the predecessor has ended and its
// writes are visible. After a copy, or a kernel without chain_begin, it starts as usual.
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;\ngriddepcontrol.launch_dependents;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A &&...args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

}  // namespace vlb
