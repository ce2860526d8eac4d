// Programmatic dependent launch, device and host side.
#pragma once

#include <cuda_runtime.h>

namespace fn {

// Programmatic dependent launch: a kernel launched with programmatic
// stream serialization may be scheduled while its predecessor drains; it
// touches nothing the predecessor writes before this wait (a no-op for a
// plain launch), and then lets its own successor be scheduled.
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}

// Launch with programmatic stream serialization (see pdl_begin): the
// kernel may be scheduled while the previous kernel on the stream drains.
template <class... KArgs, class... Args>
inline void pl_launch_pdl(bool pdl, void (*k)(KArgs...), unsigned grid, unsigned block,
                          size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, args...);
}
template <class... KArgs, class... Args>
inline void pl_launch(void (*k)(KArgs...), unsigned grid, unsigned block, size_t smem,
                      cudaStream_t st, Args... args) {
  pl_launch_pdl(true, k, grid, block, smem, st, args...);
}

}  // namespace fn
