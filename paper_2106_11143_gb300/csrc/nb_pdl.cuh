// nb_pdl.cuh -- programmatic dependent launch: a kernel's blocks are placed while
// the previous kernel of the stream drains, and wait in hardware for its end.
//
// At n of a few thousand a step is two kernels of 4 to 9 us, and the launch of
// each after the other's end a part of it.  A kernel launched by launch_pdl
// calls pdl_wait() before it touches any memory: past it the previous kernel has
// ended and its writes are visible, as after an ordinary launch.  Its blocks are
// placed as the previous kernel's blocks end.  us per step with ordinary launches
// and so: 10.95 and 10.45 at n = 1024 (fp64), 14.6 and 14.3 at 3001 (split).
// Letting the blocks in earlier (griddepcontrol.launch_dependents) was slower,
// 11.2 to 12.6 at n = 1024: they take places that leave the running kernel's or
// their own blocks unevenly spread.
#pragma once

#include <cuda_runtime.h>

namespace nb {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace nb
