// Programmatic dependent launch of the step kernels.
#pragma once
#include <cuda_runtime.h>

namespace lbm {

// Programmatic dependent launch: a launch's blocks may be scheduled while
// the one before drains and wait here until it is complete and its writes
// are visible, which hides part of the launch latency (101^2 FP32 tiles of 6
// steps: 1.01 -> 0.91 us per step).
__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename Kern, typename... Args>
cudaError_t launch_pdl(Kern kern, unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                       Args... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kern, args...);
}

}  // namespace lbm
