// Dependent launches (leakage calibration, tensor-core transform).
#pragma once

#include <cuda_runtime.h>

namespace polaris {

// One launch with programmatic stream serialisation: the kernel may be scheduled while its
// predecessor ends, and waits for it (griddepcontrol.wait) before it touches what that one, or
// the caller's earlier work, wrote.
template <typename... P, typename... Q>
static cudaError_t launch_dependent(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st, Q... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace polaris
