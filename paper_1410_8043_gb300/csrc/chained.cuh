// Launch of a kernel that may start while the kernel before it in the stream
// still runs (programmatic dependent launch); the kernel waits for that one with
// await_previous_kernel() before its first access to global memory, and reads
// as read-only data (__ldg, const __restrict__) only what no kernel writes: the
// layout of the loaded entries.
#pragma once

#include <cuda_runtime.h>

namespace esspt {

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), int blocks, int threads, cudaStream_t st, bool chained,
                           const Args&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = chained ? 1 : 0;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

}  // namespace esspt
