// Chained launches, for the passes of a solve and the layers of the network.
#pragma once
#include <cuda_runtime.h>

namespace s3ttv {

// The kernels are launched as programmatic dependents of one another: chained() is
// the first statement of each, lets the next kernel's CTAs come in as soon as this
// one's have all started, and waits for the kernel before to be done (with its
// writes), so launch latency and CTA set-up overlap the tail of the kernel before.
// No kernel touches memory ahead of it.
__device__ __forceinline__ void chained() {
  asm volatile("griddepcontrol.launch_dependents;\n griddepcontrol.wait;\n" ::: "memory");
}
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                  A... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace s3ttv
