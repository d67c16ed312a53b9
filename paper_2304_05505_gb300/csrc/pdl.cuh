// Programmatic dependent launch: a kernel launched with launch_pdl may start
// while the kernel before it on the stream is still running, so that its
// launch and its prologue overlap that kernel's last blocks.  It calls
// pdl_begin() before it touches global memory: that waits until everything
// before it on the stream is complete and visible (also when it was launched
// the plain way), and lets the kernel after it start the same way.  A build is
// 10 to 16 kernels one after the other, of a few microseconds each on small
// cells.
#pragma once

#include <cuda_runtime.h>

__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}
