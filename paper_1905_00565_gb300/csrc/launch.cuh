// Launches that follow each other on one stream (programmatic dependent
// launch): a kernel's CTAs are set up while the one before it drains, and every
// kernel first waits for that one to finish.  Small jobs are chains of kernels
// of a few microseconds, where the gaps between them count.
//
// What the kernel before writes is read with plain loads, never with __ldg: the
// read-only path asks for data that does not change while the kernel lives, and a
// chained kernel lives before its wait.  (Two kernels back is safe: a CTA is set up
// only once every CTA of the kernel before has passed its own wait.)
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "ccm_internal.h"

namespace ccm {

// First statement of every kernel launched with launch_chained: waits until the
// kernel before it on the stream has finished and its writes are visible, then
// lets the next one be set up.
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... Params, typename... Args>
cudaError_t launch_chained(void (*kernel)(Params...), dim3 grid, int threads, size_t smem,
                           LaunchStream s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s.s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = s.chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

}  // namespace ccm
