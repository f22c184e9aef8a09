// Programmatic dependent launch: a kernel's blocks may be scheduled while the kernel before it in the
// stream drains, and wait there. Every kernel launched this way calls pdl_begin() before its first
// access to global memory: it returns when the kernels before have completed and their writes are
// visible, then lets the next launch begin. (A chain of such launches is thus complete up to the
// kernel before, whichever kernels it mixes with.) It hides the 1 to 2 us from the end of one kernel
// to the start of the next, which is a tenth of the small calls' time (fit, hit index, network).
// The finder's kernels are launched plainly: its persistent blocks, scheduled while the seed states
// drain, pile up on the SMs that are free first (one event 137 against 143 us).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace kfgb {

__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
cudaError_t launch_pdl(void (*kernel)(P...), int grid, int block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(static_cast<unsigned>(block));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace kfgb
