// Launches that overlap the end of the previous kernel on the stream.
//
// A short kernel's launch costs about as much as its work: the solver's
// products with A and its small block products take 3 to 10 us each and
// follow one another by the hundred.  launch_early starts a kernel's CTAs as
// soon as every CTA of the previous kernel has passed its release_next (or
// ended); the kernel waits in wait_previous, before its first access to
// memory, until the previous kernel has completed and its writes are visible.
// Every kernel launched this way calls both, in that order, so that at most
// one kernel is ahead, and no kernel starts before its predecessor's
// predecessor has completed.
#pragma once
#include <cuda_runtime.h>

#include "sg_internal.h"

namespace sg {

__device__ __forceinline__ void wait_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
__device__ __forceinline__ void release_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// early = false: a plain launch (as while the stream is captured: there the
// predecessor may be a copy).  CTAs that start early go where there is room
// at that moment, so a kernel bound by its arithmetic loses by it once an SM
// takes several of its CTAs: the FP64-pipe products start early only with at
// most one CTA per SM (fills_once).  A training step at n = 65535 was 10 %
// slower with all of them early; a solve at n = 4096 is 15 % faster.
inline bool fills_once(dim3 grid) {
  return static_cast<int64_t>(grid.x) * grid.y * grid.z <= device_sm_count();
}

template <typename... P, typename... A>
void launch_early(bool early, void (*kernel)(P...), dim3 grid, int block, size_t smem,
                  cudaStream_t st, A&&... args) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  if (early) SG_CUDA(cudaStreamIsCapturing(st, &capture));
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(static_cast<unsigned>(block));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = early && capture == cudaStreamCaptureStatusNone ? 1 : 0;
  SG_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
}

}  // namespace sg
