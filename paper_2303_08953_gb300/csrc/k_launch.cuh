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
//
// Such a kernel is alive while its predecessor still writes, so what a kernel
// on the stream may write (vectors, blocks, partial sums, small matrices,
// matrix values) is not read-only for its lifetime, and must not be loaded as
// if it were: no __ldg, and no pointer that is both const and __restrict__.
// Its loads are plain ones, which the wait's memory clobber keeps behind it;
// where the load is an asm of its own without a clobber (__ldcs), the pointer
// is offset by the zero that wait_previous returns, so that the load depends
// on the wait.  Read-only loads remain for a matrix's index arrays, which are
// complete (a stream synchronisation) before any product is launched.
// Measured with read-only loads everywhere and so: a 20-step matrix powers
// call on the 192^3 grid 2.29 ms both, a solve of 4096 rows 5.5 ms both.
#pragma once
#include <cuda_runtime.h>

#include "sg_internal.h"

namespace sg {

// returns 0, by a value that is known after the wait only
__device__ __forceinline__ int64_t wait_previous() {
  int64_t zero;
  asm volatile("griddepcontrol.wait;\n\tmov.b64 %0, 0;" : "=l"(zero)::"memory");
  return zero;
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
