// Launches of kernels that follow one another on a stream with little work
// each (a joint of a kept round is 26 of them, most 2 to 7 us long; one of a round
// of a few attempts 6).
//
// A kernel launched by launch_next may be set up on the SMs while the one
// before it still runs; it starts with after_previous(), which waits until
// that one has ended and its writes are visible, and only then lets the next
// one be set up, so that at most one kernel waits at a time.  The order of the
// work is that of plain launches.  Only kernels of at most two blocks an SM are
// launched so: a waiting grid that fills the chip holds registers and shared
// memory that other jobs' streams could use meanwhile (24 jobs served on 16
// streams took 236 ms instead of 230 with every kernel launched so).
// Nor in a graph being captured: a branch's kernels follow each other closely
// there as it is, and the other branches want the SMs.
// Measured, a whole iteration with plain launches and so: L = 16, p = 512,
// S = 20 423 -> 357 us; a round of L = 20, p = 32, 100 attempts 131 -> 118.
#pragma once
#include <cuda_runtime.h>

namespace mcgpu {

#ifdef __CUDACC__

// (by every thread, before anything is read)
__device__ __forceinline__ void after_previous() {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
}

template <class... P, class... A>
inline cudaError_t launch_next(void (*kernel)(P...), unsigned blocks, unsigned threads, size_t smem, cudaStream_t st,
                               const A&... args) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  const cudaError_t e = cudaStreamIsCapturing(st, &capture);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = blocks <= 304 && capture == cudaStreamCaptureStatusNone ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

#endif  // __CUDACC__

}  // namespace mcgpu
