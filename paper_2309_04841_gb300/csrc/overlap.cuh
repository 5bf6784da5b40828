// overlap.cuh -- passes that may start while the one before them on the stream ends
// (programmatic stream serialisation): the launch and scheduling of a pass, its
// barriers, tables and whatever it may read early then cost no time of their own.  A
// pass waits (pdl_wait) before it touches anything that earlier passes write.  For
// the small-tile passes only: the streamed passes fill every SM with persistent CTAs,
// and the next pass's early ones cost more than they save (n = 23 p = 8 gradient 1609
// -> 1675 us, n = 30 p = 10 113.8 -> 114.7 ms).
#pragma once

#include <cuda_runtime.h>

namespace qaoa {

// Returns once every pass before this one has completed and its writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next pass on the stream start as soon as SMs have room.
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// overlap: the launch may start beside the pass before it.
template <class Kernel, class Params>
cudaError_t launch_pdl(Kernel kern, unsigned grid, int threads, size_t smem, const Params &P, bool overlap,
                       cudaStream_t s) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, P);
}

}  // namespace qaoa
