// lbm_pdl.cuh -- programmatic dependent launch of the kernels that follow one
// another step after step (sm_103a).
//
// A kernel launched by launch_dep may start its blocks while the kernel before
// it on the stream still runs, once every block of that one has passed
// allow_next() (or ended); after_previous() itself returns when the
// kernel before has completed and its writes are visible.  So the launch
// latency, the block scheduling and what a kernel does before
// after_previous() overlap the tail of the step before.  Nothing that an
// earlier kernel writes is read, and nothing that it reads is written, before
// after_previous().  Kernels launched otherwise wait for all of this as usual.
// Captured into graphs as programmatic edges.
#pragma once

#include <cuda_runtime.h>

namespace lbmk {

__device__ __forceinline__ void after_previous() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// From here on the next kernel's blocks may be placed.  Late in a kernel, so
// that they find the SMs evenly loaded: placed at its start they crowd onto
// the SMs with a slot to spare, and a grid of one wave then waits for those
// (the 256 x 256 reverse sweep 7.9 -> 8.9 ms).
__device__ __forceinline__ void allow_next() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline void launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       const A&... args) {
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);  // errors: cudaGetLastError
}

}  // namespace lbmk
