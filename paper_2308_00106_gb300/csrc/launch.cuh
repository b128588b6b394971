// launch.cuh -- kernels that follow one another on a stream without the gap
// between launches (programmatic dependent launch).
//
// A kernel started by launch_after may become resident while the kernel before
// it on the stream still runs; it calls after_previous() before its first
// access to memory that an earlier kernel writes or reads, which returns once
// that kernel has ended and its writes are visible.  (Arrays of a finished
// handle are written by nobody and may be read before.)  A kernel calls
// start_next() when its own successor may become resident: the short kernels do
// so at their start.  Without it, when its last CTA ends: the product kernels fill
// the SMs, and CTAs started early would pile up on those that free first (power
// iteration 980 us -> 1105 us with it everywhere, 805 us so).  A successor that was
// launched the usual way waits for the whole kernel as always.
#pragma once

#include "internal.cuh"

namespace maxe {

__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void start_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem, cudaStream_t st,
                         A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace maxe
