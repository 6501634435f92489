// Kernel launches of the step's chain with programmatic dependent launch: a
// kernel's blocks are scheduled as soon as the one before it has started its
// last blocks, and wait (dep_enter) until it has finished and its writes are
// visible.  The launch latency and the block start-up of each kernel then hide
// behind its predecessor, which is a large part of a small state's step (about
// 30 launches).  Every kernel launched this way calls dep_enter before it
// touches memory.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace sph {

template <class... P, class... A>
inline void launch_dep(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem,
                       cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

// Waits for the kernels before this one in the stream, then lets the next
// one's blocks be scheduled.
__device__ __forceinline__ void dep_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

}  // namespace sph
