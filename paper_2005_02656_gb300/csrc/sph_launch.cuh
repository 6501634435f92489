// Kernel launches of the step's chain with programmatic dependent launch: a
// kernel's blocks are scheduled as soon as the one before it has started its
// last blocks, and wait (dep_enter) until it has finished and its writes are
// visible.  The launch latency and the block start-up of each kernel then hide
// behind its predecessor, which is a large part of a small state's step (about
// 30 launches).  Every kernel launched this way calls dep_enter before it
// touches memory.  What the kernel before it in the stream writes is read by
// ordinary loads only: the read-only path (__ldg, const __restrict__ parameters)
// is for data that nobody writes while the grid exists, and dep_enter does not
// order it.  What was written two or more kernels back is complete when a
// kernel's blocks are scheduled (the one between was past its wait), and may be
// read either way.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace sph {

// The searches are persistent and take most of an SM's shared memory: launched
// early, some of their CTAs meet an SM that still runs the gather with a small
// shared-memory share, start late, and the whole share of cells they own with them.
// Early against plain (us per step): staged search 8,000 particles 135.5 / 139.2,
// 103,823 (stage calls) 307.4 / 311.2, 125,000: 405.8 / 400.5, 250,047: 607.8 /
// 612.3, 512,000: 1,141 / 1,125, 8.4M: 14,864 / 14,630; list search (FP64) 8,000:
// 246.3 / 247.7, 32,768: 617 / 601, 250,047: 3,379 / 3,364, 1.07M: 13,735 / 13,660.
constexpr int64_t kEarlyMasksN = 400000;
constexpr int64_t kEarlyListsN = 20000;
// The FP64 pair kernels: early CTAs take slots from the end of the pass before
// them.  Early against plain (us): 32,768 particles 601 / 606, 64,000 (20 steps and
// gradient, ms) 109.9 / 110.1, 125,000: 1,845 / 1,837, 1.07M: 13,700 / 13,521,
// 1.0M square patch (stage calls) 10,658 / 10,511.
constexpr int64_t kEarlyPairsN = 100000;

template <class... P, class... A>
inline void launch_dep_if(bool early, void (*kernel)(P...), unsigned grid, unsigned block,
                          size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = early ? 1 : 0;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}

template <class... P, class... A>
inline void launch_dep(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem,
                       cudaStream_t st, A&&... args) {
  launch_dep_if(true, kernel, grid, block, smem, st, std::forward<A>(args)...);
}

// Waits for the kernels before this one in the stream, then lets the next
// one's blocks be scheduled.
__device__ __forceinline__ void dep_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

}  // namespace sph
