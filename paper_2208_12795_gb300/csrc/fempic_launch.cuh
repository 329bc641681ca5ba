// Launches of a step's kernels, which follow each other on one stream: each may
// be set up while the one before it still runs (programmatic stream
// serialization) and waits for that one's end before its first access to
// memory.  What follows a step (another library's kernel, a copy, an event)
// is ordered as after any kernel.  A kernel is resident while the ones before it
// still write, so what they write (fields, coefficients, per-tet terms, a
// caller's DoFs) is read with plain loads; the non-coherent path (__ldg, const
// __restrict__) is for the tables that are fixed once per mesh.
#pragma once
#include <cuda_runtime.h>

namespace fempic {

// First statement of every kernel launched below: the kernels before it on the
// stream have ended and their writes are visible; the next may be set up.
__device__ __forceinline__ void grid_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... Q>
inline void launch(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st, Q&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &attr;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, P(args)...);   // errors: cudaGetLastError, as after any launch
}

}  // namespace fempic
