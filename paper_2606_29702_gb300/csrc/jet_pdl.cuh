// Programmatic dependent launch of the kernels of one call: a kernel may start
// while the one before it in the stream finishes, and waits at its first
// instructions until that one is complete and its writes are visible.  A call is
// three to five kernels, two of them of a few microseconds: back to back the
// launches and drains between them cost 7 us a call (2->64x6->1 BF16 step at 1024
// points 53.7 -> 46.0 us, 2->20x4->1 FP64 gradient at 1000 points 84 -> 77 us).
// A kernel is complete only when all its threads are past the wait, so each
// kernel's completion implies that of all before it.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace jet {

// every thread of every kernel launched by launch_dependent calls this first
__device__ __forceinline__ void dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}

}  // namespace jet
