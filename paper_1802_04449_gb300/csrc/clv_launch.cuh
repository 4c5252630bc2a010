// clv_launch.cuh -- launches that overlap the end of their predecessor.
#pragma once
#include <cuda_runtime.h>

namespace clv {

// Kernels of a chain -- a step, a freeze-out find, a training run -- start while
// their predecessor drains (programmatic dependent launch): nothing of one is
// done before its predecessor is complete and its writes visible
// (enter_step_kernel; so what the chain writes is read by plain loads, not
// through the read-only path), and the next one may be placed once every CTA of
// this one has released it or is done.  Kernels of many small blocks release it
// as they start; the stage kernels, at most one wave of large CTAs, do not: the
// small blocks of the next kernel would be placed on the SMs that are free then,
// and the others stay empty (33 x 33 x 9 in FP64, 132 CTAs on 152 SMs: 141 us a
// step instead of 84).  Nor does the direct stage kernel (kernel = 1), whose
// next launch runs the same code: ten steps of 33 x 33 x 9 viscous cells in FP32
// took 282 us with a release at its start, 273 as plain launches and 240
// without one; 45 x 45 x 21 cells 479, 494 and 424.  No effect on a plain launch.
__device__ __forceinline__ void enter_step_kernel() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void release_next_kernel() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
template <typename... P, typename... A>
inline void launch_step_kernel(void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t st,
                               const A&... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(block);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = &at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, kernel, P(args)...);   // an error is left for cudaGetLastError, as by <<<>>>
}

}  // namespace clv
