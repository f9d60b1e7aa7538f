// Programmatic dependent launch of the step kernels.
//
// A step is one or two launches of a few microseconds, each of which starts by
// reading what no launch of a run writes (row pointers, columns, couplings, row
// heads, work items). Launched with launch_pdl, a kernel's CTAs start while the last
// CTAs of the launch before still run, read those, and wait in pdl_wait() until
// that launch has finished and its writes are visible; only then do they touch x,
// y, sign bytes, U rows or anything else that a launch writes -- by plain loads:
// a read-only load (__ldg) is neither ordered by the wait nor allowed on data that
// changes while the kernel is resident. pdl_wait() then lets the next launch start in
// the same way. Every kernel launched with launch_pdl calls it in all CTAs that touch
// such data, so each launch is complete before the one after it goes on, and all
// earlier ones with it. Graph replays keep the edges. Launch by launch / with this,
// us: 400 steps and 20 readouts of 10,214 rows at R = 50 3298 / 2415, a gradient step
// of 10,878 rows at R = 32 (115 launches) 1337 / 1038.
#pragma once
#include <cuda_runtime.h>

namespace sbd {

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename A>
cudaError_t launch_pdl(void (*kernel)(A), dim3 grid, int block, const A& args, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args);
}

}  // namespace sbd
