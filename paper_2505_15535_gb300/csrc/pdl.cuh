// Programmatic dependent launch: a launch may let the stream's next launch be scheduled while it
// drains, and that one waits before it touches what earlier launches write.
#pragma once
#include <cuda_runtime.h>

namespace nhmf {

// Let the stream's next launch start once every block of this one has started; wait until the
// launches before this one are complete and their writes visible.  Both do nothing where a kernel
// is launched without the attribute.
__device__ __forceinline__ void pdl_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One launch; with `pdl` its blocks may start once every block of the launch before it has started
// (and must not touch that launch's output, or anything it reads, before pdl_wait).  Every kernel
// launched so calls pdl_wait, so that the completion of one launch is that of all before it.
// What that launch writes is no constant of this grid's lifetime, also after the wait: it is read
// through pointers without __restrict__ and not by ld.global.nc.
template <typename KernelT, typename... Args>
cudaError_t launch(KernelT kernel, dim3 grid, int threads, size_t smem, cudaStream_t s, bool pdl, Args... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace nhmf
