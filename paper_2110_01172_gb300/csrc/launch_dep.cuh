// launch_dep.cuh - programmatic dependent launch between the kernels of a
// transform (and of consecutive transforms on one stream).
//
// A kernel launched with the programmatic-serialization attribute may start
// while the previous kernel on its stream is still finishing: its CTAs take
// the SMs the previous grid's last partial wave leaves idle and run their
// prologue (index arithmetic, barrier setup).  Every thread calls
// wait_prior_grid() before its first access to global memory other than the
// plan's read-only tables; that wait returns once the previous grid has
// completed and its writes are visible, so the order of all reads and writes
// of the data is the same as without the attribute.  Each CTA calls
// launch_dependents() once its FFT is done, before its final stores, which
// lets the next kernel launch once every CTA of this grid has reached that
// point (triggering on entry instead measured slower at 4096^2, 141 vs 132 us
// per forward + inverse step: a whole wave of the next grid then sat in its
// wait on the SMs).
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace gbdct {
namespace pdl {

__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prior_grid() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with programmatic stream serialization allowed.
template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
  if (e != cudaSuccess) cudaGetLastError();  // reported here, not to the next caller that asks
  return e;
}

}  // namespace pdl
}  // namespace gbdct
