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

// Whether a launch of this many CTAs gains from starting under the previous grid.  The
// early CTAs go to whichever SMs are free first and fill them up, so a grid with room
// for one CTA on each SM ends up two or three to an SM, the others idle; far smaller
// grids find free SMs anyway.  Overlapped or not, us per forward call: 8192 x 256 (row
// pass of 128 CTAs) 16.0 / 12.5, 9 x (4096 x 64) (column pass of 144) 20.1 / 15.5,
// DST-II of 2048 x 512 (column pass of 128) 9.8 / 8.6.  Asked where it was measured: the
// four-step family's forward row pass and the two-pass family's forward column pass.
// (The forward row pass after such a column pass wants the overlap: DCT-II of 2048 x
// 512 8.8 / 9.9.)
inline bool gains_from_overlap(long long ctas, int nsm) { return 2 * ctas <= nsm || ctas > nsm; }

// Launch, with programmatic stream serialization allowed if `overlap`.
template <typename... KArgs, typename... Args>
cudaError_t launch_if(bool overlap, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                      Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
  if (e != cudaSuccess) cudaGetLastError();  // reported here, not to the next caller that asks
  return e;
}
template <typename... KArgs, typename... Args>
cudaError_t launch(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  return launch_if(true, kern, grid, block, smem, s, std::forward<Args>(args)...);
}

}  // namespace pdl
}  // namespace gbdct
