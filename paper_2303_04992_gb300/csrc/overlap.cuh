// Launches that overlap the kernel before them on the stream: a dependent kernel's
// CTAs start while the last ones of its predecessor finish (as soon as every CTA of
// that has called overlap_trigger or ended), load their tables and wait in
// overlap_wait for the predecessor's memory.  The end of a kernel and the start of
// the next otherwise stand apart by about 1.5 us, a third of a kernel at N = 32.
//
// Used for the FP32 kernels at N <= 128 (a matvec at N = 32: 630 -> 584 us, at 128:
// 2688 -> 2625).  Early CTAs go where the predecessor drains first, which unbalances
// the grids that another resource bounds: FP64 at N = 64 lost 20 % so, N = 256 3 %.
//
// Rules.  A kernel launched so touches nothing that another kernel writes, and
// returns by no path, before overlap_wait; then all that was enqueued before it is
// complete, since its predecessor too has waited.  A kernel that calls
// overlap_trigger needs every CTA of its grid started for the next one to begin, so
// a waiting CTA never holds the place of one that it waits for.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace kfbim {

__device__ __forceinline__ void overlap_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void overlap_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// on = false: an ordinary launch of the same kernel (overlap_wait and
// overlap_trigger then do nothing).
template <typename... P, typename... A>
inline cudaError_t launch_overlapped(bool on, void (*kern)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                     A&&... a) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = on ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(a)...);
}

}  // namespace kfbim
