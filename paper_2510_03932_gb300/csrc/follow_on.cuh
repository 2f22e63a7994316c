// Launches that may overlap the end of the launch before them on their stream (programmatic
// dependent launch).  The CTAs of such a launch take the SMs as the launch before it leaves them
// (once all of its CTAs have run let_next_start() or ended) instead of when it has ended.
//   wait_for_previous() returns when the launches before have ended and their writes are visible;
//   it is a no-op in a kernel that was launched in the ordinary way.  Every thread of a kernel that
//   is launched with follow_on = true runs it, before its first access to anything that an earlier
//   launch writes or reads, and in any case before its end, so that what comes after this launch
//   comes after all of them.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace ocpg {

__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch(bool follow_on, void (*kernel)(P...), int64_t grid, int threads, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = follow_on ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

}  // namespace ocpg
