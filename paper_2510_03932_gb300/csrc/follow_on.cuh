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

namespace ocpg {

__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// The start of every kernel that is launched this way: from here on it is ordered like any other.
// Its launch, its CTAs' start and its parameters' loads run beside the end of the launch before it: about 2 us
// of each short one (five callbacks of the cart-pole at N = 1e5 51.3 -> 41.8 us, three heat products of
// 37 cells at N = 7003 30.8 -> 24.6, an iteration of the constrained quadrotor at N = 33333 55.5 -> 48.8).
// A kernel lets the next one in by ending.  Let in from its start on, the next one's CTAs crowd the SMs that
// it leaves free, and FP64 work is bound by the fullest SM (the callbacks above 56.1 us, the iteration
// 61.0); from grids of at most 76 CTAs alone it gained nothing either (N = 1000: cart-pole callbacks 18.2 us
// without and 19.2 with it, step 7.1 and 7.4, Van der Pol step 6.5 and 6.8).
__device__ __forceinline__ void start_follow_on() { wait_for_previous(); }

// The launch of `kernel`: beside the end of the launch before it, or in the ordinary way.
inline cudaError_t launch_args(bool follow_on, const void* kernel, dim3 grid, int threads, size_t smem, cudaStream_t s,
                               void** args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = follow_on ? 1 : 0;
  cudaLaunchKernelExC(&cfg, kernel, args);
  return cudaGetLastError();
}
template <class T> struct Same { using type = T; };   // (arguments convert to the kernel's parameters)
template <class... P>
inline cudaError_t launch(bool follow_on, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                          typename Same<P>::type... args) {
  void* p[] = {&args...};
  return launch_args(follow_on, (const void*)kernel, grid, threads, smem, s, p);
}

}  // namespace ocpg
