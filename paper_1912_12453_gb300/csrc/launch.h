// Kernels that start while the one before them ends (programmatic dependent
// launch).  In a chain of short kernels the launch latency and the reading of
// indices is a good part of each; a kernel launched by launch_next is set up
// when its predecessor lets it and reads what does not change
// between launches -- connectivity, lists, preconditioner blocks -- before it
// waits for the predecessor's results (wait_previous).
//
// Rules that keep a chain in order:
//  - every thread of a kernel launched this way calls wait_previous before it
//    reads or writes anything that another launch writes or reads, and before
//    any return; the wait covers the predecessor's completion and, through the
//    predecessor's own wait, everything before it;
//  - wait_previous lets the next kernel start only once it has returned, so
//    at most one kernel is ahead;
//  - pointers to changing data go through wait_previous, which gives the
//    compiler a new value: no load through them moves above the wait.
#pragma once

#include <cuda_runtime.h>

namespace chns {

#ifdef __CUDACC__
template <class P>
__device__ __forceinline__ void after_wait(P &p) {
  asm volatile("" : "+l"(p)::"memory");
}
template <class... P>
__device__ __forceinline__ void wait_previous(P &...p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  (after_wait(p), ...);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
inline void launch_next(void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t st, A &&...args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}
#endif

}  // namespace chns
