// Programmatic dependent launch.
#pragma once
#include <cuda_runtime.h>

namespace rks {

// Programmatic launch: a kernel launched by launch_pdl may start before the one
// in front of it in the stream has ended; pdl_wait returns when that one has
// ended and its writes are visible (at once in a kernel launched normally).
// pdl_next lets the next such kernel start; its CTAs come in as this kernel's
// leave.  Every thread of a kernel launched so calls pdl_wait before it reads
// or writes what kernels in front of it touch; before that only data that was
// complete when the kernel in front started is read.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Loads through a const __restrict__ argument may be taken for invariant and
// moved ahead of the wait; through a pointer passed here after it they are not.
template <class T>
__device__ __forceinline__ T* pdl_fresh(T* p) {
  asm volatile("" : "+l"(p)::"memory");
  return p;
}
__device__ __forceinline__ void pdl_next() { asm volatile("griddepcontrol.launch_dependents;"); }

template <class... P, class... A>
void launch_pdl(void (*k)(P...), dim3 g, int b, size_t sm, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  cfg.gridDim = g;
  cfg.blockDim = dim3((unsigned)b);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  (void)cudaLaunchKernelEx(&cfg, k, static_cast<P>(args)...);   // an error stays in cudaGetLastError, as with <<<>>>
}

}  // namespace rks
