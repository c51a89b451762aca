// Kernel launches with programmatic dependence (internal).
//
// Every kernel of the library is launched so that its blocks may start while the kernel
// before it in the stream still runs (programmatic stream serialization), and waits in
// grid_wait() for that kernel to end before it touches global memory.  Launch latency and the
// set-up of a block (barriers, TMEM, constant operands) then run under the tail of the
// kernel before, which is most of what a small call's chain of kernels consists of.
//
// grid_trigger() lets the next kernel's blocks start once all blocks of this kernel have
// called it.  A kernel that allocates TMEM calls it after the allocation: a block of a later
// kernel that holds TMEM and waits can then never keep a block of an earlier one from its
// allocation.  Every kernel waits in every block, so that a kernel's end implies that all
// kernels before it have ended.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <utility>

namespace fs {

#ifdef __CUDACC__
__device__ __forceinline__ void grid_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Returns 0, in a form that the compiler takes for the result of the wait: indexes and
// pointers that it is added to cannot be read through before the wait, even where the data
// is declared constant.  The pointers passed by reference get it added.
template <typename... P>
__device__ __forceinline__ int64_t grid_wait(P&... p) {
  int64_t zero;
  asm volatile("griddepcontrol.wait;\n mov.b64 %0, 0;" : "=l"(zero)::"memory");
  ((p += zero), ...);
  return zero;
}
// At the top of a kernel without TMEM.
template <typename... P>
__device__ __forceinline__ int64_t grid_begin(P&... p) {
  grid_trigger();
  return grid_wait(p...);
}

template <typename... P, typename... A>
cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(std::forward<A>(args))...);
  if (e != cudaSuccess) (void)cudaGetLastError();  // reported here, not to the caller's next check
  return e;
}
#endif

}  // namespace fs
