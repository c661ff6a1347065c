// Programmatic dependent launch: a kernel launched with launch_dependent() may be set up on the SMs
// while the one before it in the stream still runs, once all CTAs of that one have called
// pdl_trigger() (or it ends).  Everything a kernel reads or writes that an earlier kernel of the
// stream may write or read comes after its pdl_wait(), which returns when the earlier kernels have
// ended and their writes are visible; before it stand index arithmetic and reads of data that no
// kernel changes.  Pointers to what earlier kernels write are not __restrict__: a load the compiler
// takes for invariant may move above the wait, and goes through the non-coherent path, where the SM's
// L1 can still hold a line from before.  Both calls do nothing in a kernel launched the ordinary way.
// The trigger comes after the wait: before it, kernel after kernel of a stream would come to sit on
// the SMs, and blocks go where one has just left instead of spreading.
#pragma once

#include <cuda_runtime.h>

#include <utility>

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool dependent, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <typename... P, typename... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  return launch_kernel(true, kernel, grid, block, smem, st, std::forward<A>(args)...);
}
