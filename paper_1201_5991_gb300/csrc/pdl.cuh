// Programmatic dependent launch for the solve phase's short kernels: a kernel launched with launch_pdl may be
// set up, and its blocks may become resident, while the kernel before it in the stream still runs; pdl_wait,
// its first instruction that touches global memory depends on, returns when that kernel has completed with
// its stores visible.  Every such kernel waits, so completion is transitive along the stream.  pdl_trigger lets
// the next kernel be set up once every block of this one has started (it would otherwise be at its end).
// Such a kernel is alive while the kernels before it still write, so what they write may not be read as data that
// is constant for the kernel's life: no __ldg, and no const __restrict__ parameter (from which the compiler
// makes the same loads), for vectors of the running solve.  Data of the set-up may be read so.
// Use only where the launch before it in the same stream is a kernel (not a copy, a memset or an event wait):
// the attribute speaks of the kernel before.  Helpers that are called in either place take after_kernel.
#pragma once

#include <cuda_runtime.h>

namespace bddc {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... P, typename... A>
inline void launch_pdl_if(int after_kernel, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = after_kernel ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

template <typename... P, typename... A>
inline void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  launch_pdl_if(1, kernel, grid, block, smem, st, args...);
}

}  // namespace bddc
