// bte_pdl.cuh -- programmatic dependent launch: the next kernel of the stream may start
// while this one runs (pdl_trigger) and waits for all of it, its writes included, before
// it touches anything that a step changes (pdl_wait).
#pragma once
#include <cuda_runtime.h>

namespace bte {

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch that may start before the stream's previous kernel has ended (early), for a
// kernel in which every CTA calls pdl_wait; otherwise an ordinary launch.
template <typename... P, typename... A>
cudaError_t launch_pdl(bool early, void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = dim3(grid);
  c.blockDim = dim3(threads);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &at;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

}  // namespace bte
