// Programmatic dependent launch: a kernel launched with launch_dependent may start while the
// kernel before it in the stream (or captured graph) is finishing, so that its launch latency
// and its prologue -- barriers, tensor memory, constant operators -- overlap that kernel's
// tail.  Every such kernel calls grid_wait() in every thread before it reads or writes anything
// that an earlier kernel touches: it returns when the kernel before it has completed and its
// writes are visible.  grid_wait() also lets the next kernel start its own prologue; as that
// happens only after the wait, at most two neighbours in a chain overlap.  Without `early` the
// launch waits for the kernel before it as any other.
//
// Pointers to what earlier kernels write carry no __restrict__ in such a kernel: with it the
// compiler may take the data for unchanging and load them ahead of the wait.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace ridg {

__device__ __forceinline__ void grid_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... Params, typename... Args>
cudaError_t launch_dependent(bool early, void (*kern)(Params...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute a;
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &a;
  c.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&c, kern, Params(std::forward<Args>(args))...);
}

}  // namespace ridg
