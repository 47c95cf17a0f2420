// Programmatic dependent launch for chains of short kernels: a kernel launched with launch_pdl may be
// put on the SMs while the one before it still runs, does what needs no memory of its (barriers,
// TMEM, descriptors), and waits in pdl_wait until that kernel has completed and its writes are
// visible.  Every kernel launched this way calls pdl_wait before its first access to global memory,
// so that the order along a stream is complete: a kernel's completion implies that of all before it.
// Between two short kernels this hides the launch and the set-up, about 2 us: the 26 operations of a
// training step at batch 4096 took 264 us and take 223, the per-species networks (136 launches for
// 131072 cells) 5337 and 5137.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace chem {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// the next kernel of the stream may be scheduled once every block has called this (or ended)
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid; c.blockDim = block; c.dynamicSmemBytes = smem; c.stream = stream;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
}

}  // namespace chem
