// Launches of a chain of dependent kernels in one stream whose launch latencies
// overlap (programmatic dependent launch): a kernel of the chain calls
// chain_enter() before anything else, waits there for the kernel before it and
// lets the next one be launched; launch_chained() permits the early launch.
// Every block has to pass chain_enter(), also one that has nothing to do: a
// kernel that could end before its predecessor would let its successor start
// too early.  The kernel is resident while its predecessor still writes, so what
// another kernel of the chain writes is read by ordinary loads after the wait,
// which its memory clobber orders.  Loads through __ldg or from const __restrict__
// parameters are defined for memory that nobody writes while the kernel lives:
// they are for links, and for the shadow vector r_hat, which only the restart
// kernels write, outside the chain (launched in the ordinary way they run alone).
#pragma once

#include <cuda_runtime.h>

namespace wd {

__device__ __forceinline__ void chain_enter() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                  A... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace wd
