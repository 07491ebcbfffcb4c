// Programmatic dependent launch.  A kernel lets the next kernel of the stream start launching as soon as
// every one of its own blocks has started (pdl_trigger), and touches no global memory before every
// kernel it depends on has completed and its writes are visible (pdl_wait).  Blocks that wait hold only
// slots the earlier grids no longer need (all their blocks are resident by then), and launch latency at
// kernel boundaries overlaps the previous kernel's tail.
#pragma once

#include <cuda_runtime.h>

namespace ms {

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with programmatic stream serialisation (the kernel waits for its predecessors itself); errors
// surface through cudaGetLastError as for <<<>>> launches.
template <typename... P, typename... A>
void launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace ms
