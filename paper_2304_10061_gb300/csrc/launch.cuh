// Kernel launches with programmatic dependent launch: a kernel's blocks are scheduled as the last
// blocks of the kernel before it leave, without waiting for the flush between the two, and wait
// (pdl_wait) until that kernel has completed and its writes are visible before they touch memory.
// An evaluation is 15 to 60 dependent kernels in a row, and launch and ramp are a good part of the
// short ones: 64 atoms 252 -> 196 us, 3,072 atoms TF32 1,240 -> 1,136 us, 4,096 atoms MD 9.20 -> 8.33 ms,
// 1,048,576 atoms 115.9 -> 115.6 ms.  No kernel signals its dependents early (launch_dependents): blocks
// that wait from a kernel's start slow the kernel they wait for (1,048,576 atoms 120.4 ms, 64 atoms
// 207 us).
// (The allocation-free neighbour search and the FP8 weight quantiser are launched plainly.)
// Every kernel launched this way calls pdl_wait before its first access to global memory, so the
// order of the kernels' effects is the stream's.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace alg {

// until every kernel before this one has completed
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// (a failure is also left for cudaGetLastError, as after <<<>>>)
template <typename... P, typename... A>
inline cudaError_t launch_cluster(int cluster, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                  A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)cluster;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  return launch_cluster(1, kernel, grid, block, smem, st, std::forward<A>(args)...);
}

}  // namespace alg
