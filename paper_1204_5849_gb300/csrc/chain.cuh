// chain.cuh -- launches of the kernels that follow one another on the pool's stream.
//
// A step is a chain of launches (restriction and fill per level, finalisation, update,
// reflux), many of them a few microseconds long, so the gap between a kernel's last block
// and the next one's first counts.  Every kernel of the chain is launched with programmatic
// stream serialisation, so that its launch and its set-up (shared-memory barriers, schedules)
// overlap the end of the kernel before.  The rules that keep the order of plain launches:
//  * every block of every chained kernel reaches chain_begin() before it ends.  It waits there
//    until the kernel before has completed and its writes are visible; that kernel waited for its
//    own predecessor, so all earlier ones have completed too.
//  * before chain_begin() a kernel touches no memory that a kernel writes.  The step kernel reads
//    its block list and the blocks' geometry there: these are written by host copies only, which
//    order like plain launches, and no kernel of the chain may ever write them.
//  * after chain_release() (or its end) a block may still write: the next kernel, though set up,
//    waits for the whole of this one.  finalize_kernel releases first of all, the step kernel before
//    its last reductions, the others with their end.
//
// Per pass, plain launches -> this: 2D MMC 128^2, ten steps 246 -> 245 us; 2D HLLC 720x528, four
// steps 288 -> 281; 3D MMC 112x80x96, four steps 1096 -> 1086; rotor quadtree, four steps 1007 ->
// 1000 (each with a CUDA graph per step).  The next kernel let in at the start of each kernel gave
// 3 us more on the first and took 40 us from the 8^3 octree step (4990 -> 5030: waiting blocks hold
// register and shared-memory space while the step kernel's last blocks run).
#pragma once
#include <cuda_runtime.h>

namespace mapgb {

__device__ __forceinline__ void chain_begin() { cudaGridDependencySynchronize(); }

// Lets the next kernel of the chain be set up once every block has called this or ended.
__device__ __forceinline__ void chain_release() { cudaTriggerProgrammaticLaunchCompletion(); }

template <typename... P, typename... A>
inline cudaError_t launch_chained(void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

}  // namespace mapgb
