// chain.cuh -- launches of the kernels that follow one another on the pool's stream.
//
// A step is a chain of launches (restriction and fill per level, finalisation, update,
// reflux), many of them a few microseconds long, so the gap between a kernel's last block
// and the next one's first counts.  Every kernel of the chain is launched with programmatic
// stream serialisation and calls chain_begin() before it touches global memory: it waits
// there until the kernels before it have completed and their writes are visible.  The order
// of all accesses is that of plain launches; only the launch and the set-up before the wait
// (shared-memory barriers, schedules) overlap the end of the kernel before.
//
// Per pass, plain launches -> this (graph-replayed steps): 2D MMC 128^2, ten steps 246 -> 245
// us; 2D HLLC 720x528, four steps 288 -> 281; 3D MMC 112x80x96, four steps 1096 -> 1086;
// rotor quadtree, four steps 1007 -> 1000.  Letting the next kernel's blocks in at the start
// of each kernel (an explicit trigger) gave 3 us more on the first and took 40 us from the
// 8^3 octree step (4990 -> 5030: waiting blocks hold register and shared-memory space while
// the step kernel's last blocks run), so the trigger is left to each kernel's end.
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
