// Programmatic dependent launch: a kernel launched through launch_pdl may start (block scheduling, barrier
// and tensor-memory set-up, descriptor prefetch) while the kernel before it on the stream is still draining;
// pdl_wait() then blocks until that kernel has completed and its memory is visible.  Nothing before
// pdl_wait() may touch global memory written by earlier kernels.  Outside such a launch both calls are no-ops.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>

__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A kernel may read, before its own pdl_wait(), what was complete before the launch in front of it began -- where that launch
// raises a flag after its own pdl_wait(), and before it lets its dependents start (pdl_raise, by one thread of it, then
// pdl_launch_dependents).  The reader's threads meet at pdl_early(): it sees the flag, and with it everything that the launch in
// front waited for, or else waits itself, so that a launch in front that raises none, or triggers first, costs time and not
// results.  The reader's last act is pdl_lower(), after its pdl_wait().
__device__ __forceinline__ void pdl_raise(int32_t* flag) { asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(flag), "r"(1) : "memory"); }
__device__ __forceinline__ void pdl_early(const int32_t* flag) {         // block-wide
  int32_t up = 1;
  if (threadIdx.x == 0) asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(up) : "l"(flag) : "memory");
  if (!__syncthreads_and(up == 1)) pdl_wait();
}
__device__ __forceinline__ void pdl_lower(int32_t* flag) { *flag = 0; }

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
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
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// With thread-block clusters of `cluster` blocks along x; `pdl`: as launch_pdl, else as launch_serial.
template <typename... KArgs, typename... Args>
cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, int cluster, bool pdl, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim = {(unsigned)cluster, 1, 1};
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// The same launch without the attribute: the kernel starts only when everything before it on the stream has
// completed (pdl_wait() inside it is then a no-op); the kernel behind it may still be launched through launch_pdl.
template <typename... KArgs, typename... Args>
cudaError_t launch_serial(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = nullptr;
  cfg.numAttrs = 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
