// Programmatic dependent launch: kernels launched this way may be scheduled while the kernel before
// them on the stream is still draining (their launch latency then overlaps its tail).  They wait in
// the kernel until that one has completed and its writes are visible, before they touch global
// memory, and let their own successor be scheduled early in turn.  Launched the ordinary way, both
// device calls are no-ops.
#pragma once

#include "fasa_common.cuh"

__device__ __forceinline__ void pdl_wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

struct fasa_launch_shape {
  dim3 grid, block;
  size_t smem;
  int cluster_x;           // > 0: the CTAs of a grid row form one thread-block cluster of that size
  bool early;              // may be scheduled before its predecessor has completed
};
template <typename... Params, typename... Args>
cudaError_t fasa_launch(void (*kernel)(Params...), const fasa_launch_shape& l, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = l.grid;
  cfg.blockDim = l.block;
  cfg.dynamicSmemBytes = l.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  if (l.early) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (l.cluster_x > 0) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)l.cluster_x;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
template <typename... Params, typename... Args>
cudaError_t launch_after_predecessor(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     int cluster_x, Args... args) {
  return fasa_launch(kernel, fasa_launch_shape{grid, block, smem, cluster_x, true}, stream, args...);
}
