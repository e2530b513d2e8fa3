// Programmatic dependent launches: a kernel's launch and prologue overlap the tail of the
// stream's previous kernel.
//
// A kernel launched by launch_dependent calls pdl_wait() before it reads or writes memory
// that earlier work in the stream may touch (constant tables of the context aside), in every
// CTA, and pdl_trigger() after it, which lets the stream's next such launch be scheduled once
// every CTA of this grid is running: a waiting grid can therefore not keep this one's CTAs
// from an SM.  A pass that triggers still writes W after it: whoever launches a dependent behind
// it waits before reading W, as these kernels do.  As each of these grids waits for its predecessor before it does anything, its
// completion implies that of all earlier work.  The long tensor-core weight passes do not
// trigger: the next pass's coefficient kernel, resident beside them from their start, cost
// the 7B set's r = 32 pass 4% (4.16 ms against 3.99).
//
// The refresh's launches are dependent ones where few chunks make them latency-bound
// (zo_cholqr.cu).
//
// A pass of one 2048 x 2048 matrix at r = 32 went from 26.7 us (four ordinary launches) to
// 16.2 us (three dependent ones).
#pragma once

#include <cuda_runtime.h>

namespace zo {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// cluster: CTAs per cluster (1: none, or the kernel's own __cluster_dims__).  dependent =
// false: an ordinary launch, after everything before it has completed.
template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, unsigned block, size_t smem,
                             cudaStream_t s, unsigned cluster, bool dependent, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (dependent) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace zo
