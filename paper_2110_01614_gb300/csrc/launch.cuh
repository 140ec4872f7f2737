// Launches that may overlap the end of the kernel before them on the stream.
//
// A kernel launched with launch_overlapped is set up while its predecessor still
// runs; it touches global memory only after wait_for_predecessor(), which returns
// once the predecessor has finished and its writes are visible.  It calls
// release_successor() after that, so that no more than one such kernel waits at a
// time, and a kernel with TMEM only once a block barrier has followed its allocation:
// the successor's CTAs hold what they allocate until this kernel is done, so nothing
// that this kernel still needs may be left for them to take.  Its global loads are
// plain ones: a load marked invariant (__ldg, const __restrict__) might be moved
// ahead of the wait.  Kernels launched the ordinary way are unaffected on either
// side.  For kernels of a few microseconds the gap between two launches is a large
// part of a call.
#pragma once

#include <cuda_runtime.h>

namespace nsdf {

__device__ __forceinline__ void wait_for_predecessor() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ void release_successor() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

template <typename... P, typename... A>
cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t s,
                              A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace nsdf
