// Kernels of one call that follow each other on a stream, launched so that the next one's
// CTAs are placed as the last ones of its predecessor end, without waiting for the launch in
// between (programmatic dependent launch). Every kernel launched with `after` waits for its
// predecessor's end (grid_wait) before it reads anything that the call computes. The order is
// that of the stream: a kernel ends behind its own wait, so behind everything before it.
// What bounds the small products is the latency of these kernels one after the other: a
// 200 x 136 x 311 tile took 65.0 us, 59.4 now; dense 1100 111.2 and 106.3; Bernoulli 2048
// 107.8 and 103.0. Letting the successor in any earlier (griddepcontrol.launch_dependents at
// the top of the exponent and slicing kernels) takes its places from the predecessor's own
// work: Bernoulli 2048 111.1 us, a batch of 48 products 18.2 ms against 17.7.
#ifndef BSMM_OVERLAP_CUH
#define BSMM_OVERLAP_CUH

#include <cuda_runtime.h>

namespace bsmm {

__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// after: the stream's previous operation is a kernel of the same call
template <class... P, class... T>
cudaError_t launch_kernel(bool after, void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st,
                          unsigned cluster, const T&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2] = {};
  cfg.attrs = at;
  if (cluster > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[cfg.numAttrs].val.clusterDim.x = cluster;
    at[cfg.numAttrs].val.clusterDim.y = at[cfg.numAttrs].val.clusterDim.z = 1;
    cfg.numAttrs++;
  }
  if (after) {
    at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs++;
  }
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace bsmm

#endif
