// Launches of the kernels that follow one another within and between steps.
#pragma once

#include <cuda_runtime.h>

namespace crkfr {

// SMs of the GPU (asked once; 0 if the query failed)
inline int sm_count() {
  static const int sms = [] {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    return v;
  }();
  return sms;
}

// A launch that may be scheduled while the kernel before it in the stream
// finishes (programmatic stream serialization): its blocks take free places
// once all blocks of that kernel have come to chain_end() (or left) and wait in
// chain_begin() until it has completed and its writes are visible.  Saves 1.2
// us of the gap between two kernels: 20 steps of 100 elements 132 -> 109 us, 8
// steps of 65 x 47 elements (two kernels each) 208 -> 188 us.  In a stream
// capture the launch is an ordinary one.
// `cluster`: the grid as one cluster of that many blocks (0: none).
template <class... P>
int launch_chained_cluster(void (*kernel)(P...), dim3 grid, unsigned block, unsigned cluster,
                           cudaStream_t s, P... args) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  const bool plain = cudaStreamIsCapturing(s, &capture) != cudaSuccess ||
                     capture != cudaStreamCaptureStatusNone;
  if (plain) cudaGetLastError();
  cudaLaunchAttribute attr[2] = {};
  unsigned attrs = 0;
  if (cluster) {
    attr[attrs].id = cudaLaunchAttributeClusterDimension;
    attr[attrs].val.clusterDim.x = cluster;
    attr[attrs].val.clusterDim.y = 1;
    attr[attrs].val.clusterDim.z = 1;
    ++attrs;
  }
  if (!plain) {
    attr[attrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[attrs].val.programmaticStreamSerializationAllowed = 1;
    ++attrs;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = attrs;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  const cudaError_t last = cudaGetLastError();
  return (int)(e != cudaSuccess ? e : last);
}

template <class... P>
int launch_chained(void (*kernel)(P...), dim3 grid, unsigned block, cudaStream_t s, P... args) {
  return launch_chained_cluster<P...>(kernel, grid, block, 0, s, args...);
}

#ifdef __CUDACC__
// First statement of a kernel launched by launch_chained that touches global
// memory: waits for the kernel before.
__device__ __forceinline__ void chain_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
// Lets the next kernel of the stream be scheduled once every block has come
// here: late in a kernel, when its blocks are about to leave.  (Said at the
// start, the next kernel's blocks filled the few free places left beside a
// small grid, several to an SM: the residual of 60 x 40 elements at N = 2 took
// 33.5 us, 21.5 unchained and 17.5 now; 65 x 47 elements 171 -> 161 us.  Large
// meshes pay 1 %: 1024 x 1024, N = 3, 5.22 -> 5.27 ms for two steps.)
__device__ __forceinline__ void chain_end() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
#endif

}  // namespace crkfr
