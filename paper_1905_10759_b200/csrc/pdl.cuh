// Programmatic dependent launch: a kernel launched with launch_pdl may be scheduled while the kernel before
// it in the stream is still running (as soon as every CTA of that kernel has executed
// pdl_launch_dependents or exited), so its launch latency and per-CTA set-up (barrier initialisation,
// tensor-memory allocation, address tables) overlap the predecessor's tail.  It must execute pdl_wait in
// every thread before it touches global memory: the wait returns when the preceding kernel has completed
// and its writes are visible -- which also keeps the ordering transitive along a chain of such kernels.
// Short kernels without set-up (streams, matrix-vector, integer tiles) wait and never signal: their end does.  A signal as
// the first instruction lets every following launch of the stream move in while this one still works -- graph replays of
// binarize_dense of 4646 x 688 at beta 48 91 us instead of 34, 1702 rows quantized at beta 8 3.1 instead of 2.0, of
// hbmm_gemm on 3 rows of 2057 x 5248 6.6 instead of 4.4; with the wait alone all of them are at or below a plain launch.
// The quantizer signals after its wait, for the set-up of the contraction behind it (2 % of that pair).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cstdint>
#include <utility>

namespace hbmm {

__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// One element, as fp32, of a tensor that the kernel before may have written.  Volatile, so that it stays behind pdl_wait (and where
// it is written, among other such loads), and a plain load: the read-only kind (__ldg, ld.global.nc) promises memory that nobody
// writes while this kernel lives, and its life began before the wait.
template <typename T> __device__ __forceinline__ float load_elem(const void* p);
template <> __device__ __forceinline__ float load_elem<float>(const void* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return v;
}
template <> __device__ __forceinline__ float load_elem<__nv_bfloat16>(const void* p) {
  unsigned short v;
  asm volatile("ld.global.u16 %0, [%1];" : "=h"(v) : "l"(p));
  return __uint_as_float(static_cast<uint32_t>(v) << 16);
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(std::forward<Args>(args))...);
}

// The same in clusters of `cluster` consecutive CTAs (the grid is a multiple of it).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, unsigned cluster, size_t smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(std::forward<Args>(args))...);
}

}  // namespace hbmm
