// Four consecutive elements of a row that may end inside them: absent elements read as zeros and are not written.
// VEC: the row starts on a 16-byte boundary (8 bytes for a bf16 row that is written) and k is a multiple of four.
#pragma once
#include <cuda_bf16.h>
#include <cstdint>

namespace hbmm {
namespace rowio {

template <bool VEC>
__device__ __forceinline__ void load4(const float* row, int64_t k, int64_t K, float (&v)[4]) {
  if (VEC && k + 4 <= K) {
    const float4 x = __ldg(reinterpret_cast<const float4*>(row + k));
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  } else {
#pragma unroll
    for (int e = 0; e < 4; e++) v[e] = k + e < K ? __ldg(row + k + e) : 0.0f;
  }
}

template <bool VEC>
__device__ __forceinline__ void store4(float* row, int64_t k, int64_t K, const float (&o)[4]) {
  if (VEC && k + 4 <= K) {
    *reinterpret_cast<float4*>(row + k) = make_float4(o[0], o[1], o[2], o[3]);
  } else {
#pragma unroll
    for (int e = 0; e < 4; e++)
      if (k + e < K) row[k + e] = o[e];
  }
}

__device__ __forceinline__ uint32_t bf16_pair(float lo, float hi) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&p);
}
template <bool VEC>
__device__ __forceinline__ void store4(__nv_bfloat16* row, int64_t k, int64_t K, const float (&o)[4]) {
  if (VEC && k + 4 <= K) {
    *reinterpret_cast<uint2*>(row + k) = make_uint2(bf16_pair(o[0], o[1]), bf16_pair(o[2], o[3]));
  } else {
#pragma unroll
    for (int e = 0; e < 4; e++)
      if (k + e < K) row[k + e] = __float2bfloat16_rn(o[e]);
  }
}

}  // namespace rowio
}  // namespace hbmm
