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

// A group sum as a mean, for the group that holds a lane's element e of four (the lane starts at k, k a multiple of four,
// groups of BETA from the row's start, the last one of its own length).  A whole group's length is a power of two: the
// product with its inverse is the quotient, bit for bit, and takes one instruction where the division takes a dozen.
template <int BETA>
__device__ __forceinline__ float group_mean(float sum, int64_t k, int e, int64_t K) {
  const int64_t left = K - (BETA >= 4 ? k / BETA * BETA : k + e / BETA * BETA);      // elements from the group's start on
  if (left >= BETA) return sum * (1.0f / static_cast<float>(BETA));
  return sum / static_cast<float>(left > 0 ? left : 1);
}

// Whether a warp per 128 elements of a row beats a thread per group.  Rows shorter than 64 leave more than half of its lanes
// idle, and a group of four is one 16-byte load for the thread that owns it, so that at beta 4 the warp has to be nearly
// full: backward of 85523 x 64, padded, at beta 4 16 us per group and 28 per warp, of 10302 x 1728 51 and 40.  Groups of
// eight that leave as bf16 want it well above half full: dense of 73938 x 64 15.4 and 17.6 us.
inline bool warp_per_run_pays(int64_t beta, int64_t K, bool half_out = false) {
  const int64_t lanes_for = (K + 127) / 128 * 128;
  if ((beta & (beta - 1)) != 0 || beta > 128 || K < 64) return false;
  return beta == 4 ? 5 * K >= 4 * lanes_for : beta != 8 || !half_out || 5 * K >= 3 * lanes_for;
}

}  // namespace rowio
}  // namespace hbmm
