// Pieces shared by the workspace-free contractions: scales of consecutive segments of a row, and the counts of all
// sub-word segments of a word at once.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace hbmm {
namespace popc {

__device__ __forceinline__ float load_scale(const void* s, int bf16, int64_t idx) {
  if (bf16) return __uint_as_float(static_cast<uint32_t>(__ldg(reinterpret_cast<const unsigned short*>(s) + idx)) << 16);
  return __ldg(reinterpret_cast<const float*>(s) + idx);
}

// The scales of SPC consecutive segments of one row from segment s0 on; 0 past the last group.  One group per segment,
// in order: 16-byte loads of fp32 scales, 4-byte loads of bf16 pairs (s0 is a multiple of SPC, rows are 16-byte vectors);
// otherwise one load per segment.
template <int SPC>
__device__ __forceinline__ void load_scales(const void* s, int bf16, int64_t row_off, int64_t s0, int64_t r, int64_t G, bool in, float (&v)[SPC]) {
#pragma unroll
  for (int i = 0; i < SPC; i++) v[i] = 0.0f;
  if (!in) return;
  if (SPC >= 4 && r == 1 && !bf16) {
#pragma unroll
    for (int q = 0; q < SPC / 4; q++)
      if (s0 + 4 * q < G) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(s) + row_off + s0 + 4 * q));
        v[(4 * q) % SPC] = x.x;
        if (s0 + 4 * q + 1 < G) v[(4 * q + 1) % SPC] = x.y;
        if (s0 + 4 * q + 2 < G) v[(4 * q + 2) % SPC] = x.z;
        if (s0 + 4 * q + 3 < G) v[(4 * q + 3) % SPC] = x.w;
      }
    return;
  }
  if (SPC == 2 && r == 1 && !bf16) {
    if (s0 < G) {
      const float2 x = __ldg(reinterpret_cast<const float2*>(reinterpret_cast<const float*>(s) + row_off + s0));
      v[0] = x.x;
      if (s0 + 1 < G) v[SPC - 1] = x.y;
    }
    return;
  }
  if (SPC >= 2 && r == 1 && bf16) {
#pragma unroll
    for (int q = 0; q < SPC / 2; q++)
      if (s0 + 2 * q < G) {
        const uint32_t x = __ldg(reinterpret_cast<const uint32_t*>(reinterpret_cast<const unsigned short*>(s) + row_off + s0 + 2 * q));
        v[(2 * q) % SPC] = __uint_as_float(x << 16);
        if (s0 + 2 * q + 1 < G) v[(2 * q + 1) % SPC] = __uint_as_float(x & 0xFFFF0000u);
      }
    return;
  }
  int64_t g = s0, rem = 0;
  if (r != 1) { g = s0 / r; rem = s0 - g * r; }
#pragma unroll
  for (int i = 0; i < SPC; i++) {
    if (g < G) v[i] = load_scale(s, bf16, row_off + g);
    if (++rem >= r) { rem = 0; g++; }
  }
}

// Doubled counts of a word's segments p, p + PARTS, p + 2 PARTS, .. (PARTS = 8 / SEG) as the four bytes of a word: the
// fields of the part are brought one bit above the bottom of their bytes by a rotation.
template <int SEG>
__device__ __forceinline__ uint32_t doubled_counts(uint32_t x, int p) {
  const uint32_t c2 = x - ((x >> 1) & 0x55555555u);
  if constexpr (SEG == 2) return __funnelshift_r(c2, c2, 2 * p + 31) & 0x06060606u;
  const uint32_t c4 = (c2 & 0x33333333u) + ((c2 >> 2) & 0x33333333u);
  if constexpr (SEG == 4) return __funnelshift_r(c4, c4, 4 * p + 31) & 0x0E0E0E0Eu;
  return ((c4 << 1) & 0x0E0E0E0Eu) + ((c4 >> 3) & 0x0E0E0E0Eu);
}

}  // namespace popc
}  // namespace hbmm
