// Pieces shared by the integer-pipe contractions: scales of consecutive segments of a row, and the counts of all
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

// s / r for segment numbers.  The 64-bit division is a noticeable part of a chunk's instructions (5104 x 536 x 6912 at beta
// 256 / 16 550 us with it, 520 with the 32-bit one); r is a power of two unless a group is three words or the like.
__device__ __forceinline__ int64_t div_segments(int64_t s, int64_t r) {
  if ((r & (r - 1)) == 0) return s >> (63 - __clzll(r));
  if (((s | r) >> 32) == 0) return static_cast<uint32_t>(s) / static_cast<uint32_t>(r);
  return s / r;
}

// The scales of SPC consecutive segments of one row from segment s0 on, r segments to a group; 0 past the last of the T
// segments.  One group per segment, in order: 16-byte loads of fp32 scales, 4-byte loads of bf16 pairs (s0 is a multiple of
// SPC, rows are 16-byte vectors); otherwise one load per segment, or one for all.
template <int SPC>
__device__ __forceinline__ void load_scales(const void* s, int bf16, int64_t row_off, int64_t s0, int64_t r, int64_t T, bool in, float (&v)[SPC]) {
#pragma unroll
  for (int i = 0; i < SPC; i++) v[i] = 0.0f;
  if (!in) return;
  if (SPC >= 4 && r == 1 && !bf16) {
#pragma unroll
    for (int q = 0; q < SPC / 4; q++)
      if (s0 + 4 * q < T) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(s) + row_off + s0 + 4 * q));
        v[(4 * q) % SPC] = x.x;
        if (s0 + 4 * q + 1 < T) v[(4 * q + 1) % SPC] = x.y;
        if (s0 + 4 * q + 2 < T) v[(4 * q + 2) % SPC] = x.z;
        if (s0 + 4 * q + 3 < T) v[(4 * q + 3) % SPC] = x.w;
      }
    return;
  }
  if (SPC == 2 && r == 1 && !bf16) {
    if (s0 < T) {
      const float2 x = __ldg(reinterpret_cast<const float2*>(reinterpret_cast<const float*>(s) + row_off + s0));
      v[0] = x.x;
      if (s0 + 1 < T) v[SPC - 1] = x.y;
    }
    return;
  }
  if (SPC >= 2 && r == 1 && bf16) {
#pragma unroll
    for (int q = 0; q < SPC / 2; q++)
      if (s0 + 2 * q < T) {
        const uint32_t x = __ldg(reinterpret_cast<const uint32_t*>(reinterpret_cast<const unsigned short*>(s) + row_off + s0 + 2 * q));
        v[(2 * q) % SPC] = __uint_as_float(x << 16);
        if (s0 + 2 * q + 1 < T) v[(2 * q + 1) % SPC] = __uint_as_float(x & 0xFFFF0000u);
      }
    return;
  }
  if (s0 >= T) return;
  if (r == 1) {
#pragma unroll
    for (int i = 0; i < SPC; i++)
      if (s0 + i < T) v[i] = load_scale(s, bf16, row_off + s0 + i);
    return;
  }
  if (r % SPC == 0 || SPC % r == 0) {          // whole groups, or all inside one: a load per group
    const int64_t g0 = div_segments(s0, r);
    const int mask = r < SPC ? static_cast<int>(r) - 1 : SPC - 1;
    int64_t g = row_off + g0;
    float x = 0.0f;
#pragma unroll
    for (int i = 0; i < SPC; i++) {
      if ((i & mask) == 0 && s0 + i < T) x = load_scale(s, bf16, g++);
      if (s0 + i < T) v[i] = x;
    }
    return;
  }
  int64_t g = div_segments(s0, r), rem = s0 - g * r;
#pragma unroll
  for (int i = 0; i < SPC; i++) {
    if (s0 + i < T) v[i] = load_scale(s, bf16, row_off + g);
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
