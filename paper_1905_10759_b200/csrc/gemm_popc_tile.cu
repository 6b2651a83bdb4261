// HBMM contraction of two packed operands by warp-level integer matrix instructions (Section 4.2, Eq. 7): the workspace-free
// path, and the path of every K that is no whole number of words.  A segment is the finer of the two groupings: 2, 4, 8 or 16
// bits of a word, or 1, 2, 4 or 8 words; per output and segment  C += (deltaA deltaW) D,  D the segment's dot of signs.
//
// The dots D of a word's segments are formed by mma.sync on bytes of +-64: exact integers, in the registers that scale them (a
// tcgen05 accumulator would have to come out of tensor memory once per segment), and, started from the bits of 1.5 2^23, already
// floats.  16 x 8 outputs over 32 elements cost 8.4 clk of a scheduler's tensor unit; the population counts they replace, at 16
// /clk/SM, 32 clk for whole words, and 75 issue slots for all of a word's segments of 2 to 8 bits.  Segments shorter than a word
// take one product each, the first operand zeroed outside the segment.  Which element sits at which K index of the instruction
// is free as long as both operands agree: byte j of register r of lane t of a quad holds bit 8 j + 2 t + r of the word, so that
// expanding a register is one shift and one three-input operation, and the segments of 16 and 8 bits are bytes, those of 4 and
// 2 bits bytes of some lanes.  (e4m3 bytes, whose products are fp32 by themselves, run at 0.8 of the rate of s8 and are
// converted on the way: 0.8 .. 1.0 of the counts' speed.)
// What bounds it: the loads of a warp's own operands and scales, the three fp32 operations per output and segment (issued two
// outputs at a time); and, for the products this path really gets (a few hundred rows, K some thousand), how many warps have
// work at all.  So a warp owns a whole 32 x 32 tile of C, stages its own operands (no barrier between warps in the K loop; the
// next chunk's loads are in flight while the current one is computed), and up to eight warps of a CTA split the K range of a
// tile; their partial sums meet in shared memory at the end, always in the same order.
// Against the same tiles on population counts, us: conv3_x matrix (50176 x 128 x 1152) at beta 2 / 4 / 8 / 16 / 32 / 64 / 128 / 256
// 923 / 544 / 325 / 158 / 82.6 / 74.8 / 66.7 / 72.4 -> 807 / 441 / 239 / 124 / 75.0 / 60.6 / 47.6 / 43.8; 333 x 720 x 1000 at beta
// 16 9.0 -> 7.8; 691 x 1216 x 5032 at beta 8 194 -> 146; 3325 x 872 x 2946 at beta 64 104 -> 86; 320 x 1480 x 8376 at beta 2 553 ->
// 483; 5104 x 536 x 6912 at beta 256 / 16 504 -> 426; 9 x 1000 x 4097 at beta 32 10.0 -> 9.8; 82 x 2880 x 152 at beta 32 / 64 3.4 /
// 3.5 -> 3.3 / 3.1; level or slower by 0.3 us where a warp has one chunk and the last one ends early (100 x 1000 x 500 at beta 32 3.1
// -> 3.4).
#include <type_traits>
#include "kernels.h"
#include "pdl.cuh"
#include "popc_common.cuh"

namespace hbmm {
namespace {

using namespace popc;

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int TS = 32;                 // tile side of a warp

struct TileArgs {
  const uint32_t* a_bits; const void* a_scales;
  const uint32_t* w_bits; const void* w_scales;
  float* C;
  int64_t M, N, K, lda_w, ldw_w, lda_s, ldw_s, ldc;
  int64_t ra, rw;              // segments per A group / per W group
  int64_t T;                   // segments per row
  int64_t n_words, n_chunks;
  int32_t a_bf16, w_bf16;
  int32_t ks_log2;             // warps that share a tile's K range: 1 << ks_log2
};

template <int SEG>
struct Cfg {
  static constexpr int SW = SEG >= 32 ? SEG / 32 : 1;                          // words per segment
  static constexpr int CW = SEG <= 4 ? 1 : (SEG == 8 ? 2 : (SEG == 256 ? 8 : 4));   // words per chunk
  static constexpr int SPC = CW * 32 / SEG;                                    // segments per chunk
  static constexpr int SPW = SEG < 32 ? 32 / SEG : 1;                          // segments per word
  static constexpr int WARP_WORDS = (2 * CW + 2 * SPC) * TS;                   // a warp's staging area
  static constexpr int SMEM_WORDS = WARP_WORDS > TS * TS ? WARP_WORDS : TS * TS;   // ... which its partial sums reuse
};

// s / r for segment numbers.  The 64-bit division is a noticeable part of a chunk's instructions (5104 x 536 x 6912 at beta
// 256 / 16 550 us with it, 516 without); r is a power of two unless a group is three words or the like.
__device__ __forceinline__ int64_t div_segments(int64_t s, int64_t r) {
  if ((r & (r - 1)) == 0) return s >> (63 - __clzll(r));
  if (((s | r) >> 32) == 0) return static_cast<uint32_t>(s) / static_cast<uint32_t>(r);
  return s / r;
}

// The scales of SPC consecutive segments of one row from segment s0 on, r segments to a group; 0 past the last of the T
// segments.  One group per segment, in order: 16-byte loads of fp32 scales, 4-byte loads of bf16 pairs (s0 is a multiple of
// SPC, rows are 16-byte vectors); otherwise one load per segment, or one for all.
template <int SPC>
__device__ __forceinline__ void chunk_scales(const void* s, int bf16, int64_t row_off, int64_t s0, int64_t r, int64_t T, bool in, float (&v)[SPC]) {
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

// The CW packed words of one row from word w0 on (rows are padded to a multiple of four words).
template <int CW>
__device__ __forceinline__ void load_words(const uint32_t* row, int64_t w0, int64_t ld, bool in, uint32_t (&v)[CW]) {
#pragma unroll
  for (int i = 0; i < CW; i++) v[i] = 0u;
  if (CW >= 4) {
#pragma unroll
    for (int q = 0; q < CW / 4; q++)
      if (in && w0 + 4 * q < ld) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(row + w0 + 4 * q));
        v[(4 * q) % CW] = x.x; v[(4 * q + 1) % CW] = x.y; v[(4 * q + 2) % CW] = x.z; v[(4 * q + 3) % CW] = x.w;
      }
  } else if (CW == 2) {
    if (in && w0 < ld) {
      const uint2 x = __ldg(reinterpret_cast<const uint2*>(row + w0));
      v[0] = x.x; v[CW - 1] = x.y;
    }
  } else {
    if (in && w0 < ld) v[0] = __ldg(row + w0);
  }
}

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
// acc += sa sw D for two neighbouring outputs.  DOT_FIRST: the first product is D sa, so that a segment whose signs cancel adds
// 0 also where the product of its scales leaves the range of fp32 (groups of whole words; shorter ones take the product of the
// scales first).
template <bool DOT_FIRST>
__device__ __forceinline__ void add_term(uint64_t& acc, uint32_t d0, uint32_t d1, uint64_t sa, uint64_t sw) {
  uint64_t f, d = pack2(__uint_as_float(d0), __uint_as_float(d1));
  const uint64_t unit = pack2(0x1p-12f, 0x1p-12f), bias = pack2(-3072.0f, -3072.0f);
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(d), "l"(unit), "l"(bias));      // the dot, exactly
  if constexpr (DOT_FIRST) {
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(f) : "l"(d), "l"(sa));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(f), "l"(sw));
  } else {
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(f) : "l"(sa), "l"(sw));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(f), "l"(d));
  }
}

// d = c + a b^T, 16 x 8 outputs over 32 elements of +-64: 4096 times the dot
__device__ __forceinline__ void mma_s8(uint32_t (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2], const uint32_t (&c)[4]) {
  asm("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %11, %12, %13};"
      : "=r"(d[0]), "=r"(d[1]), "=r"(d[2]), "=r"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "r"(c[0]), "r"(c[1]), "r"(c[2]), "r"(c[3]));
}
// Bits 8 j + b of a word (b = 7 - shift) as four bytes: 1 -> +64, 0 -> -64.
__device__ __forceinline__ uint32_t expand(uint32_t word, int shift) { return ((word << shift) & 0x80808080u) ^ 0xC0C0C0C0u; }
constexpr uint32_t kBias = 0x4B400000u;      // 1.5 2^23: an integer sum started from here is that float plus the sum

// MIXED: some group spans several segments (ra, rw not both 1).  The lookup for that, in every kernel, costs the uniform
// groupings registers: 2 % at 2-bit segments, 5 % at 32.
template <int SEG, bool MIXED>
__global__ void __launch_bounds__(kThreads, 2)
gemm_popc_tile_kernel(const TileArgs g) {
  pdl_wait();
  pdl_launch_dependents();      // a convolution's next front end sets itself up meanwhile
  using P = Cfg<SEG>;
  // The next chunk waits in registers, except for the finest segments, whose scales are 16 and 8 to a word and operand: at 2-bit
  // segments they do not fit (36 and 156 bytes of spills), and a chunk is 1000 instructions and more there, which the other
  // warps fill a load's latency with.
  constexpr bool kAhead = SEG > 4;
  __shared__ __align__(16) uint32_t smem[kWarps * P::SMEM_WORDS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KS = 1 << g.ks_log2;
  const int part = warp & (KS - 1);
  const int64_t m0 = (static_cast<int64_t>(blockIdx.y) * (blockDim.x >> (5 + g.ks_log2)) + (warp >> g.ks_log2)) * TS;
  const int64_t n0 = static_cast<int64_t>(blockIdx.x) * TS;
  const int qt = lane & 3, qg = lane >> 2;              // lane of its quad, quad: rows qg + 8 i, columns 8 j + 2 qt and the next
  // Whole-word segments: the rows are staged in the order a lane reads them in, as 16-byte pieces -- row 8 i + qg at 4 qg + i, the
  // scale of column 8 j + 2 qt + e at 8 qt + 2 j + e.  One by one they are 20 loads a segment, which bounded single words
  // (50176 x 128 x 1152 at beta 32 76.0 us so, 73.7 in pieces).  Shorter segments keep the row order: the pieces' registers cost
  // them 3 .. 8 %.
  constexpr bool VEC = SEG >= 32;
  const int row_at = VEC ? (lane & 7) * 4 + (lane >> 3) : lane, col_at = VEC ? ((lane >> 1) & 3) * 8 + (lane >> 3) * 2 + (lane & 1) : lane;
  uint32_t* as = smem + warp * P::SMEM_WORDS;           // [CW][32]
  uint32_t* ws = as + P::CW * TS;                       // [CW][32]
  float* sa_s = reinterpret_cast<float*>(ws + P::CW * TS);   // [SPC][32]
  float* sw_s = sa_s + P::SPC * TS;                     // [SPC][32]
  const int64_t m = m0 + lane, n = n0 + lane;           // the rows this lane stages
  const bool ain = m < g.M, win = n < g.N;
  const uint32_t* arow = g.a_bits + (ain ? m : 0) * g.lda_w;
  const uint32_t* wrow = g.w_bits + (win ? n : 0) * g.ldw_w;
  const int64_t aoff = (ain ? m : 0) * g.lda_s, woff = (win ? n : 0) * g.ldw_s;

  uint64_t acc[4][4];                                   // [8 rows apart][8 columns apart], two neighbouring columns each
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) acc[i][j] = 0ull;

  uint32_t pa[P::CW], pw[P::CW];
  float psa[P::SPC], psw[P::SPC];
  auto fetch = [&](int64_t c) {
    load_words<P::CW>(arow, c * P::CW, g.lda_w, ain, pa);
    load_words<P::CW>(wrow, c * P::CW, g.ldw_w, win, pw);
    if constexpr (MIXED) {
      chunk_scales<P::SPC>(g.a_scales, g.a_bf16, aoff, c * P::SPC, g.ra, g.T, ain, psa);
      chunk_scales<P::SPC>(g.w_scales, g.w_bf16, woff, c * P::SPC, g.rw, g.T, win, psw);
    } else {
      load_scales<P::SPC>(g.a_scales, g.a_bf16, aoff, c * P::SPC, 1, g.T, ain, psa);
      load_scales<P::SPC>(g.w_scales, g.w_bf16, woff, c * P::SPC, 1, g.T, win, psw);
    }
  };
  if (m0 < g.M && part < g.n_chunks) {                  // warp-uniform
    if (kAhead) fetch(part);
    for (int64_t c = part; c < g.n_chunks; c += KS) {
      if (!kAhead) fetch(c);
      __syncwarp();
#pragma unroll
      for (int i = 0; i < P::CW; i++) { as[i * TS + row_at] = pa[i]; ws[i * TS + row_at] = pw[i]; }
#pragma unroll
      for (int i = 0; i < P::SPC; i++) { sa_s[i * TS + row_at] = psa[i]; sw_s[i * TS + col_at] = psw[i]; }
      __syncwarp();
      if (kAhead && c + KS < g.n_chunks) fetch(c + KS);
      const int64_t left_chunk = g.K - c * (P::CW * 32);              // elements from the chunk's start to the row's end
      // the dots of one segment in 16 rows from 16 r on, d[column block of 8], into the sums
      auto segment = [&](int s, int r, const uint32_t (&d)[4][4]) {
        uint64_t sa[2], sw[4];
        if constexpr (VEC) {
          const float2 v = *reinterpret_cast<const float2*>(sa_s + s * TS + 4 * qg + 2 * r);
          sa[0] = pack2(v.x, v.x);
          sa[1] = pack2(v.y, v.y);
#pragma unroll
          for (int h = 0; h < 2; h++) {
            const float4 u = *reinterpret_cast<const float4*>(sw_s + s * TS + 8 * qt + 4 * h);
            sw[2 * h] = pack2(u.x, u.y);
            sw[2 * h + 1] = pack2(u.z, u.w);
          }
        } else {
#pragma unroll
          for (int i = 0; i < 2; i++) {
            const float v = sa_s[s * TS + 16 * r + 8 * i + qg];
            sa[i] = pack2(v, v);
          }
#pragma unroll
          for (int j = 0; j < 4; j++) {
            const float2 u = *reinterpret_cast<const float2*>(sw_s + s * TS + 8 * j + 2 * qt);
            sw[j] = pack2(u.x, u.y);
          }
        }
#pragma unroll
        for (int i = 0; i < 2; i++)
#pragma unroll
          for (int j = 0; j < 4; j++) add_term<(SEG >= 32)>(acc[2 * r + i][j], d[j][2 * i], d[j][2 * i + 1], sa[i], sw[j]);
      };
      // word i of the chunk as operand registers; elements past the row's end are 0 in the first operand
      auto words = [&](int i, uint32_t (&a)[2][4], uint32_t (&w)[4][2], auto whole) {
        const int s0 = 7 - 2 * qt, s1 = s0 - 1;
        uint32_t av[4], wv[4];
        if constexpr (VEC) {
          const uint4 a4 = *reinterpret_cast<const uint4*>(as + i * TS + 4 * qg), w4 = *reinterpret_cast<const uint4*>(ws + i * TS + 4 * qg);
          av[0] = a4.x; av[1] = a4.y; av[2] = a4.z; av[3] = a4.w;
          wv[0] = w4.x; wv[1] = w4.y; wv[2] = w4.z; wv[3] = w4.w;
        } else {
#pragma unroll
          for (int r = 0; r < 4; r++) { av[r] = as[i * TS + 8 * r + qg]; wv[r] = ws[i * TS + 8 * r + qg]; }
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
          a[r >> 1][r & 1] = expand(av[r], s0);
          a[r >> 1][2 + (r & 1)] = expand(av[r], s1);
          w[r][0] = expand(wv[r], s0);
          w[r][1] = expand(wv[r], s1);
        }
        const int64_t left = left_chunk - 32 * i;
        if (!decltype(whole)::value && left < 32) {
          uint32_t k0 = 0u, k1 = 0u;
#pragma unroll
          for (int j = 0; j < 4; j++) {
            if (8 * j + 2 * qt < left) k0 |= 0xFFu << (8 * j);
            if (8 * j + 2 * qt + 1 < left) k1 |= 0xFFu << (8 * j);
          }
#pragma unroll
          for (int r = 0; r < 2; r++) { a[r][0] &= k0; a[r][1] &= k0; a[r][2] &= k1; a[r][3] &= k1; }
        }
      };
      const uint32_t bias[4] = {kBias, kBias, kBias, kBias};
      if constexpr (SEG < 32) {
#pragma unroll 1
        for (int i = 0; i < P::CW; i++) {
          if (P::CW > 1 && left_chunk <= 32 * i) break;      // words past the row's end
          uint32_t a[2][4], w[4][2];
          words(i, a, w, std::false_type{});
          constexpr int PER_BYTE = SEG < 8 ? 8 / SEG : 1, BYTES = SEG < 8 ? 1 : SEG / 8;     // segments of a byte, bytes of a segment
#pragma unroll 2
          for (int s = 0; s < P::SPW; s++) {
            const uint32_t bytes = (BYTES == 2 ? 0xFFFFu : 0xFFu) << (8 * BYTES * (s / PER_BYTE));
            const uint32_t keep = PER_BYTE == 1 || qt / (4 / PER_BYTE) == s % PER_BYTE ? bytes : 0u;
#pragma unroll
            for (int r = 0; r < 2; r++) {
              const uint32_t part[4] = {a[r][0] & keep, a[r][1] & keep, a[r][2] & keep, a[r][3] & keep};
              uint32_t d[4][4];
#pragma unroll
              for (int j = 0; j < 4; j++) mma_s8(d[j], part, w[j], bias);
              segment(i * P::SPW + s, r, d);
            }
          }
        }
      } else {
        // whole: nothing of the chunk lies past the row's end.  Without tests between them its segments overlap, where a loop
        // waited at each for the products of the last (50176 x 128 x 1152 at beta 32 82.8 -> 76.0 us, at 256 47.0 -> 43.8).
        auto one = [&](int s, auto whole) {
          constexpr bool WHOLE = decltype(whole)::value;
          uint32_t d[2][4][4];
#pragma unroll
          for (int q = 0; q < P::SW; q++) {
            if (!WHOLE && P::SW > 1 && left_chunk <= 32 * (s * P::SW + q)) break;
            uint32_t a[2][4], w[4][2];
            words(s * P::SW + q, a, w, whole);
#pragma unroll
            for (int r = 0; r < 2; r++)
#pragma unroll
              for (int j = 0; j < 4; j++) {
                if (q == 0) mma_s8(d[r][j], a[r], w[j], bias);
                else mma_s8(d[r][j], a[r], w[j], d[r][j]);
              }
          }
          segment(s, 0, d[0]);
          segment(s, 1, d[1]);
        };
        if (left_chunk >= P::CW * 32) {
#pragma unroll
          for (int s = 0; s < P::SPC; s++) one(s, std::true_type{});
        } else {
#pragma unroll 2
          for (int s = 0; s < P::SPC; s++) {
            if (left_chunk <= s * SEG) break;
            one(s, std::false_type{});
          }
        }
      }
    }
  }
  // The warp's tile (the staging area is its own) row by row, the 16-byte pieces of a row permuted by its number, so that both
  // the pairs of columns that come and the pieces that leave are spread over the banks; the KS partial tiles are added in
  // order of their part, four rows a turn, and leave as whole rows.  (As pairs of columns out of the registers' order, sixteen
  // turns: 82 x 2880 x 152 at beta 64 3.9 us, 3.4 so; 5184 x 448 x 640 16.9, 15.9.)
  __syncwarp();
  float* mine = reinterpret_cast<float*>(smem + warp * P::SMEM_WORDS);
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++)
      *reinterpret_cast<uint64_t*>(mine + (8 * i + qg) * TS + (((2 * j + (qt >> 1)) ^ qg) << 2) + 2 * (qt & 1)) = acc[i][j];
  if (KS == 1) __syncwarp();
  else __syncthreads();
  const int first = warp - part;                        // the warps first .. first + KS - 1 hold this tile
#pragma unroll 2
  for (int b = part; b < 8; b += KS) {                  // the rows shared out among the KS warps
    const int r = 4 * b + (lane >> 3);
    const int at = r * TS + (((lane & 7) ^ (r & 7)) << 2);
    float4 sum = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(smem + first * P::SMEM_WORDS) + at);
    for (int q = 1; q < KS; q++) {
      const float4 v = *reinterpret_cast<const float4*>(reinterpret_cast<const float*>(smem + (first + q) * P::SMEM_WORDS) + at);
      sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
    }
    const int64_t row = m0 + r, col = n0 + 4 * (lane & 7);
    if (row >= g.M) continue;
    float* dst = g.C + row * g.ldc + col;
    const float o[4] = {sum.x, sum.y, sum.z, sum.w};
    if (col + 3 < g.N) *reinterpret_cast<float4*>(dst) = sum;
    else
      for (int e = 0; e < 4; e++)
        if (col + e < g.N) dst[e] = o[e];
  }
}

template <int SEG>
cudaError_t launch_seg(TileArgs g, int sms, cudaStream_t stream) {
  g.n_chunks = (g.n_words + Cfg<SEG>::CW - 1) / Cfg<SEG>::CW;
  // sixteen warps per SM (two CTAs): split K until the machine has them, as long as every part has a chunk
  const int64_t tiles_m = (g.M + TS - 1) / TS, tiles_n = (g.N + TS - 1) / TS, want = static_cast<int64_t>(sms) * 16;
  g.ks_log2 = 0;
  while (g.ks_log2 < 3 && (tiles_m * tiles_n << g.ks_log2) < want && (2ll << g.ks_log2) <= g.n_chunks) g.ks_log2++;
  // short rows leave whole tiles to a warp; where eight of them to a CTA leave SMs without one, fewer
  int warps = kWarps;
  while (warps > (1 << g.ks_log2) && tiles_n * ((tiles_m * (1 << g.ks_log2) + warps - 1) / warps) < 2 * sms) warps /= 2;
  const int64_t per_cta = warps >> g.ks_log2;
  const dim3 grid(static_cast<unsigned>(tiles_n), static_cast<unsigned>((tiles_m + per_cta - 1) / per_cta));
  if (g.ra == 1 && g.rw == 1) launch_pdl(gemm_popc_tile_kernel<SEG, false>, dim3(grid), dim3(warps * 32), 0, stream, g);
  else launch_pdl(gemm_popc_tile_kernel<SEG, true>, dim3(grid), dim3(warps * 32), 0, stream, g);
  return cudaGetLastError();
}

// Bits per segment (the finer grouping; a single group per row takes the other operand's), 0: not this kernel's.
int segment_bits(const PackedView& A, const PackedView& W) {
  const int64_t a = A.beta >= A.K ? A.K : A.beta, w = W.beta >= W.K ? W.K : W.beta;
  int64_t seg = a < w ? a : w;
  if (seg >= A.K) seg = (A.K + 31) / 32 * 32;           // one group per row in both: one segment
  switch (seg) {
    case 2: case 4: case 8: case 16: case 32: case 64: case 128: case 256: return static_cast<int>(seg);
    default: return 0;
  }
}

}  // namespace

bool gemm_popc_tile_supported(const PackedView& A, const PackedView& W) { return segment_bits(A, W) != 0; }

cudaError_t launch_gemm_popc_tile(const PackedView& A, const PackedView& W, float* C, int64_t ldc, cudaStream_t stream) {
  TileArgs g{};
  g.a_bits = A.bits; g.a_scales = A.scales; g.w_bits = W.bits; g.w_scales = W.scales; g.C = C;
  g.M = A.rows; g.N = W.rows; g.K = A.K;
  g.lda_w = A.ld_words; g.ldw_w = W.ld_words; g.lda_s = A.ld_scales; g.ldw_s = W.ld_scales; g.ldc = ldc;
  g.a_bf16 = A.scale_bf16; g.w_bf16 = W.scale_bf16;
  const int seg = segment_bits(A, W);
  const int64_t T = (A.K + seg - 1) / seg;
  g.ra = A.beta >= A.K ? T : A.beta / seg;
  g.rw = W.beta >= W.K ? T : W.beta / seg;
  g.T = T;
  g.n_words = (A.K + 31) / 32;
  int dev = 0, sms = 0;
  if (current_device(&dev, &sms) != cudaSuccess) return cudaErrorInvalidDevice;
  switch (seg) {
    case 2: return launch_seg<2>(g, sms, stream);
    case 4: return launch_seg<4>(g, sms, stream);
    case 8: return launch_seg<8>(g, sms, stream);
    case 16: return launch_seg<16>(g, sms, stream);
    case 32: return launch_seg<32>(g, sms, stream);
    case 64: return launch_seg<64>(g, sms, stream);
    case 128: return launch_seg<128>(g, sms, stream);
    case 256: return launch_seg<256>(g, sms, stream);
    default: return cudaErrorNotSupported;
  }
}

}  // namespace hbmm
