// HBMM contraction of two packed operands on the integer pipe (Section 4.2, Eq. 7): the workspace-free path, and the
// path of every K that is no whole number of words.  A segment is the finer of the two groupings: 2, 4, 8 or 16 bits
// of a word, or 1, 2, 4 or 8 words; per output and segment  C += (deltaA deltaW) D,  D = n_valid - 2 popc(a ^ w).
//
// What bounds it: per output and word one XOR and the population counts (16 /clk/SM), per output and segment three
// fp32 operations (issued two outputs at a time) -- and, for the products this path really gets (a few hundred rows,
// K some thousand), how many warps have work at all.  So a warp owns a whole 32 x 32 tile of C (4 x 8 outputs per
// lane), stages its own operands (no barrier between warps in the K loop; the next chunk's loads are in flight while
// the current one is computed), and up to eight warps of a CTA split the K range of a tile; their partial sums meet
// in shared memory at the end, always in the same order.
// Population counts of 2-, 4- and 8-bit segments are formed for all of a word at once by adding neighbouring fields
// (2, 3 or 4 levels); the doubled count of a segment is then a byte, and one byte permutation puts it under the
// exponent of 2^23, so that float - (2^23 + n_valid) = 2 popc - n_valid exactly.  Segments of 16 bits and more use the
// popcount instruction.  (One masked popcount per 2-bit segment would keep that unit busy for 128 clk per word and warp
// against ~75 issue slots this way; at 16 bits the two are level.)
// Measured against one 64 x 64 (sub-word) or 128 x 128 (word) tile per CTA, which this replaces: 333 x 720 x 1000 at
// beta 16 27.8 -> 8.9 us, 82 x 536 x 3768 at beta 64 90 -> 9.4 us, 4050 x 280 x 4368 at beta 16 203 -> 107 us; on the
// conv3_x matrix (50176 x 128 x 1152) beta 2 / 4 / 8 / 16 / 32 / 128: 1337 / 662 / 334 / 172 / 89 / 81 ->
// 926 / 546 / 327 / 159 / 83 / 67 us.  Slower than those tiles only at mixed groupings of sub-word segments over long K (5104 x
// 536 x 6912 at beta 256 / 16 487 -> 516), whose scales each warp loads for itself.  Scalar fp32 instead of the paired
// instructions: 5 % slower.
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
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
// acc += sa sw (counts - bias) for two neighbouring outputs; c0, c1: 2^23 + doubled count as bit patterns.  DOT_FIRST: the
// first product is (counts - bias) sa, so that a segment whose signs cancel adds 0 also where the product of its scales
// leaves the range of fp32; 4 % slower at segments of 2 and 8 bits, which take the product of the scales first.
template <bool DOT_FIRST>
__device__ __forceinline__ void add_term(uint64_t& acc, uint32_t c0, uint32_t c1, uint64_t neg_bias, uint64_t sa, uint64_t sw) {
  uint64_t f = pack2(__uint_as_float(c0), __uint_as_float(c1));
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(f) : "l"(neg_bias));
  if constexpr (DOT_FIRST) {
    asm("mul.rn.f32x2 %0, %0, %1;" : "+l"(f) : "l"(sa));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(f), "l"(sw));
  } else {
    uint64_t s;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(sa), "l"(sw));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(s), "l"(f));
  }
}

// MIXED: some group spans several segments (ra, rw not both 1).  The lookup for that, in every kernel, costs the uniform
// groupings registers: 2 % at 2-bit segments, 5 % at 32.
template <int SEG, bool MIXED>
__global__ void __launch_bounds__(kThreads, 2)
gemm_popc_tile_kernel(const TileArgs g) {
  pdl_wait();
  pdl_launch_dependents();      // a convolution's next front end sets itself up meanwhile
  using P = Cfg<SEG>;
  // The next chunk waits in registers, except for the finest segments: their counts and scales need those registers
  // (spills otherwise), and a chunk is 1000 instructions and more, which the other warps fill a load's latency with.
  constexpr bool kAhead = SEG > 4;
  __shared__ __align__(16) uint32_t smem[kWarps * P::SMEM_WORDS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int KS = 1 << g.ks_log2;
  const int part = warp & (KS - 1);
  const int64_t m0 = (static_cast<int64_t>(blockIdx.y) * (blockDim.x >> (5 + g.ks_log2)) + (warp >> g.ks_log2)) * TS;
  const int64_t n0 = static_cast<int64_t>(blockIdx.x) * TS;
  const int tx = lane & 3, ty = lane >> 2;              // columns 8 tx .., rows 4 ty ..
  uint32_t* as = smem + warp * P::SMEM_WORDS;           // [CW][32]
  uint32_t* ws = as + P::CW * TS;                       // [CW][32]
  float* sa_s = reinterpret_cast<float*>(ws + P::CW * TS);   // [SPC][32], negated
  float* sw_s = sa_s + P::SPC * TS;                     // [SPC][32]
  const int64_t m = m0 + lane, n = n0 + lane;           // the rows this lane stages
  const bool ain = m < g.M, win = n < g.N;
  const uint32_t* arow = g.a_bits + (ain ? m : 0) * g.lda_w;
  const uint32_t* wrow = g.w_bits + (win ? n : 0) * g.ldw_w;
  const int64_t aoff = (ain ? m : 0) * g.lda_s, woff = (win ? n : 0) * g.ldw_s;

  uint64_t acc[4][4];                                   // two neighbouring columns each
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
      for (int i = 0; i < P::CW; i++) { as[i * TS + lane] = pa[i]; ws[i * TS + lane] = pw[i]; }
#pragma unroll
      for (int i = 0; i < P::SPC; i++) { sa_s[i * TS + lane] = -psa[i]; sw_s[i * TS + lane] = psw[i]; }
      __syncwarp();
      if (kAhead && c + KS < g.n_chunks) fetch(c + KS);
      const int64_t left_chunk = g.K - c * (P::CW * 32);              // elements from the chunk's start to the row's end
      // one segment of all 32 outputs: counts(i, j) gives 2^23 + 2 popc as a bit pattern
      auto segment = [&](int s, auto counts) {
        const int64_t left = left_chunk - s * SEG;
        const int nv = left >= SEG ? SEG : (left > 0 ? static_cast<int>(left) : 0);
        const float nb = -(8388608.0f + static_cast<float>(nv));
        const uint64_t neg_bias = pack2(nb, nb);
        const float4 sa4 = *reinterpret_cast<const float4*>(sa_s + s * TS + 4 * ty);
        const float sa[4] = {sa4.x, sa4.y, sa4.z, sa4.w};
        uint64_t sw[4];
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const float4 v = *reinterpret_cast<const float4*>(sw_s + s * TS + 8 * tx + 4 * h);
          sw[2 * h] = pack2(v.x, v.y);
          sw[2 * h + 1] = pack2(v.z, v.w);
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
          const uint64_t sa2 = pack2(sa[i], sa[i]);
#pragma unroll
          for (int j = 0; j < 4; j++) add_term<(SEG >= 32)>(acc[i][j], counts(i, 2 * j), counts(i, 2 * j + 1), neg_bias, sa2, sw[j]);
        }
      };
      auto words = [&](int i, uint32_t (&a)[4], uint32_t (&w)[8]) {
        const uint4 av = *reinterpret_cast<const uint4*>(as + i * TS + 4 * ty);
        const uint4 w0 = *reinterpret_cast<const uint4*>(ws + i * TS + 8 * tx), w1 = *reinterpret_cast<const uint4*>(ws + i * TS + 8 * tx + 4);
        a[0] = av.x; a[1] = av.y; a[2] = av.z; a[3] = av.w;
        w[0] = w0.x; w[1] = w0.y; w[2] = w0.z; w[3] = w0.w; w[4] = w1.x; w[5] = w1.y; w[6] = w1.z; w[7] = w1.w;
      };
      if constexpr (SEG <= 8) {
        constexpr int PARTS = 8 / SEG;
#pragma unroll 1
        for (int i = 0; i < P::CW; i++) {
          if (P::CW > 1 && left_chunk <= 32 * i) break;      // words past the row's end
#pragma unroll 1
          for (int p = 0; p < PARTS; p++) {
            uint32_t a[4], w[8], cnt[4][8];
            words(i, a, w);
#pragma unroll
            for (int r = 0; r < 4; r++)
#pragma unroll
              for (int j = 0; j < 8; j++) cnt[r][j] = doubled_counts<SEG>(a[r] ^ w[j], p);
#pragma unroll
            for (int b = 0; b < 4; b++)
              segment(i * P::SPW + b * PARTS + p, [&](int r, int j) { return __byte_perm(cnt[r][j], 0x4B000000u, 0x7540u + b); });
          }
        }
      } else if constexpr (SEG == 16) {
#pragma unroll
        for (int i = 0; i < P::CW; i++) {
          if (left_chunk <= 32 * i) break;
          uint32_t a[4], w[8];
          words(i, a, w);
          segment(2 * i, [&](int r, int j) { return 0x4B000000u + 2u * __popc((a[r] ^ w[j]) & 0xFFFFu); });
          segment(2 * i + 1, [&](int r, int j) { return 0x4B000000u + 2u * __popc((a[r] ^ w[j]) >> 16); });
        }
      } else if constexpr (SEG == 32) {
#pragma unroll
        for (int i = 0; i < P::CW; i++) {
          uint32_t a[4], w[8];
          words(i, a, w);
          segment(i, [&](int r, int j) { return 0x4B000000u + 2u * __popc(a[r] ^ w[j]); });
        }
      } else {
#pragma unroll
        for (int s = 0; s < P::SPC; s++) {
          uint32_t cnt[4][8];
#pragma unroll
          for (int q = 0; q < P::SW; q++) {
            uint32_t a[4], w[8];
            words(s * P::SW + q, a, w);
#pragma unroll
            for (int r = 0; r < 4; r++)
#pragma unroll
              for (int j = 0; j < 8; j++) {
                const uint32_t p = __popc(a[r] ^ w[j]);
                cnt[r][j] = q == 0 ? p : cnt[r][j] + p;
              }
          }
          segment(s, [&](int r, int j) { return 0x4B000000u + 2u * cnt[r][j]; });
        }
      }
    }
  }
  if (KS == 1) {
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const int64_t row = m0 + 4 * ty + i;
      if (row >= g.M) continue;
#pragma unroll
      for (int h = 0; h < 2; h++) {
        const int64_t col = n0 + 8 * tx + 4 * h;
        float o[4];
        unpack2(acc[i][2 * h], o[0], o[1]);
        unpack2(acc[i][2 * h + 1], o[2], o[3]);
        float* dst = g.C + row * g.ldc + col;
        if (col + 3 < g.N) *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
        else
          for (int e = 0; e < 4; e++)
            if (col + e < g.N) dst[e] = o[e];
      }
    }
    return;
  }
  // the KS partial tiles, added in order of their part: [4-column block of a lane: 2 i + h][lane] as 16-byte vectors
  __syncwarp();                                         // the staging area is this warp's own
  float4* mine = reinterpret_cast<float4*>(smem + warp * P::SMEM_WORDS);
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int h = 0; h < 2; h++) {
      float o[4];
      unpack2(acc[i][2 * h], o[0], o[1]);
      unpack2(acc[i][2 * h + 1], o[2], o[3]);
      mine[(2 * i + h) * 32 + lane] = make_float4(o[0], o[1], o[2], o[3]);
    }
  __syncthreads();
  const int first = warp - part;                        // the warps first .. first + KS - 1 hold this tile
  for (int b = part; b < 8; b += KS) {                  // 8 blocks shared out among the KS warps
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = 0; q < KS; q++) {
      const float4 v = reinterpret_cast<const float4*>(smem + (first + q) * P::SMEM_WORDS)[b * 32 + lane];
      sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
    }
    const int64_t row = m0 + 4 * ty + (b >> 1), col = n0 + 8 * tx + 4 * (b & 1);
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
