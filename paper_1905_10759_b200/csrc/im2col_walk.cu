// Packed convolution front end for 3 x 3 filters at stride 1: every element of the image is read once per output row
// segment and shared by the taps it is part of, instead of being gathered again for each of them.
//
// A lane owns an input column of one image (neighbouring lanes neighbouring columns) and CH channels of it, and walks down the
// rows.  Per row it forms
//   signs: the channels' sign bits, with the neighbouring columns' (shuffles of a 32-bit word) spread to the nine-bit spacing
//          the row of K has (k = (c, i, j), nine taps per channel): four channels x three columns at a time, by replicating a
//          nibble over four bytes and keeping one bit of each;
//   sums:  |x| added over the channels whose nine taps all fall into one scale group, once per column, then over the three
//          columns (two shuffles per group instead of nine loads per channel); a channel that a group boundary cuts keeps
//          its three columns apart where the cut is.
// The output row whose window ends there then needs only its three input rows' words OR-ed and sums added: the rows' words, and
// the sums of the output rows under way, stay in registers.  Finished words and means go through shared memory (two buffers,
// one barrier per row) and leave as 16-byte pieces of consecutive words; the next row's loads are in flight meanwhile.
//
// Lanes: an image row is cut into strips of Pw output columns; a strip takes Pw + 2 lanes, a warp as many (image, row
// segment, strip) triples as fit.  The input needs no particular width, alignment or type: plain loads,
// consecutive lanes on consecutive columns.
//
// What bounds it: the load / shuffle / shared-memory pipe (some 120 instructions per row of 32 channels, against 290 gathered
// loads), then memory.  Against the staged tiles and the gathers it replaces, beta 32 unless said, us: 64 x 64 x 56 x 56
// 48.1 -> 22.6 (bf16 119 -> 23.6); 64 x 128 x 28 x 28 29.3 -> 14.2, at beta 16 / 8 / 4 / 2 42.9 / 46.3 / 63.4 / 90.3 -> 15.5 /
// 18.8 / 27.5 / 40.3; 64 x 256 x 14 x 14 17.5 -> 9.5; 20 x 192 x 55 x 55 at beta 2 434 -> 75; 16 x 100 x 27 x 27 bf16 at beta 16
// 26.4 -> 7.5; one image of 512 x 7 x 7 4.1 -> 3.5.  The same at stride 2, two columns per lane, was level with the staged tiles
// (32 x 64 x 56 x 56 12.0 against 12.3, one image of 512 x 7 x 7 3.5 against 5.5) and is not built.
#include <cuda_bf16.h>
#include "kernels.h"
#include "gemm_umma_prep.cuh"
#include "gemm_fold_prep.cuh"
#include "pdl.cuh"

namespace hbmm {
namespace {

constexpr int kMaxWarps = 8;
// Warps an SM holds at once (128 registers a thread).  A row takes a warp the same time whether 8 or 16 of them are there
// (64 x 64 x 56 x 56: 40.3 us in segments of 14 rows, 8 warps per SM; 22.6 in segments of 7), so time goes in turns of 16.
constexpr int kWarpsAtOnce = 16;

// Channels a lane holds: a whole chunk of 32 where its groups are those of whole words (nine), else as few as leave whole bytes
// of packed words (8 channels = 72 bits) and two groups per channel or fewer.  At beta 16, 32 / 16 channels, us: 64 x 128 x 28 x
// 28 20.2 / 15.5, 64 x 64 x 56 x 56 35.5 / 27.8, 8 x 48 x 16 x 16 6.9 / 3.5, one image of 512 x 7 x 7 5.5 / 3.7.
__host__ __device__ constexpr int channels_for(int beta) { return beta >= 32 ? 32 : (beta >= 8 ? 16 : 8); }

struct FastDiv {
  uint32_t d, magic;             // quotients of numbers below 2^16 by d below 2^16
  static FastDiv make(uint32_t d) { return FastDiv{d, d <= 1 ? 0u : static_cast<uint32_t>(((uint64_t{1} << 32) + d - 1) / d)}; }
  __device__ __forceinline__ uint32_t div(uint32_t n) const { return magic == 0 ? n : __umulhi(n, magic); }
};

struct WalkPlan {
  int32_t strips, Pw, P, L;      // strips per row, their output columns and lanes, strips per warp
  int32_t R, nseg;               // output rows of a segment, segments per image
  int32_t n_units;               // B * nseg * strips
  int32_t pieces, ranges;        // pieces of CH channels per CTA, channel ranges
  int32_t sets;                  // warps = sets * pieces
  int32_t slots;                 // output columns of a CTA: sets * L * Pw
  int32_t ldb, lds;              // pitch of the staged words and sums (32-bit units)
  int32_t words, groups;         // packed words and scales a range other than the last leaves per output column
  int32_t max_words, max_groups; // ... and the most of any range, the row's padding included
  int32_t gw;                    // words per scale group (1 up to beta = 32)
  int32_t vec_bits, vec_scales;  // every range's words / scales are whole 16-byte pieces
};
inline size_t walk_smem_bytes(const WalkPlan& p) { return static_cast<size_t>(p.slots) * 8 + 2 * static_cast<size_t>(p.slots) * (p.ldb + p.lds) * 4; }

__device__ __forceinline__ void store_one(void* scales, int bf16, int64_t idx, float v) {
  if (bf16) reinterpret_cast<__nv_bfloat16*>(scales)[idx] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(scales)[idx] = v;
}

// Scale group of tap t of channel c of a unit of BETA channels (9 BETA elements: nine groups).
template <int BETA>
struct Cut {
  __host__ __device__ static constexpr int group(int c, int t) { return (9 * c + t) / BETA; }
  __host__ __device__ static constexpr bool whole(int c) { return group(c, 0) == group(c, 8); }
};

// LIVE: no channel beyond it in any lane.  An image of fewer channels than a lane holds spent the time of a full chunk on them,
// more than the tiles and gathers before it.  Those / all channels / LIVE of them, us: 8 x 8 x 56 x 56 at beta 32 4.6 / 7.4 /
// 3.1, 33 x 20 x 28 x 28 at beta 96 7.5 / 8.9 / 7.2, 64 x 16 x 7 x 7 bf16 at beta 16 7.8 / 9.8 / 3.5.
template <int BETA, int LIVE, typename T>
__global__ void __launch_bounds__(kMaxWarps * 32, 2)
im2col_walk_kernel(const T* __restrict__ x, const ConvGeom g, const WalkPlan p, const FastDiv by_bits, const FastDiv by_scales,
                   const __grid_constant__ UmmaPrepJob prep, int n_prep, uint32_t* __restrict__ bits, int64_t ld_words,
                   void* __restrict__ scales, int64_t ld_scales, int scale_bf16) {
  constexpr int CH = channels_for(BETA), UNITS = CH / BETA, G = 9 * UNITS, Q = CH / 4;
  using C = Cut<BETA>;
  pdl_launch_dependents();
  if (static_cast<int>(blockIdx.x) < n_prep) {      // the weight operand of the contraction that follows: one task per CTA
    pdl_wait();
    const int st = blockIdx.x % prep.n_stages, tile_n = blockIdx.x / prep.n_stages;
    if (prep.tn == 64) { if (threadIdx.x < 64) fold::prepare_w_task<64>(prep.f, prep.out, prep.out_down, st, tile_n, threadIdx.x); }
    else if (threadIdx.x < 128) fold::prepare_w_task<128>(prep.f, prep.out, prep.out_down, st, tile_n, threadIdx.x);
    return;
  }
  extern __shared__ __align__(16) uint32_t walk_smem[];
  const int cta = blockIdx.x - n_prep;
  const int range = cta % p.ranges, first_unit = cta / p.ranges * (p.sets * p.L);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int piece = warp % p.pieces, set = warp / p.pieces;
  const int gl = lane / p.P, xl = lane - gl * p.P;
  const int unit = first_unit + set * p.L + gl;
  const bool active = gl < p.L && unit < p.n_units;
  const int strip = unit % p.strips, rest = unit / p.strips, seg = rest % p.nseg, b = rest / p.nseg;
  const int y0 = seg * p.R;
  // the lane's column is the middle one of its output column's three; the first and last lanes of a strip only lend theirs
  const int xo = strip * p.Pw + xl - 1, xin = xo + 1 - g.pw;
  const bool col_ok = active && xin >= 0 && xin < g.W;
  const int slot = (set * p.L + gl) * p.Pw + xl - 1;
  const bool out_ok = active && xl >= 1 && xl <= p.Pw && xo < g.Wo;
  const int c_first = (range * p.pieces + piece) * CH;
  const int nch = g.C - c_first < CH ? (g.C > c_first ? g.C - c_first : 0) : CH;

  const int buf_words = p.slots * (p.ldb + p.lds);
  int2* slot_at = reinterpret_cast<int2*>(walk_smem);                 // per output column: its first row's m, its rows
  uint32_t* stage0 = walk_smem + 2 * p.slots;
  for (int i = threadIdx.x; i < p.slots; i += blockDim.x) {
    const int u = first_unit + i / p.Pw, col = i % p.Pw;
    const int s = u % p.strips, r = u / p.strips, sg = r % p.nseg, bb = r / p.nseg;
    const int cx = s * p.Pw + col;
    int2 v = make_int2(0, 0);
    if (u < p.n_units && cx < g.Wo) {
      v.x = (bb * g.Ho + sg * p.R) * g.Wo + cx;
      v.y = g.Ho - sg * p.R < p.R ? g.Ho - sg * p.R : p.R;
    }
    slot_at[i] = v;
  }
  for (int i = threadIdx.x; i < 2 * buf_words; i += blockDim.x) stage0[i] = 0u;      // padding words and scales stay zero
  pdl_wait();

  const uint32_t plane = static_cast<uint32_t>(g.H) * static_cast<uint32_t>(g.W);
  const uint32_t plane_bytes = plane * static_cast<uint32_t>(sizeof(T));
  // byte offset of (channel c_first, first input row, column xin) modulo 2^32; the whole tensor is below 4 GB, and a position
  // left of or above it is stepped past before it is used
  uint32_t off = ((static_cast<uint32_t>(b) * g.C + c_first) * plane + static_cast<uint32_t>((y0 - g.ph) * g.W + xin)) * static_cast<uint32_t>(sizeof(T));
  const char* xb = reinterpret_cast<const char*>(x);

  float a1[G], a2[G];            // sums of the output rows under way
  uint32_t h1[Q], h2[Q];         // sign bits of the two rows before, nine bits per channel
#pragma unroll
  for (int i = 0; i < G; i++) { a1[i] = 0.0f; a2[i] = 0.0f; }
#pragma unroll
  for (int i = 0; i < Q; i++) { h1[i] = 0u; h2[i] = 0u; }

  const int64_t word0 = static_cast<int64_t>(range) * p.words, group0 = static_cast<int64_t>(range) * p.groups;
  // the last range also writes the row's padding (the staged zeros behind its words)
  const uint32_t run_words = range == p.ranges - 1 ? static_cast<uint32_t>(ld_words - word0) : p.words;
  const uint32_t run_groups = range == p.ranges - 1 ? static_cast<uint32_t>(ld_scales - group0) : p.groups;
  __syncthreads();

  float v[CH];                   // the lane's column of a row
  auto load_row = [&](int r) {
#pragma unroll
    for (int c = 0; c < CH; c++) v[c] = 0.0f;
    if (col_ok && r >= 0 && r < g.H) {
      if (LIVE == CH && nch == CH) {
#pragma unroll
        for (int c = 0; c < CH; c++) v[c] = load_elem<T>(xb + static_cast<size_t>(c) * plane_bytes + off);
      } else {
#pragma unroll
        for (int c = 0; c < LIVE; c++)
          if (c < nch) v[c] = load_elem<T>(xb + static_cast<size_t>(c) * plane_bytes + off);
      }
    }
    off += static_cast<uint32_t>(g.W) * static_cast<uint32_t>(sizeof(T));
  };
  // The row in v: its sign bits to h, and to cont[i][q] what it adds to group q of an output row in whose window it is row i
  // (has: whether that is anything, known at compile time).
  auto take_row = [&](uint32_t (&h)[Q], float (&cont)[3][G], bool (&has)[3][G]) {
    // ---- signs (x + 0 so that -0 counts as +0) of the window's three columns
    uint32_t pat = 0;
#pragma unroll
    for (int c = CH - 1; c >= 0; c--) pat = __funnelshift_l(__float_as_uint(v[c] + 0.0f), pat, 1);
    const uint32_t bo = ~pat, bl = __shfl_up_sync(0xFFFFFFFFu, bo, 1), br = __shfl_down_sync(0xFFFFFFFFu, bo, 1);
    {
      // nibbles of even and odd index, one per byte; the middle and the right column shifted to their place
      const uint32_t m4 = 0x0F0F0F0Fu;
      const uint32_t le = bl & m4, lo = (bl >> 4) & m4, ce = (bo & m4) << 1, co = (bo >> 3) & (m4 << 1), re = (br & m4) << 2, ro = (br >> 2) & (m4 << 2);
#pragma unroll
      for (int q = 0; q < Q; q++) {
        if (4 * q >= LIVE) { h[q] = 0u; continue; }
        const uint32_t sel = 0x1111u * (q >> 1);
        uint32_t o = __byte_perm((q & 1) ? lo : le, 0, sel) & 0x08040201u;
        o |= __byte_perm((q & 1) ? co : ce, 0, sel) & 0x10080402u;
        o |= __byte_perm((q & 1) ? ro : re, 0, sel) & 0x20100804u;
        h[q] = o;
      }
    }
    // ---- sums
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
      for (int q = 0; q < G; q++) { has[i][q] = false; cont[i][q] = 0.0f; }
    auto add = [&](int i, int q, float s) { cont[i][q] = has[i][q] ? cont[i][q] + s : s; has[i][q] = true; };
#pragma unroll
    for (int u = 0; u < UNITS; u++) {
#pragma unroll
      for (int q = 0; q < 9; q++) {
        float col = 0.0f;
        bool any = false;
#pragma unroll
        for (int c = 0; c < BETA; c++)
          if (C::whole(c) && C::group(c, 0) == q && u * BETA + c < LIVE) { col = any ? col + fabsf(v[u * BETA + c]) : fabsf(v[u * BETA + c]); any = true; }
        if (any) {
          const float s = (__shfl_up_sync(0xFFFFFFFFu, col, 1) + col) + __shfl_down_sync(0xFFFFFFFFu, col, 1);
          add(0, u * 9 + q, s); add(1, u * 9 + q, s); add(2, u * 9 + q, s);
        }
      }
#pragma unroll
      for (int c = 0; c < BETA; c++) {
        if (C::whole(c) || u * BETA + c >= LIVE) continue;
        const float m = v[u * BETA + c], l = __shfl_up_sync(0xFFFFFFFFu, m, 1), rr = __shfl_down_sync(0xFFFFFFFFu, m, 1);
        const float lm = fabsf(l) + fabsf(m), mr = fabsf(m) + fabsf(rr), all = lm + fabsf(rr);
#pragma unroll
        for (int i = 0; i < 3; i++) {
          const int g0 = C::group(c, 3 * i), g1 = C::group(c, 3 * i + 1), g2 = C::group(c, 3 * i + 2);
          if (g0 == g2) add(i, u * 9 + g0, all);
          else if (g0 == g1) { add(i, u * 9 + g0, lm); add(i, u * 9 + g2, fabsf(rr)); }
          else { add(i, u * 9 + g0, fabsf(l)); add(i, u * 9 + g2, mr); }
        }
      }
    }
  };

  load_row(y0 - g.ph);
  for (int t = 0; t < p.R + 2; t++) {       // a turn takes one row, the last of output row t - 2's window
    uint32_t h0[Q];
    float fin[G];
    {
      float cont[3][G];
      bool has[3][G];
      take_row(h0, cont, has);
#pragma unroll
      for (int q = 0; q < G; q++) {
        const bool f0 = has[0][q], f1 = has[1][q], f2 = has[2][q];
        fin[q] = (f0 || f1) ? (f2 ? a2[q] + cont[2][q] : a2[q]) : cont[2][q];
        a2[q] = f0 ? (f1 ? a1[q] + cont[1][q] : a1[q]) : cont[1][q];
        a1[q] = cont[0][q];
      }
    }
    if (t < p.R + 1) load_row(y0 - g.ph + t + 1);      // in flight while this row is staged and leaves
    const int row = t - 2;
    // ---- the output row whose window ends here
    uint32_t* stage = stage0 + (t & 1) * buf_words;
    if (row >= 0 && out_ok && nch > 0) {
      uint64_t V[Q];             // 36 bits: four channels' nine taps
#pragma unroll
      for (int q = 0; q < Q; q++) V[q] = static_cast<uint64_t>(h2[q]) + (static_cast<uint64_t>(h1[q]) << 3) + (static_cast<uint64_t>(h0[q]) << 6);
      uint32_t wd[(9 * CH + 31) / 32];
#pragma unroll
      for (int q = 0; q < (9 * CH + 31) / 32; q++) {
        uint32_t o = q < Q ? static_cast<uint32_t>(V[q < Q ? q : 0]) << ((4 * q) & 31) : 0u;
        if (q > 0) o |= static_cast<uint32_t>(V[q > 0 ? q - 1 : 0] >> (36 - 4 * q));
        wd[q] = o;
      }
      uint32_t* sb = stage + slot * p.ldb;
      float* ss = reinterpret_cast<float*>(stage + p.slots * p.ldb) + slot * p.lds + piece * G;
      const int valid = 9 * nch;                            // elements of the row that this piece has
      if constexpr (CH == 32) {
#pragma unroll
        for (int q = 0; q < 9; q++) {
          if (LIVE == CH && nch == CH) sb[piece * 9 + q] = wd[q];
          else if (32 * q < valid) sb[piece * 9 + q] = valid - 32 * q >= 32 ? wd[q] : wd[q] & ((1u << (valid - 32 * q)) - 1u);
        }
      } else if constexpr (CH == 16) {
        unsigned short* by = reinterpret_cast<unsigned short*>(sb) + piece * 9;
#pragma unroll
        for (int q = 0; q < 9; q++) {
          const uint32_t o = (wd[q >> 1] >> (16 * (q & 1))) & 0xFFFFu;
          if (LIVE == CH && nch == CH) by[q] = static_cast<unsigned short>(o);
          else if (16 * q < valid) by[q] = static_cast<unsigned short>(valid - 16 * q >= 16 ? o : o & ((1u << (valid - 16 * q)) - 1u));
        }
      } else {
        unsigned char* by = reinterpret_cast<unsigned char*>(sb) + piece * (9 * CH / 8);
#pragma unroll
        for (int q = 0; q < 9 * CH / 8; q++) {
          const uint32_t o = (wd[q >> 2] >> (8 * (q & 3))) & 0xFFu;
          if (nch == CH) by[q] = static_cast<unsigned char>(o);
          else if (8 * q < valid) by[q] = static_cast<unsigned char>(valid - 8 * q >= 8 ? o : o & ((1u << (valid - 8 * q)) - 1u));
        }
      }
      const float inv = p.gw > 1 ? 1.0f : 1.0f / BETA;      // groups of several words are divided when their words are added
      if (LIVE == CH && nch == CH) {
#pragma unroll
        for (int q = 0; q < G; q++) ss[q] = fin[q] * inv;
      } else {
        float last = 0.0f;       // of the row's short last group
#pragma unroll
        for (int q = 0; q < (9 * LIVE + BETA - 1) / BETA; q++) {
          if (BETA * (q + 1) <= valid) ss[q] = fin[q] * inv;
          else if (BETA * q < valid) last = fin[q];
        }
        const int n = valid % BETA;
        if (n != 0) ss[valid / BETA] = p.gw > 1 ? last : last / static_cast<float>(n);
      }
    }
#pragma unroll
    for (int q = 0; q < Q; q++) { h2[q] = h1[q]; h1[q] = h0[q]; }
    if (row < 0) continue;
    __syncthreads();
    // ---- leave: consecutive threads on consecutive pieces of an output column's words.  One barrier per row is enough: the
    // next row is staged in the other buffer, and the one after it behind the next barrier.
    auto leave = [&](const FastDiv& by, uint32_t step, uint32_t n, auto&& store) {
      for (uint32_t i = threadIdx.x; i < static_cast<uint32_t>(p.slots) * by.d; i += blockDim.x) {
        const uint32_t sl = by.div(i), w = (i - sl * by.d) * step;
        const int2 at = slot_at[sl];
        if (row < at.y && w < n) store(sl, w, static_cast<int64_t>(at.x) + static_cast<int64_t>(row) * g.Wo);
      }
    };
    if (p.vec_bits) {
      leave(by_bits, 4, run_words, [&](uint32_t sl, uint32_t w, int64_t m) {
        const uint32_t* s = stage + sl * p.ldb + w;
        *reinterpret_cast<uint4*>(bits + m * ld_words + word0 + w) = make_uint4(s[0], s[1], s[2], s[3]);
      });
    } else {
      leave(by_bits, 1, run_words, [&](uint32_t sl, uint32_t w, int64_t m) { bits[m * ld_words + word0 + w] = stage[sl * p.ldb + w]; });
    }
    const float* sums = reinterpret_cast<const float*>(stage + p.slots * p.ldb);
    if (p.gw > 1) {
      const int64_t K = static_cast<int64_t>(g.C) * 9, beta = 32LL * p.gw;
      leave(by_scales, 1, run_groups, [&](uint32_t sl, uint32_t q, int64_t m) {
        const int64_t left = K - (group0 + q) * beta;
        float s = 0.0f;
        if (left > 0) {
          for (int w = 0; w < p.gw && w * 32 < left; w++) s += sums[sl * p.lds + q * p.gw + w];
          s /= static_cast<float>(left < beta ? left : beta);
        }
        store_one(scales, scale_bf16, m * ld_scales + group0 + q, s);
      });
    } else if (p.vec_scales) {
      leave(by_scales, 4, run_groups, [&](uint32_t sl, uint32_t q, int64_t m) {
        const float* s = sums + sl * p.lds + q;
        const int64_t idx = m * ld_scales + group0 + q;
        if (scale_bf16) {
          const __nv_bfloat162 lo = __floats2bfloat162_rn(s[0], s[1]), hi = __floats2bfloat162_rn(s[2], s[3]);
          *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(scales) + idx) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
        } else {
          *reinterpret_cast<float4*>(reinterpret_cast<float*>(scales) + idx) = make_float4(s[0], s[1], s[2], s[3]);
        }
      });
    } else {
      leave(by_scales, 1, run_groups, [&](uint32_t sl, uint32_t q, int64_t m) { store_one(scales, scale_bf16, m * ld_scales + group0 + q, sums[sl * p.lds + q]); });
    }
  }
}

inline bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

bool make_walk_plan(const ConvGeom& g, int32_t beta, int elem_bytes, int sms, int64_t ld_words, int64_t ld_scales, WalkPlan* out) {
  if (g.kh != 3 || g.kw != 3 || g.sh != 1 || g.sw != 1 || g.ph > 2 || g.pw > 2) return false;
  const int64_t K = static_cast<int64_t>(g.C) * 9, M = static_cast<int64_t>(g.B) * g.Ho * g.Wo;
  const bool sub = beta == 2 || beta == 4 || beta == 8 || beta == 16;
  if (beta >= K || !(sub || (beta >= 32 && beta % 32 == 0 && beta / 32 <= 64))) return false;
  // 32-bit byte offsets into the image, 32-bit output rows
  if (static_cast<int64_t>(g.B) * g.C * g.H * g.W * elem_bytes >= (int64_t{1} << 32) || M >= (int64_t{1} << 31)) return false;
  WalkPlan p{};
  p.gw = beta > 32 ? beta / 32 : 1;
  const int ch = channels_for(beta < 32 ? beta : 32);
  const int n_chunks = (g.C + 31) / 32, n_pieces = (g.C + ch - 1) / ch, per_chunk = 32 / ch;
  // channels of a CTA: four warps' worth; ranges start at whole words (and, at four chunks, at whole 16-byte pieces of them)
  int chunks = per_chunk == 4 ? 1 : 4;
  if (chunks > n_chunks) chunks = n_chunks;
  if ((chunks * 9) % p.gw != 0 && chunks < n_chunks) chunks = n_chunks <= kMaxWarps ? n_chunks : kMaxWarps;
  if ((chunks * 9) % p.gw != 0 && chunks < n_chunks) return false;      // a group would straddle two ranges
  p.pieces = chunks * per_chunk < n_pieces ? chunks * per_chunk : n_pieces;
  p.ranges = (n_chunks + chunks - 1) / chunks;
  p.sets = (4 + p.pieces - 1) / p.pieces;
  if (p.pieces * p.sets > kMaxWarps) return false;
  // strips: as many of a warp's lanes on output columns as possible
  double best = 0.0;
  for (int n = 1; n <= g.Wo; n++) {
    const int pw = (g.Wo + n - 1) / n, lanes = pw + 2;
    if (lanes > 32) continue;
    const int l = 32 / lanes;
    const double eff = static_cast<double>(l) * g.Wo / n;
    if (eff > best * 1.0001) { best = eff; p.strips = n; p.Pw = pw; p.P = lanes; p.L = l; }
    if (pw <= 2) break;
  }
  p.slots = p.sets * p.L * p.Pw;
  p.words = chunks * 9;
  p.groups = static_cast<int32_t>(p.gw > 1 ? chunks * 9 / p.gw : static_cast<int64_t>(chunks) * 288 / beta);
  if (p.ranges == 1) { p.words = static_cast<int32_t>(ld_words); p.groups = static_cast<int32_t>(ld_scales); }
  // rows of a segment: every segment reads two rows more than it leaves, a CTA more than the machine holds costs a turn.  (With
  // the warps per SM counted one by one instead of in turns, beta 32 unless said, us: 33 x 96 x 40 x 40 at beta 8 25.7 against
  // 19.3, 20 x 192 x 55 x 55 at beta 2 94 / 75, 128 x 64 x 56 x 56 47.2 / 41.4, 100 x 256 x 14 x 14 15.1 / 12.6, 64 x 512 x 7 x 7
  // 9.9 / 9.0, 64 x 128 x 28 x 28 at beta 4 29.9 / 27.1; none slower.)
  int64_t cost = 0;
  for (int r = 1; r <= g.Ho; r++) {
    const int nseg = (g.Ho + r - 1) / r;
    if (r > 1 && (g.Ho + r - 2) / (r - 1) == nseg) continue;      // the same segments, less evenly
    const int64_t units = static_cast<int64_t>(g.B) * nseg * p.strips;
    const int64_t ctas = (units + p.sets * p.L - 1) / (p.sets * p.L) * p.ranges;
    const int64_t at_once = static_cast<int64_t>(sms) * (kWarpsAtOnce / (p.sets * p.pieces));
    const int64_t c = (r + 2) * ((ctas + at_once - 1) / at_once);
    if (cost == 0 || c < cost) { cost = c; p.R = r; p.nseg = nseg; }
  }
  const int64_t units = static_cast<int64_t>(g.B) * p.nseg * p.strips;
  if (units >= (int64_t{1} << 28)) return false;
  p.n_units = static_cast<int32_t>(units);
  const int64_t last_words = ld_words - static_cast<int64_t>(p.ranges - 1) * p.words, last_groups = ld_scales - static_cast<int64_t>(p.ranges - 1) * p.groups;
  const int64_t max_words = last_words > p.words ? last_words : p.words, max_groups = last_groups > p.groups ? last_groups : p.groups;
  const int64_t max_sums = p.gw > 1 ? chunks * 9 : max_groups;
  // odd pitches: consecutive output columns in different banks
  p.ldb = static_cast<int32_t>(max_words | 1);
  p.lds = static_cast<int32_t>(max_sums | 1);
  p.max_words = static_cast<int32_t>(max_words);
  p.max_groups = static_cast<int32_t>(max_groups);
  *out = p;
  return walk_smem_bytes(p) <= 100 * 1024;
}

template <int BETA, int LIVE, typename T>
cudaError_t launch_walk_live(const void* x, const ConvGeom& g, WalkPlan p, const UmmaPrepJob* prep, uint32_t* bits, int64_t ld_words, void* scales,
                               int64_t ld_scales, int scale_bf16, int dev, cudaStream_t stream) {
  static DeviceOnce configured;
  if (configured.pending(dev)) {
    const cudaError_t e = cudaFuncSetAttribute(im2col_walk_kernel<BETA, LIVE, T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    if (e != cudaSuccess) return e;
    configured.mark(dev);
  }
  UmmaPrepJob job{};
  int n_prep = 0;
  if (prep) {
    job = *prep;
    n_prep = job.n_stages * job.tiles_n;
    if (n_prep > 4096) return cudaErrorNotSupported;       // the caller expands large weight operands on its own
  }
  // 16-byte pieces where every range starts and ends on one
  p.vec_bits = ld_words % 4 == 0 && aligned16(bits) && (p.ranges == 1 || p.words % 4 == 0);
  p.vec_scales = p.gw == 1 && ld_scales % 4 == 0 && aligned16(scales) && (p.ranges == 1 || p.groups % 4 == 0);
  const FastDiv by_bits = FastDiv::make(p.vec_bits ? (p.max_words + 3) / 4 : p.max_words);
  const FastDiv by_scales = FastDiv::make(p.vec_scales ? (p.max_groups + 3) / 4 : p.max_groups);
  const int64_t ctas = (static_cast<int64_t>(p.n_units) + p.sets * p.L - 1) / (p.sets * p.L) * p.ranges;
  return launch_pdl(im2col_walk_kernel<BETA, LIVE, T>, dim3(static_cast<unsigned>(ctas + n_prep)), dim3(static_cast<unsigned>(p.sets * p.pieces * 32)),
                    walk_smem_bytes(p), stream, static_cast<const T*>(x), g, p, by_bits, by_scales, job, n_prep, bits, ld_words, scales, ld_scales, scale_bf16);
}

// The kernel for as few channels as the image has.
template <int BETA, typename T, typename... Rest>
cudaError_t launch_walk(const void* x, const ConvGeom& g, Rest... rest) {
  constexpr int CH = channels_for(BETA);
  if constexpr (CH >= 16) {
    if (g.C <= 8) return launch_walk_live<BETA, 8, T>(x, g, rest...);
  }
  if constexpr (CH == 32) {
    if (g.C <= 16) return launch_walk_live<BETA, 16, T>(x, g, rest...);
    if (g.C <= 24) return launch_walk_live<BETA, 24, T>(x, g, rest...);
  }
  return launch_walk_live<BETA, CH, T>(x, g, rest...);
}

template <typename T>
cudaError_t launch_walk_beta(const void* x, const ConvGeom& g, int32_t beta, const WalkPlan& p, const UmmaPrepJob* prep, uint32_t* bits,
                             int64_t ld_words, void* scales, int64_t ld_scales, int scale_bf16, int dev, cudaStream_t stream) {
  switch (beta) {
    case 2: return launch_walk<2, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
    case 4: return launch_walk<4, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
    case 8: return launch_walk<8, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
    case 16: return launch_walk<16, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
    default: return launch_walk<32, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
  }
}

}  // namespace

// ld_words, ld_scales as the packed operand of the convolution has them.
bool im2col_walk_supported(int x_bf16, const ConvGeom& g, int32_t beta, int64_t ld_words, int64_t ld_scales) {
  int dev = 0, sms = 0;
  WalkPlan p;
  return current_device(&dev, &sms) == cudaSuccess && make_walk_plan(g, beta, x_bf16 ? 2 : 4, sms, ld_words, ld_scales, &p);
}

cudaError_t launch_im2col_walk(const void* x, int x_bf16, const ConvGeom& g, int32_t beta, uint32_t* bits, int64_t ld_words, void* scales,
                               int64_t ld_scales, int scale_bf16, cudaStream_t stream, const UmmaPrepJob* prep) {
  int dev = 0, sms = 0;
  WalkPlan p;
  const cudaError_t e = current_device(&dev, &sms);
  if (e != cudaSuccess) return e;
  if (!make_walk_plan(g, beta, x_bf16 ? 2 : 4, sms, ld_words, ld_scales, &p)) return cudaErrorNotSupported;
  if (x_bf16) return launch_walk_beta<__nv_bfloat16>(x, g, beta, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
  return launch_walk_beta<float>(x, g, beta, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, dev, stream);
}

}  // namespace hbmm
