// Packed convolution front end for 1 x 1 filters: a row of K is one pixel's channels, so nothing is shared between output pixels
// and nothing is staged.  A thread forms one K-word of one output pixel (one scale group where that is several words): 32
// loads in flight, consecutive lanes on consecutive pixels of a channel plane, a sign shift and an addition per element, the
// word and its means stored where they belong.  Any stride, padding, type and alignment of the image.
// What bounds it: reading the image once.  The tiles of im2col_tma.cu hold 112 pixels and leave twelve warps four words'
// work per chunk of 32 channels, the gathers of im2col.cu divide per element.  Against them, us: 38 x 192 x 55 x 55 at
// stride 2, beta 4 / 32 26.8 / 24.6 -> 7.1 / 6.2; 64 x 192 x 7 x 7 bf16, beta 8 10.9 -> 2.2; 64 x 256 x 14 x 14, beta 32 / 2 6.0 / 9.7
// -> 3.8 / 6.0; 20 x 512 x 28 x 28, beta 128 10.5 -> 7.7, bf16 at beta 16 24.0 -> 6.1; one image of 512 x 7 x 7, beta 32 / 256 2.7 /
// 6.9 -> 1.8 / 4.9; 35 x 64 x 56 x 56, beta 64 (one group per row) 29.6 -> 5.8.
#include <cuda_bf16.h>
#include "kernels.h"
#include "gemm_umma_prep.cuh"
#include "gemm_fold_prep.cuh"
#include "pdl.cuh"

namespace hbmm {
namespace {

constexpr int kPixels = 128;           // output pixels (threads) of a CTA
constexpr int kMostWords = 8;          // of a scale group: longer ones would leave too few threads

struct PointArgs {
  int64_t M, blocks_m;                 // output pixels, CTAs per unit
  int32_t gw, n_words, units, G;       // words per unit, words of a row, units (words or groups) of a row, scale groups
  int32_t vec;                         // a word's scales are stored as vectors
  int32_t row_bits, row_scales;        // rows of one word / of one group that are 16 bytes long: stored whole, padding and all
};

__device__ __forceinline__ void store_one(void* scales, int bf16, int64_t idx, float v) {
  if (bf16) reinterpret_cast<__nv_bfloat16*>(scales)[idx] = __float2bfloat16_rn(v);
  else reinterpret_cast<float*>(scales)[idx] = v;
}

// BETA: 2 .. 16, or 32 for groups of whole words.  LIVE: no channel beyond it (a row of one word).
template <int BETA, int LIVE, typename T>
__global__ void __launch_bounds__(kPixels)
im2col_point_kernel(const T* __restrict__ x, const ConvGeom g, const PointArgs p, const __grid_constant__ UmmaPrepJob prep, int n_prep,
                    uint32_t* __restrict__ bits, int64_t ld_words, void* __restrict__ scales, int64_t ld_scales, int scale_bf16) {
  constexpr int SUB = 32 / BETA;
  pdl_launch_dependents();
  pdl_wait();
  if (static_cast<int>(blockIdx.x) < n_prep) {      // the weight operand of the contraction that follows: one task per CTA
    const int st = blockIdx.x % prep.n_stages, tile_n = blockIdx.x / prep.n_stages;
    if (prep.tn == 64) { if (threadIdx.x < 64) fold::prepare_w_task<64>(prep.f, prep.out, prep.out_down, st, tile_n, threadIdx.x); }
    else fold::prepare_w_task<128>(prep.f, prep.out, prep.out_down, st, tile_n, threadIdx.x);
    return;
  }
  const uint32_t cta = blockIdx.x - n_prep;
  const int unit = static_cast<int>(cta / static_cast<uint32_t>(p.blocks_m));
  const int64_t m = static_cast<int64_t>(cta - unit * static_cast<uint32_t>(p.blocks_m)) * kPixels + threadIdx.x;
  if (m >= p.M) return;
  const uint32_t mi = static_cast<uint32_t>(m), row = mi / static_cast<uint32_t>(g.Wo);
  const int xo = static_cast<int>(mi - row * g.Wo), b = static_cast<int>(row / static_cast<uint32_t>(g.Ho)), yo = static_cast<int>(row - b * static_cast<uint32_t>(g.Ho));
  const int y = yo * g.sh - g.ph, xx = xo * g.sw - g.pw;
  const bool inside = y >= 0 && y < g.H && xx >= 0 && xx < g.W;
  const int64_t plane = static_cast<int64_t>(g.H) * g.W;
  const T* px = x + (static_cast<int64_t>(b) * g.C * g.H + (inside ? y : 0)) * g.W + (inside ? xx : 0);
  float total = 0.0f;
  for (int w = unit * p.gw; w < (unit + 1) * p.gw && w < p.n_words; w++) {
    const int nk = g.C - 32 * w < 32 ? g.C - 32 * w : 32;
    const T* pc = px + static_cast<int64_t>(32 * w) * plane;
    float v[32];
    if (LIVE == 32 && nk == 32 && inside) {
#pragma unroll
      for (int e = 0; e < 32; e++) v[e] = load_elem<T>(pc + e * plane);
    } else {
#pragma unroll
      for (int e = 0; e < 32; e++) v[e] = e < LIVE && inside && e < nk ? load_elem<T>(pc + e * plane) : 0.0f;
    }
    uint32_t pat = 0;
#pragma unroll
    for (int e = 31; e >= 0; e--) pat = __funnelshift_l(__float_as_uint(v[e] + 0.0f), pat, 1);      // + 0: -0 counts as +0
    const uint32_t word = ~pat & (nk == 32 ? 0xFFFFFFFFu : (1u << nk) - 1u);
    if (p.row_bits) *reinterpret_cast<uint4*>(bits + m * 4) = make_uint4(word, 0u, 0u, 0u);
    else bits[m * ld_words + w] = word;
    if constexpr (SUB == 1) {
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int e = 0; e < LIVE; e++) s[e & 3] += fabsf(v[e]);
      total += (s[0] + s[1]) + (s[2] + s[3]);
    } else {
      float mean[SUB];
#pragma unroll
      for (int i = 0; i < SUB; i++) {
        if (i * BETA >= LIVE) { mean[i] = 0.0f; continue; }
        float s0 = 0.f, s1 = 0.f;
#pragma unroll
        for (int e = 0; e < BETA; e += 2) { s0 += fabsf(v[i * BETA + e]); s1 += fabsf(v[i * BETA + e + 1]); }
        const int cnt = nk - i * BETA;
        mean[i] = cnt >= BETA ? (s0 + s1) * (1.0f / BETA) : (cnt > 0 ? (s0 + s1) / static_cast<float>(cnt) : 0.0f);
      }
      const int64_t at = m * ld_scales + static_cast<int64_t>(w) * SUB;
      if (p.vec && nk == 32) {
        float* d = reinterpret_cast<float*>(scales) + at;
        if constexpr (SUB == 2) {
          *reinterpret_cast<float2*>(d) = make_float2(mean[0], mean[1]);
        } else {
#pragma unroll
          for (int i = 0; i < SUB; i += 4) *reinterpret_cast<float4*>(d + i) = make_float4(mean[i], mean[(i + 1) % SUB], mean[(i + 2) % SUB], mean[(i + 3) % SUB]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < SUB; i++)
          if (i * BETA < nk) store_one(scales, scale_bf16, at + i, mean[i]);
      }
    }
  }
  if constexpr (SUB == 1) {
    const int left = g.C - unit * p.gw * 32, n = left < p.gw * 32 ? left : p.gw * 32;
    const float mean = total / static_cast<float>(n);
    if (p.row_scales) {
      const uint32_t first = scale_bf16 ? __bfloat16_as_ushort(__float2bfloat16_rn(mean)) : __float_as_uint(mean);
      reinterpret_cast<uint4*>(scales)[m] = make_uint4(first, 0u, 0u, 0u);
    } else {
      store_one(scales, scale_bf16, m * ld_scales + unit, mean);
    }
  }
  if (unit == p.units - 1) {           // the row's padding
    if (!p.row_bits)
      for (int64_t w = p.n_words; w < ld_words; w++) bits[m * ld_words + w] = 0u;
    if (!p.row_scales)
      for (int64_t q = p.G; q < ld_scales; q++) store_one(scales, scale_bf16, m * ld_scales + q, 0.0f);
  }
}

bool make_point_args(const ConvGeom& g, int32_t beta, PointArgs* out) {
  if (g.kh != 1 || g.kw != 1) return false;
  const bool sub = beta == 2 || beta == 4 || beta == 8 || beta == 16;
  const bool one = beta >= g.C;          // one group per row
  PointArgs p{};
  p.M = static_cast<int64_t>(g.B) * g.Ho * g.Wo;
  p.n_words = (g.C + 31) / 32;
  p.gw = one ? p.n_words : (beta > 32 ? beta / 32 : 1);
  if (!(one || sub || (beta >= 32 && beta % 32 == 0)) || p.gw > kMostWords) return false;
  p.units = (p.n_words + p.gw - 1) / p.gw;
  p.G = one ? 1 : (g.C + beta - 1) / beta;
  p.blocks_m = (p.M + kPixels - 1) / kPixels;
  *out = p;
  return p.M < (int64_t{1} << 31) && p.blocks_m * p.units < (int64_t{1} << 30);
}

template <int BETA, int LIVE, typename T>
cudaError_t launch_point_live(const void* x, const ConvGeom& g, PointArgs p, const UmmaPrepJob* prep, uint32_t* bits, int64_t ld_words, void* scales,
                         int64_t ld_scales, int scale_bf16, cudaStream_t stream) {
  UmmaPrepJob job{};
  int n_prep = 0;
  if (prep) {
    job = *prep;
    n_prep = job.n_stages * job.tiles_n;
    if (n_prep > 4096) return cudaErrorNotSupported;       // the caller expands large weight operands on its own
  }
  // Rows of a few channels are all stores and absent channels: 128 images of 3 x 112 x 112 with padding 1, one group per row, took
  // 42.4 us bf16 with stores element by element and 32 channels' instructions (a thread per row, without this kernel, 30.3), 39.2
  // with whole rows, 20.6 with whole rows and eight channels' instructions.
  p.row_bits = p.n_words == 1 && ld_words == 4 && reinterpret_cast<uintptr_t>(bits) % 16 == 0;
  p.row_scales = BETA == 32 && p.G == 1 && ld_scales == (scale_bf16 ? 8 : 4) && reinterpret_cast<uintptr_t>(scales) % 16 == 0;
  p.vec = !scale_bf16 && reinterpret_cast<uintptr_t>(scales) % 16 == 0 && ld_scales % 4 == 0;
  return launch_pdl(im2col_point_kernel<BETA, LIVE, T>, dim3(static_cast<unsigned>(p.blocks_m * p.units + n_prep)), dim3(kPixels), 0, stream,
                    static_cast<const T*>(x), g, p, job, n_prep, bits, ld_words, scales, ld_scales, scale_bf16);
}

// Up to eight channels: a kernel without the others (figures in launch_point_live).
template <int BETA, typename T, typename... Rest>
cudaError_t launch_point(const void* x, const ConvGeom& g, Rest... rest) {
  if constexpr (BETA <= 4 || BETA == 32) {
    if (g.C <= 8) return launch_point_live<BETA, 8, T>(x, g, rest...);
  }
  return launch_point_live<BETA, 32, T>(x, g, rest...);
}

template <typename T>
cudaError_t launch_point_beta(const void* x, const ConvGeom& g, int32_t beta, const PointArgs& p, const UmmaPrepJob* prep, uint32_t* bits,
                              int64_t ld_words, void* scales, int64_t ld_scales, int scale_bf16, cudaStream_t stream) {
  switch (beta >= g.C ? 32 : beta) {
    case 2: return launch_point<2, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
    case 4: return launch_point<4, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
    case 8: return launch_point<8, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
    case 16: return launch_point<16, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
    default: return launch_point<32, T>(x, g, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
  }
}

}  // namespace

bool im2col_point_supported(const ConvGeom& g, int32_t beta) {
  PointArgs p;
  return make_point_args(g, beta, &p);
}

cudaError_t launch_im2col_point(const void* x, int x_bf16, const ConvGeom& g, int32_t beta, uint32_t* bits, int64_t ld_words, void* scales,
                                int64_t ld_scales, int scale_bf16, cudaStream_t stream, const UmmaPrepJob* prep) {
  PointArgs p;
  if (!make_point_args(g, beta, &p)) return cudaErrorNotSupported;
  if (x_bf16) return launch_point_beta<__nv_bfloat16>(x, g, beta, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
  return launch_point_beta<float>(x, g, beta, p, prep, bits, ld_words, scales, ld_scales, scale_bf16, stream);
}

}  // namespace hbmm
