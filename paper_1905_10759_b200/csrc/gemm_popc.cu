// HBMM contraction of two packed operands on the integer pipe (Section 4.2, Eq. 7) for segment lengths the tiled kernel
// (gemm_popc_tile.cu) has no instantiation for -- three words, five, a whole long row -- and the integer partial sums of
// word segments.  For every output element and every 32-bit K-word: p = popc(a ^ w); the signed +-1 dot of a K-segment is
// D = n_valid - 2 * sum(p); C += (deltaA * deltaW) * D in fp32.  The segment is min(beta_a, beta_w); the operand with the
// coarser groups reuses its scale across segments.  Pad bits are zero in both operands.
#include "kernels.h"
#include "popc_common.cuh"

namespace hbmm {
namespace {

using popc::load_scale;

constexpr int kThreads = 256;

struct GemmArgs {
  const uint32_t* a_bits; const void* a_scales;
  const uint32_t* w_bits; const void* w_scales;
  float* C;
  int64_t M, N, K, lda_w, ldw_w, lda_s, ldw_s, ldc;
  int32_t a_bf16, w_bf16;
  int32_t ra, rw;        // groups: A group = segment / ra, W group = segment / rw
  int64_t n_words;       // ceil(K/32)
  int64_t T;             // number of segments
  int32_t seg_words;     // words per segment
};

// Any segment length (in whole words): integer popcounts are carried across K-words and flushed
// with the scales at each segment end.  One thread per 4x4 outputs, operands read through L1.
__global__ void __launch_bounds__(kThreads)
gemm_popc_generic_kernel(const GemmArgs g) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t m0 = static_cast<int64_t>(blockIdx.y) * 64 + ty * 4, n0 = static_cast<int64_t>(blockIdx.x) * 64 + tx * 4;
  float acc[4][4];
  int pc[4][4];
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) { acc[i][j] = 0.0f; pc[i][j] = 0; }
  int64_t seg = 0;
  int in_seg = 0;
  for (int64_t kw = 0; kw < g.n_words; kw++) {
    uint32_t a[4], w[4];
#pragma unroll
    for (int i = 0; i < 4; i++) a[i] = (m0 + i < g.M) ? __ldg(g.a_bits + (m0 + i) * g.lda_w + kw) : 0u;
#pragma unroll
    for (int j = 0; j < 4; j++) w[j] = (n0 + j < g.N) ? __ldg(g.w_bits + (n0 + j) * g.ldw_w + kw) : 0u;
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) pc[i][j] += __popc(a[i] ^ w[j]);
    in_seg++;
    if (in_seg == g.seg_words || kw == g.n_words - 1) {
      const int64_t k0 = seg * g.seg_words * 32;
      int64_t nv = g.K - k0;
      if (nv > static_cast<int64_t>(g.seg_words) * 32) nv = static_cast<int64_t>(g.seg_words) * 32;
      const int64_t ga = seg / g.ra, gw = seg / g.rw;
      float sa[4], sw[4];
#pragma unroll
      for (int i = 0; i < 4; i++) sa[i] = (m0 + i < g.M) ? load_scale(g.a_scales, g.a_bf16, (m0 + i) * g.lda_s + ga) : 0.0f;
#pragma unroll
      for (int j = 0; j < 4; j++) sw[j] = (n0 + j < g.N) ? load_scale(g.w_scales, g.w_bf16, (n0 + j) * g.ldw_s + gw) : 0.0f;
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const float d = static_cast<float>(static_cast<int>(nv) - 2 * pc[i][j]);
          acc[i][j] = fmaf(d * sa[i], sw[j], acc[i][j]);
          pc[i][j] = 0;
        }
      seg++;
      in_seg = 0;
    }
  }
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++)
      if (m0 + i < g.M && n0 + j < g.N) g.C[(m0 + i) * g.ldc + n0 + j] = acc[i][j];
}

// Integer partial sums only: D[m,n,t] = n_valid(t) - 2 * popc over the words of segment t.
__global__ void __launch_bounds__(kThreads)
partials_popc_kernel(const GemmArgs g, int32_t* __restrict__ D) {
  const int64_t total = g.M * g.N * g.T;
  for (int64_t idx = static_cast<int64_t>(blockIdx.x) * kThreads + threadIdx.x; idx < total;
       idx += static_cast<int64_t>(gridDim.x) * kThreads) {
    const int64_t t = idx % g.T, mn = idx / g.T;
    const int64_t n = mn % g.N, m = mn / g.N;
    const int64_t w0 = t * g.seg_words;
    int64_t w1 = w0 + g.seg_words;
    if (w1 > g.n_words) w1 = g.n_words;
    int p = 0;
    for (int64_t w = w0; w < w1; w++) p += __popc(g.a_bits[m * g.lda_w + w] ^ g.w_bits[n * g.ldw_w + w]);
    int64_t nv = g.K - w0 * 32;
    if (nv > static_cast<int64_t>(g.seg_words) * 32) nv = static_cast<int64_t>(g.seg_words) * 32;
    D[idx] = static_cast<int32_t>(nv) - 2 * p;
  }
}

GemmArgs make_args(const PackedView& A, const PackedView& W, float* C, int64_t ldc) {
  GemmArgs g;
  g.a_bits = A.bits; g.a_scales = A.scales; g.w_bits = W.bits; g.w_scales = W.scales; g.C = C;
  g.M = A.rows; g.N = W.rows; g.K = A.K;
  g.lda_w = A.ld_words; g.ldw_w = W.ld_words; g.lda_s = A.ld_scales; g.ldw_s = W.ld_scales; g.ldc = ldc;
  g.a_bf16 = A.scale_bf16; g.w_bf16 = W.scale_bf16;
  g.n_words = (A.K + 31) / 32;
  const bool a_one = A.beta >= A.K, w_one = W.beta >= W.K;  // one group per row
  int64_t seg;
  if (a_one && w_one) seg = g.n_words * 32;
  else if (a_one) seg = W.beta;
  else if (w_one) seg = A.beta;
  else seg = A.beta < W.beta ? A.beta : W.beta;
  g.seg_words = static_cast<int32_t>(seg / 32);
  g.T = (A.K + seg - 1) / seg;
  g.ra = static_cast<int32_t>(a_one ? g.T : A.beta / seg);
  g.rw = static_cast<int32_t>(w_one ? g.T : W.beta / seg);
  return g;
}

}  // namespace

cudaError_t launch_gemm_popc(const PackedView& A, const PackedView& W, float* C, int64_t ldc,
                             cudaStream_t stream) {
  const GemmArgs g = make_args(A, W, C, ldc);
  dim3 grid(static_cast<unsigned>((g.N + 63) / 64), static_cast<unsigned>((g.M + 63) / 64));
  gemm_popc_generic_kernel<<<grid, kThreads, 0, stream>>>(g);
  return cudaGetLastError();
}

cudaError_t launch_partials_popc(const PackedView& A, const PackedView& W, int32_t* D, cudaStream_t stream) {
  const GemmArgs g = make_args(A, W, nullptr, 0);
  const int64_t total = g.M * g.N * g.T;
  int64_t blocks = (total + kThreads - 1) / kThreads;
  if (blocks > 148 * 32) blocks = 148 * 32;
  if (blocks < 1) blocks = 1;
  partials_popc_kernel<<<static_cast<unsigned>(blocks), kThreads, 0, stream>>>(g, D);
  return cudaGetLastError();
}

}  // namespace hbmm
