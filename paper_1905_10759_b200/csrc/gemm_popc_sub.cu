// Integer partial sums of sub-word segments (Section 4.2, Eq. 7 with the group sizes of the paper's experiments,
// beta = 2 .. 16): the segment min(beta_a, beta_w) is 2, 4, 8 or 16 bits, so one XOR word holds 32 / segment group dots,
// each read with a shifted, masked popcount: D = n_valid - 2 * popc(((a ^ w) >> shift) & mask).
#include "kernels.h"

namespace hbmm {
namespace {

struct SubArgs {
  const uint32_t* a_bits;
  const uint32_t* w_bits;
  int64_t M, N, K, lda_w, ldw_w;
  int32_t seg;                 // bits per segment: 2, 4, 8 or 16
  int64_t T;                   // segments per row: ceil(K / seg)
};

// D[m,n,t] = n_valid(t) - 2 * popc over the bits of segment t.
__global__ void __launch_bounds__(256)
partials_popc_sub_kernel(const SubArgs g, int32_t* __restrict__ D) {
  const int64_t total = g.M * g.N * g.T;
  const uint32_t mask = (1u << g.seg) - 1u;
  for (int64_t idx = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; idx < total; idx += static_cast<int64_t>(gridDim.x) * 256) {
    const int64_t t = idx % g.T, mn = idx / g.T;
    const int64_t n = mn % g.N, m = mn / g.N;
    const int64_t k0 = t * g.seg;
    const uint32_t x = g.a_bits[m * g.lda_w + (k0 >> 5)] ^ g.w_bits[n * g.ldw_w + (k0 >> 5)];
    const int64_t left = g.K - k0;
    const int nv = left < g.seg ? static_cast<int>(left) : g.seg;
    D[idx] = nv - 2 * __popc((x >> (k0 & 31)) & mask);
  }
}

SubArgs make_args(const PackedView& A, const PackedView& W) {
  const int64_t a = A.beta >= A.K ? A.K : A.beta, w = W.beta >= W.K ? W.K : W.beta;
  SubArgs g;
  g.a_bits = A.bits; g.w_bits = W.bits;
  g.M = A.rows; g.N = W.rows; g.K = A.K;
  g.lda_w = A.ld_words; g.ldw_w = W.ld_words;
  g.seg = static_cast<int32_t>(a < w ? a : w);
  g.T = (A.K + g.seg - 1) / g.seg;
  return g;
}

}  // namespace

// The finer of the two groupings is a sub-word power of two (and not a whole row).
bool gemm_subword(const PackedView& A, const PackedView& W) {
  const int64_t a = A.beta >= A.K ? A.K : A.beta, w = W.beta >= W.K ? W.K : W.beta;
  const int64_t seg = a < w ? a : w;
  return seg < 32 && (seg == 2 || seg == 4 || seg == 8 || seg == 16) && seg < A.K;
}

cudaError_t launch_partials_popc_sub(const PackedView& A, const PackedView& W, int32_t* D, cudaStream_t stream) {
  const SubArgs g = make_args(A, W);
  const int64_t total = g.M * g.N * g.T;
  int64_t blocks = (total + 255) / 256;
  if (blocks > 148 * 32) blocks = 148 * 32;
  if (blocks < 1) blocks = 1;
  partials_popc_sub_kernel<<<static_cast<unsigned>(blocks), 256, 0, stream>>>(g, D);
  return cudaGetLastError();
}

}  // namespace hbmm
