// How many CTAs share an output tile of the folded contraction in split mode (host code, no CUDA).
#pragma once
#include <atomic>
#include <cstdint>

namespace hbmm {

constexpr int kMaxSplit = 8;            // CTAs that may share a tile (the portable cluster size)
// 256 x 256 x 256 (four stages) takes 7.4 us whole and 7.8 us in two parts; from six stages on parts of two stages win
// (64 x 1024 x 1024, 16 stages: 17.4 -> 8.0 us in eight parts).
constexpr int64_t kSplitMinStages = 2;
constexpr int64_t kSplitFromStages = 6;

// The largest number of CTAs per tile (2 .. 8, at least two stages each) for which every tile's cluster is resident at once;
// 1: not worth it.  Taken where the tiles cover at most half of the machine.  Against the balanced schedule, whose last CTA
// adds the partial tiles through global memory (12 .. 20 rounds of loads by four warps): 256 x 1000 x 4096 28.4 -> 16.2 us,
// 256 x 4096 x 4096 39 -> 30, 256 x 4096 x 9216 61.5 -> 56, 49 x 512 x 4608 26.6 -> 12.2, 1024^3 24.2 -> 13.2 us; and the
// second accumulator brings the error of a result from 4e-7 .. 4e-6 to 1e-7 .. 1.8e-6.
// known[s]: clusters of s CTAs the device holds, plus one; 0: not asked yet.  ask(s, &clusters) asks the device; an answer is
// kept, a failure is not: it costs this call the split into s parts and no later one.
template <typename Ask>
int choose_split(std::atomic<int> (&known)[kMaxSplit + 1], int64_t sms, int64_t tiles, int64_t n_stages, Ask ask) {
  if (2 * tiles > sms || n_stages < kSplitFromStages) return 1;
  int64_t most = n_stages / kSplitMinStages;
  if (most > kMaxSplit) most = kMaxSplit;
  for (int s = static_cast<int>(most); s >= 2; s--) {
    if (tiles * s > sms) continue;
    int n = known[s].load(std::memory_order_relaxed);
    if (n == 0) {
      int clusters = 0;
      if (!ask(s, &clusters)) continue;
      n = clusters + 1;
      known[s].store(n, std::memory_order_relaxed);
    }
    if (tiles <= n - 1) return s;
  }
  return 1;
}

}  // namespace hbmm
