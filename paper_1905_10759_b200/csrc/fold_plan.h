// The folded contraction's workspace and schedule as numbers: what the query reports, what a launch may touch of a workspace of
// a given size, and which launches are balanced (host code, no CUDA).
#pragma once
#include <cstddef>
#include <cstdint>

namespace hbmm {

constexpr int kEpilogueWarps = 4;

struct FoldShape {
  int64_t M, N, n_words;          // K in 32-bit words
  int32_t tn;                     // columns of a tile: 64 or 128
  bool a_subword;                 // activation groups shorter than a word
  static constexpr int64_t kRows = 128, kWords = 2;       // rows of a tile, words of a stage
  static constexpr size_t kRowBytes = 2 * 128;            // a weight row's share of a stage: both pieces, 64 fp16 each
  int64_t stages() const { return (n_words + kWords - 1) / kWords; }        // per tile
  int64_t tiles_n() const { return (N + tn - 1) / tn; }
  int64_t tiles() const { return (M + kRows - 1) / kRows * tiles_n(); }
  size_t weight_bytes() const { return static_cast<size_t>(tiles_n() * stages()) * tn * kRowBytes; }
};

// Balanced schedule: worth its reduction traffic when the tiles are few waves of the machine and a tile's K walk is
// long enough to cut.  The workspace is sized for any device of up to kMaxBalancedCtas multiprocessors.
constexpr int64_t kMaxBalancedCtas = 256;
constexpr int64_t kBalancedWaves = 4;
constexpr int64_t kBalancedMinStages = 4;
constexpr int64_t kBalancedMaxShare = 4;
// The arrival counters take the first kCounterCount words of the area, for the most tiles a balanced launch may have, so
// that they lie at the same place and are all zeroed by whichever call expands the weights, whatever its number of rows:
// prepared calls with more and fewer rows follow it.  (Sized for the call's own tiles, they lay under another call's partial
// tiles.)  The area holds them without being larger: of its min(units, 256) pairs of slots a launch uses at most
// min(units / kBalancedMinStages, kMaxBalancedCtas - 1), and one pair is four times the counters.
constexpr int64_t kCounterCount = kBalancedWaves * kMaxBalancedCtas * kEpilogueWarps;
static_assert(2 * FoldShape::kRows * 64 * sizeof(float) >= kCounterCount * sizeof(int32_t), "a pair of slots holds the counters");

inline bool balanced_possible(const FoldShape& f, int64_t sms) {
  return sms <= kMaxBalancedCtas && f.stages() >= kBalancedMinStages && f.tiles() < kBalancedWaves * sms;
}
inline size_t slot_bytes(const FoldShape& f) { return static_cast<size_t>(FoldShape::kRows) * f.tn * sizeof(float); }
inline size_t balanced_bytes(const FoldShape& f) {
  if (!balanced_possible(f, kMaxBalancedCtas)) return 0;
  const int64_t units = f.tiles() * f.stages(), ctas = units < kMaxBalancedCtas ? units : kMaxBalancedCtas;
  const size_t counters = (static_cast<size_t>(f.tiles()) * kEpilogueWarps * sizeof(int32_t) + 255) / 256 * 256;
  return counters + static_cast<size_t>(2 * ctas) * slot_bytes(f);
}
// [W stages][one float per weight row][counters][partial slots][one float per activation row: its largest scale]
inline size_t balanced_offset(const FoldShape& f) {
  return (f.weight_bytes() + static_cast<size_t>(f.tiles_n() * f.tn) * sizeof(float) + 255) / 256 * 256;
}
inline size_t rowmax_offset(const FoldShape& f) { return (balanced_offset(f) + balanced_bytes(f) + 255) / 256 * 256; }
inline size_t fold_bytes(const FoldShape& f) {
  return f.a_subword ? rowmax_offset(f) + static_cast<size_t>(f.M) * sizeof(float) : balanced_offset(f) + balanced_bytes(f);
}

// The balanced schedule's part of a workspace of `have` bytes.  counters: there, and zeroed by a call that expands the weights.
// A product with too many tiles for the schedule has no such part; its counters are zeroed all the same where the workspace
// reaches that far, for prepared calls with fewer rows.  slots: the partial tiles too.
struct FoldArea { bool counters, slots; size_t at, slots_at; };
inline FoldArea fold_area(const FoldShape& f, size_t have) {
  FoldArea a{};
  a.at = balanced_offset(f);
  a.slots_at = a.at + kCounterCount * sizeof(int32_t);
  const size_t own = balanced_bytes(f);
  a.slots = own != 0 && have >= a.at + own;
  a.counters = a.slots || (own == 0 && !f.a_subword && f.stages() >= kBalancedMinStages && have >= a.slots_at);
  return a;
}

// Equal runs of (tile, stage) pairs, one per CTA: they pay when they shorten the longest CTA's walk by a tenth or more.
struct Runs { int64_t run, ctas, walk; bool pay; };
inline Runs balanced_runs(const FoldShape& f, int64_t sms, size_t have) {
  Runs r{};
  const int64_t n_stages = f.stages(), tiles = f.tiles(), units = tiles * n_stages;
  r.ctas = units / kBalancedMinStages < sms ? units / kBalancedMinStages : sms;
  if (r.ctas > kMaxBalancedCtas - 1) r.ctas = kMaxBalancedCtas - 1;
  if (r.ctas < 1) r.ctas = 1;
  r.run = (units + r.ctas - 1) / r.ctas;
  // a tile is shared by at most kBalancedMaxShare + 1 CTAs: the CTA that completes it adds the others' partial
  // accumulators one after the other, which costs more than the shorter walk saves beyond that
  const int64_t min_run = (n_stages + kBalancedMaxShare - 1) / kBalancedMaxShare;
  if (r.run < min_run) r.run = min_run;
  r.walk = (tiles + sms - 1) / sms * n_stages;
  r.pay = balanced_possible(f, sms) && fold_area(f, have).slots && r.run * 10 <= r.walk * 9;
  r.ctas = (units + r.run - 1) / r.run;                     // no CTA without work
  return r;
}
// Whole short 128-column tiles with the wide accumulator instead of the balanced schedule of narrow ones, whose reduction costs
// some 9 us.  In hundredths of a us: a stage 46 of a whole tile, 42 of a run, a turn's exposed epilogue 150.  Balanced / whole
// wide, us: 25088 x 128 x 576 21.4 / 17.3, 12544 x 128 x 1152 19.7 / 15.5, 4096 x 960 x 256 21.0 / 13.5, 1000 x 3000 x 640 27.3 /
// 18.3, 50176 x 128 x 576 27.0 / 24.0; level at 12544 x 256 x 1152, slower at 50176 x 128 x 1152 (34.4 / 35.6) and 2048 x 4096 x
// 768 (40.9 / 45.2).  The error against 64 bits falls to a third.  (Whole narrow tiles take 14.8 us of the first, but sum all of
// K in one accumulator with the small products: 6.5e-7 balanced, 7.7e-7 narrow, 2.3e-7 wide.)
inline bool whole_wide_pays(const Runs& r, int64_t n_stages) {
  return r.pay && 46 * r.walk + 150 * (r.walk / n_stages) < 900 + 42 * r.run;
}

// Whether finished blocks may leave by tensor copies, whose coordinates are 32-bit numbers.  A product with more rows is one launch
// all the same, with stores of its own: cut into parts, a part would not find in the whole product's workspace what a product
// of its size asks for (2^30 + 25600 rows of K = 256, N = 4 report 65,792 bytes, the 25600 rows alone 16.8 MB).
inline bool copies_reach(const FoldShape& f) { return f.M < (int64_t{1} << 31) && f.N < (int64_t{1} << 31); }

}  // namespace hbmm
