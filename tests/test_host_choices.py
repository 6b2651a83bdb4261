"""Host-side choices that need no GPU: the split of a tile between CTAs when the occupancy query fails, what a folded contraction
may touch of its workspace, and the stream handle the binding passes on."""
import os
import subprocess

import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SPLIT = r"""
#include <cstdio>
#include "split_choice.h"
int main() {
  std::atomic<int> known[hbmm::kMaxSplit + 1] = {};
  bool fail = true;
  int asked = 0;
  auto ask = [&](int, int* clusters) { asked++; *clusters = 16; return !fail; };
  const int during = hbmm::choose_split(known, 148, 8, 64, ask);       // eight tiles of 64 stages: eight parts fit
  fail = false;
  const int after = hbmm::choose_split(known, 148, 8, 64, ask);
  const int seen = asked;
  const int again = hbmm::choose_split(known, 148, 8, 64, ask);
  std::printf("%d %d %d %d %d\n", during, after, again, asked - seen, hbmm::choose_split(known, 148, 8, 5, ask));
}
"""


def test_failed_occupancy_query_is_not_kept(tmp_path):
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(SPLIT)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1905_10759_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["1", "8", "8", "0", "1"]


PLAN = r"""
#include <cstdio>
#include <initializer_list>
#include "fold_plan.h"
using namespace hbmm;
int main() {
  const int64_t big = int64_t{1} << 30, rows[] = {1, 127, 129, 25600, 131072, big - 1, big, big + 1, big + 25600, 2 * big - 1, 2 * big, 2 * big + 25600};
  const int64_t words[] = {1, 7, 8, 72, 288};
  int bad = 0, balanced = 0, copied = 0;
  for (int64_t M : rows)
    for (int64_t N : {1, 4, 64, 65, 1000})
      for (int64_t nw : words)
        for (int sub = 0; sub < 2; sub++)
          for (int64_t sms : {1, 74, 132, 148, 256, 300}) {
            const FoldShape f{M, N, nw, N <= 64 ? 64 : 128, sub != 0};
            const size_t have = fold_bytes(f);                     // what the query reports
            const FoldArea area = fold_area(f, have);
            const Runs r = balanced_runs(f, sms, have);
            if (r.pay) {
              balanced++;
              // two slots per CTA, a counter per tile and warp: all there, and zeroed by the call that expands the weights
              bad += !area.slots || !area.counters || area.slots_at + 2 * r.ctas * slot_bytes(f) > have;
              bad += f.tiles() * kEpilogueWarps > kCounterCount || area.at + f.tiles() * kEpilogueWarps * 4 > area.slots_at;
              // a workspace that ends before the last slot keeps the tiles whole
              bad += balanced_runs(f, sms, area.at + balanced_bytes(f) - 1).pay;
            }
            bad += area.counters && area.slots_at > have;
            copied += copies_reach(f);
            bad += copies_reach(f) != (M < 2 * big);
          }
  // 25600 rows in the workspace of 2^30 + 25600: neither slots nor counters that nobody zeroed
  const FoldShape whole{big + 25600, 4, 8, 64, false}, rest{25600, 4, 8, 64, false};
  const FoldArea part = fold_area(rest, fold_bytes(whole));
  bad += part.slots || part.counters || balanced_runs(rest, 148, fold_bytes(whole)).pay || !balanced_runs(rest, 148, fold_bytes(rest)).pay;
  std::printf("%d %d %d %zu", bad, balanced > 0, copied > 0, fold_bytes(whole));
}
"""


def test_folded_launches_stay_in_the_reported_workspace(tmp_path):
    """Products of up to 2^31 rows and more: no launch uses more of the workspace than the query reports, and none counts in
    arrival counters that the call did not zero."""
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(PLAN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_1905_10759_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0", "1", "1", "65792"]


def test_stream_handle_without_private_functions(monkeypatch):
    from paper_1905_10759_b200 import hbmm

    class Stream:
        cuda_stream = 7

    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: Stream())
    monkeypatch.setattr(hbmm, "_device_index", lambda: 3)
    for raw, want in ((lambda device: 40 + device, 43), (None, 7)):
        monkeypatch.setattr(hbmm, "_raw_stream", raw)
        assert hbmm._stream(None) == want
        assert hbmm._stream(Stream()) == 7
