"""Host-side choices that need no GPU: the split of a tile between CTAs when the occupancy query fails, and the stream handle
the binding passes on."""
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
