"""The look-ahead of the FP16 kernel's issuing warp: whether the next unit's scores can be issued before this unit's weights are
complete has to have one answer in all lanes, although each looks at the barriers for itself.  Compiled for the host: 32 threads
take the lanes' part, each looking at moments of its own while the barriers' phases end."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")

HARNESS = r"""
#include <atomic>
#include <barrier>
#include <cstdio>
#include <random>
#include <thread>
#include <vector>
#include "bounded_wait.cuh"
int main() {
  constexpr int kLanes = 32, kRounds = 400;
  std::barrier<> sync(kLanes);
  std::atomic<int> vote[kRounds + 1] = {};
  std::vector<std::vector<int>> answer(kLanes, std::vector<int>(kRounds)), saw(answer);
  volatile int abort_word = 0;
  auto lane = [&](int id) {
    std::mt19937 rng(id);
    for (int r = 0; r < kRounds; ++r) {
      // the lane's looks: `first` has come from its look a on, `second` from b on (the same for all lanes, seen at different looks)
      int look = 0, a = (int)(rng() % 6), b = (int)(rng() % 6);
      auto first = [&] { const bool yes = look >= a; saw[id][r] |= yes; return yes; };
      auto second = [&] { return look++ >= b; };
      auto wait = [&](auto probe) { lynx::bounded_wait(probe, [] { return (uint64_t)1; }, &abort_word); };
      auto any = [&](bool x) { if (x) vote[r] = 1; sync.arrive_and_wait(); return vote[r].load() != 0; };
      answer[id][r] = lynx::first_of(wait, first, second, any);
    }
  };
  std::vector<std::thread> t;
  for (int i = 0; i < kLanes; ++i) t.emplace_back(lane, i);
  for (auto& x : t) x.join();
  int split = 0, wrong = 0, mixed = 0;
  for (int r = 0; r < kRounds; ++r) {
    int any = 0, all = 1;
    for (int i = 0; i < kLanes; ++i) { any |= saw[i][r]; all &= saw[i][r]; split += answer[i][r] != answer[0][r]; }
    wrong += answer[0][r] != any;
    mixed += any != all;
  }
  std::printf("%d %d %d", split, wrong, mixed);
}
"""


def test_lanes_that_saw_different_things_answer_alike(tmp_path):
    src, exe = tmp_path / "v.cpp", tmp_path / "v"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O1", "-std=c++20", "-pthread", "-x", "c++", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    split, wrong, mixed = (int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert split == 0 and wrong == 0
    assert mixed > 100, "the lanes see different things in many rounds"


def test_the_issuing_warp_asks_the_vote():
    """Nothing in the issuing warp branches on one lane's own look at a barrier."""
    code = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "attention_f16.cuh")).read())
    warp = code[code.index("if (warp == 20)"):]
    looks = [m.start() for m in re.finditer(r"\bmbar_test\(", warp)]
    ask = re.search(r"if \(first_of\(.*?\[\]\(bool seen\) \{ return __any_sync\(0xFFFFFFFFu, seen\) != 0; \}\)\)\s*qk\(next\+\+\);", warp, re.S)
    assert ask and looks and all(ask.start() < x < ask.end() for x in looks)
