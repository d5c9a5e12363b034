"""The ring that hands positions from the chain to the absorbing warps (csrc/rt_handover.h): every order in which the warps can
run, with mbarriers that answer parities, is walked through on the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# A state is the progress of the chain (hand-overs published) and of each absorbing warp (hand-overs absorbed).  An mbarrier whose
# current phase is the c-th lets a wait for parity p through when (c & 1) != p.
PROGRAM = r"""
#include <array>
#include <cstdio>
#include <set>
#include <vector>
#include "rt_handover.h"

struct OneReadyBarrier : rt::Handover {                       // the scheme with a single ready barrier
  static constexpr int kReadyBars = 1;
  static constexpr int ready_bar(int) { return 0; }
  static constexpr unsigned ready_parity(int j) { return (unsigned)j & 1u; }
};

constexpr int kWarps = 4, kCount = 14;

template <class S> int walk() {                                // 0: sound, 1: a state that nobody leaves, 2: an entry that is not the awaited one
  using State = std::array<int, kWarps + 1>;                   // chain, warps
  std::set<State> seen;
  std::vector<State> todo{State{}};
  while (!todo.empty()) {
    const State s = todo.back();
    todo.pop_back();
    if (!seen.insert(s).second) continue;
    bool moved = false, done = s[0] == kCount;
    auto read_phases = [&](int slot) {                         // completed phases of a read barrier: entries that all warps have read
      int n = 0;
      for (int j = slot; j < kCount; j += S::kSlots) {
        int readers = 0;
        for (int w = 1; w <= kWarps; ++w) readers += s[w] > j;
        if (readers < kWarps) break;
        ++n;
      }
      return n;
    };
    if (s[0] < kCount) {
      const int j = s[0];
      if (j < S::kSlots || (unsigned)(read_phases(S::slot(j)) & 1) != S::read_parity(j - S::kSlots)) {
        State n = s;
        ++n[0];
        for (int w = 1; w <= kWarps; ++w)
          if (j >= S::kSlots && s[w] <= j - S::kSlots) return 2;                             // overwrites an entry still to be read
        todo.push_back(n);
        moved = true;
      }
    }
    for (int w = 1; w <= kWarps; ++w) {
      done = done && s[w] == kCount;
      if (s[w] == kCount) continue;
      const int j = s[w];
      int phases = 0;                                          // completed phases of the ready barrier it waits on
      for (int k = 0; k < s[0]; ++k) phases += S::ready_bar(k) == S::ready_bar(j);
      if ((unsigned)(phases & 1) == S::ready_parity(j)) continue;
      if (s[0] <= j) return 2;                                 // let through before the entry was there
      State n = s;
      ++n[w];
      todo.push_back(n);
      moved = true;
    }
    if (!moved && !done) return 1;
  }
  return 0;
}

int main() { std::printf("%d %d\n", walk<rt::Handover>(), walk<OneReadyBarrier>()); }
"""


def test_no_order_of_the_warps_stops_the_ring(tmp_path):
    src = tmp_path / "walk.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "walk"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2604_21215_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    ring, one_barrier = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert ring == "0"
    assert one_barrier != "0"                                  # (the walk does find the dead end of a single ready barrier)


def test_both_kernels_use_the_ring():
    for name in ("rt_leaf_small.cu", "rt_backward_loop.cu"):
        text = open(os.path.join(ROOT, "paper_2604_21215_b200", "csrc", name)).read()
        for call in ("Handover::ready_bar(", "Handover::ready_parity(", "Handover::read_parity("):
            assert call in text, (name, call)
