"""The schedule of layers side by side (csrc/rt_wave.h), compiled for the host: every leaf of every layer comes once, after the same leaf of the layer below
and the one before of its own layer, never more than fit; the number of launches is the one that the planner counts with; and planning a call does not
take longer for longer prompts."""
import os
import subprocess
import time

from paper_2604_21215_b200 import rt

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "rt_wave.h"

int main() {
  for (int layers = 1; layers <= rt::kWaveBand; ++layers)
    for (int places = 1; places <= 8; ++places)
      for (int leaves = 1; leaves <= 90; ++leaves) {
        rt::WaveOrder order(layers, leaves);
        std::vector<int> done(layers, 0);
        int layer[8], leaf[8];
        long long launches = 0;
        for (int n; (n = order.next(places, layer, leaf)) > 0; ++launches) {
          const std::vector<int> before = done;
          if (n > places) return 1;
          for (int i = 0; i < n; ++i) {
            if (leaf[i] != before[layer[i]] || done[layer[i]] != before[layer[i]]) return 2;           // its layer's next leaf, once in a launch
            if (layer[i] > 0 && before[layer[i] - 1] <= leaf[i]) return 3;                             // done below in an earlier launch
            ++done[layer[i]];
          }
        }
        for (int l = 0; l < layers; ++l) if (done[l] != leaves) return 4;
        if (launches != rt::wave_launches(layers, leaves, places)) { std::printf("%d layers, %d leaves, %d places\n", layers, leaves, places); return 5; }
      }
  return 0;
}
"""


def test_every_leaf_comes_once_and_in_order(tmp_path):
    src, exe = tmp_path / "wave.cpp", tmp_path / "wave"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2604_21215_b200", "csrc"), "-o", str(exe), str(src)], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, (run.returncode, run.stdout)


def test_planning_takes_no_longer_for_longer_prompts():
    # the call itself plans the same way before its first launch; a walk over the whole schedule took seconds at this length (the best of three calls, which
    # now takes a few microseconds; the loop over the modelled leaves of the counters is what is left)
    cfg = rt.make_config(512, 8, 2048, dtype="bf16")
    best = 1e9
    for _ in range(3):
        t0 = time.perf_counter()
        rt.rt_plan_counters(cfg, 1, 65536, 16)
        best = min(best, time.perf_counter() - t0)
    assert best < 0.02, best
