"""The adjoint evaluator's entry numbers are shared by a warp (WarpInts of
pc_adjoint.cuh: every lane writes the same number and reads it later).  The
struct's own text runs here on 32 host threads, with __syncwarp as a barrier
and one lane held back before each of its reads: every lane must read what
was written, however far the others run ahead."""
import os
import re
import subprocess

import pytest

from conftest import ROOT

HARNESS = r"""
#include <barrier>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#define __device__
#define __forceinline__ inline
static std::barrier<> warp(32);
static void __syncwarp() { warp.arrive_and_wait(); }
%s
int main() {
  std::vector<int> mem(8, -1), bad(32, 0);
  std::vector<std::thread> lanes;
  for (int lane = 0; lane < 32; ++lane)
    lanes.emplace_back([&, lane] {
      const WarpInts w{mem.data()};
      for (int i = 0; i < 12; ++i) {
        for (int s = 0; s < 8; ++s) w.set(s, 100 * i + s);
        if (lane == i) std::this_thread::sleep_for(std::chrono::milliseconds(20));
        for (int s = 7; s >= 0; --s) bad[lane] += w.get(s) != 100 * i + s;
      }
    });
  for (auto &t : lanes) t.join();
  int n = 0;
  for (int b : bad) n += b;
  std::printf("%%d\n", n);
}
"""


def test_a_lane_behind_reads_its_own_numbers(tmp_path):
    src = open(os.path.join(ROOT, "paper_2108_03076_gb300", "csrc", "pc_adjoint.cuh")).read()
    struct = re.search(r"^struct WarpInts \{.*?^\};", src, re.S | re.M).group(0)
    cpp, exe = tmp_path / "warp.cpp", tmp_path / "warp"
    cpp.write_text(HARNESS % struct)
    subprocess.run(["g++", "-std=c++20", "-O0", "-pthread", str(cpp), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120, check=True).stdout
    assert int(out) == 0, f"{out.strip()} stale reads"
