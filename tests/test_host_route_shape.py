"""The chain router's launch shape, without a GPU: the host header compiled by itself."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include "route_shape.h"
#include <algorithm>
#include <cstdio>
int main() {
  // group, split, warps along the experts, chains per thread: the kernel's forms
  const int forms[][4] = {{16, 1, 4, 1}, {16, 1, 8, 1}, {2, 1, 2, 1}, {2, 2, 4, 1}, {16, 1, 2, 2}, {16, 1, 4, 2}, {2, 1, 1, 2},
                          {2, 1, 2, 2}, {2, 3, 2, 2}, {2, 4, 2, 2}, {8, 1, 2, 8}, {8, 3, 2, 8}, {8, 4, 2, 8}};
  for (const auto& f : forms)
    for (int H : {64, 1024, 7168})
      for (int T = 1; T <= 40000; T += 1 + T / 300) {
        const int group = f[0], split = f[1], ew = f[2], chains = f[3], max_tw = 24 / ew, sms = 148;
        const int tw = moehub::route_token_warps(T, H, group, split, ew, chains, max_tw, sms);
        if (tw < 1 || tw > max_tw) return 1;
        const long long ctas = (long long)((T + group * tw - 1) / (group * tw)) * split, waves = (ctas + sms - 1) / sms;
        // Warps of an SM scheduler over all waves (at least one and a half per wave: a chain's latency) against an even
        // share of all warps, rounded up to whole waves of the fullest CTAs.
        const double spent = (double)waves * std::max(1.5, ew * tw / 4.0);
        const double even = (double)((T + group - 1) / group) * split * ew / (4.0 * sms);
        if (spent > 1.6 * even + std::max(1.5, ew / 2.0) + 6.0 * (even > ew * max_tw / 4.0)) {
          std::printf("T %d H %d form %d %d %d %d: tw %d, %lld waves, %.1f against %.1f\n", T, H, group, split, ew, chains, tw, waves, spent, even);
          return 2;
        }
      }
  return 0;
}
"""


def test_no_batch_falls_into_many_waves_of_small_ctas(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", os.path.join(ROOT, "paper_2605_05888_b200", "csrc"), str(src), "-o", str(exe)], check=True)
    got = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert got.returncode == 0, got.stdout
