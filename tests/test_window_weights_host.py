"""The multiply-add by which a chain's or a pass's int32 sum enters an int64 window word of the
difference-plane kernel (ozg_window.h), compiled for the host with the undefined-behaviour sanitizer:
exact modulo 2^64 for every weight a window has and sums up to the 2^30 of 64 chains."""
import os
import random
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2503_22875_gb300", "csrc", "ozg_window.h")
HARNESS = r"""
#include <cstdint>
#include <cstdio>
#include "HEADER"
int main() {
  unsigned long long W, w;
  int v;
  while (std::scanf("%llu %d %llu", &W, &v, &w) == 3) std::printf("%llu\n", ozg::kd_mac(W, v, ozg::kd_weight(w)));
  for (int n = 0; n < 9; ++n) std::printf("%llu\n", ozg::kd_geom(n));
  return 0;
}
"""


def test_weighted_sums_are_exact_modulo_2_64(tmp_path):
    src, exe = tmp_path / "mac.cpp", tmp_path / "mac"
    src.write_text(HARNESS.replace("HEADER", HEADER))
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all", str(src), "-o",
                    str(exe)], check=True)
    geom = [sum(128 ** j for j in range(n + 1)) for n in range(9)]
    weights = geom + [128 ** n for n in range(9)]
    g = random.Random(7)
    cases = [(g.randrange(2 ** 64), v, w) for w in weights
             for v in [0, 1, -1, 2 ** 24, -2 ** 24, 2 ** 30, -2 ** 30] + [g.randrange(-2 ** 30, 2 ** 30 + 1) for _ in range(40)]]
    run = subprocess.run([str(exe)], input="".join(f"{W} {v} {w}\n" for W, v, w in cases), capture_output=True, text=True)
    assert run.returncode == 0, run.stderr[-500:]
    out = [int(x) for x in run.stdout.split()]
    assert out == [(W + v * w) % 2 ** 64 for W, v, w in cases] + geom
