"""How much memory a call's faster, larger layout may take (ozg_planes.h, compiled for the host): what the
workspace already has, and of what the least layout leaves free a quarter."""
import os
import random
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2503_22875_gb300", "csrc", "ozg_planes.h")
HARNESS = r"""
#include <cstdio>
#define __host__
#define __device__
#include "HEADER"
int main() {
  unsigned long long cap, lean, bytes, free_bytes;
  while (std::scanf("%llu %llu %llu %llu", &cap, &lean, &bytes, &free_bytes) == 4)
    std::printf("%d %llu\n", (int)ozg::layout_room(cap, lean, bytes, free_bytes),
                (unsigned long long)ozg::workspace_size(bytes));
  return 0;
}
"""
MB, GB = 1 << 20, 1 << 30


def test_larger_layouts_leave_three_quarters_of_the_free_memory(tmp_path):
    src, exe = tmp_path / "room.cpp", tmp_path / "room"
    src.write_text(HARNESS.replace("HEADER", HEADER))
    subprocess.run(["g++", "-O1", "-std=c++17", str(src), "-o", str(exe)], check=True)
    g = random.Random(3)
    cases = [(0, 400 * MB, 900 * MB, 250 * GB), (0, 400 * MB, 900 * MB, 1536 * MB), (2 * GB, 400 * MB, 900 * MB, 0),
             (0, 400 * MB, 400 * MB, 0), (0, 60 * GB, 61 * GB, 68 * GB), (0, 5 * GB, 5 * GB + 100 * MB, 4 * GB),
             (450 * MB, 400 * MB, 900 * MB, 1536 * MB), (0, 1, 2, 0)]
    for _ in range(3000):
        lean = int(2 ** g.uniform(10, 38))
        cases.append((g.choice([0, lean, int(2 ** g.uniform(20, 38))]), lean, int(lean * g.uniform(1, 9)),
                      int(2 ** g.uniform(20, 38))))
    out = subprocess.run([str(exe)], input="".join("%d %d %d %d\n" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.split()
    allowed = [x == "1" for x in out[::2]]
    sizes = [int(x) for x in out[1::2]]
    assert allowed[:8] == [True, False, True, True, False, False, False, True]
    for (cap, lean, size, free), ok, want in zip(cases, allowed, sizes):
        assert want >= size * 9 // 8 and want % MB == 0
        least = max(cap, -(-(lean + lean // 8) // MB) * MB if lean > cap else cap)
        left = cap + free - least  # free with the least layout
        if size <= cap:
            assert ok
        elif ok and want > least:  # what the program keeps
            assert left >= 0 and cap + free - want >= left - left // 4 - 1
        elif not ok:
            assert want - least > left // 4
