"""The split trace's walk from tile to tile, its step taken from the kernel's
source (as a function of its own it made the kernel 3 % slower) for the host:
every ray leaves the grid within its tiles' count, also one whose origin or
direction has become infinite or NaN and grids so wide that they overflow."""
import os
import subprocess

import pytest

from paper_1912_03998_gb300 import build_lib

PROGRAM = r"""
#include <math.h>
#include <stdio.h>
#include "bt_internal.cuh"
using bt::kInf;
static bool leave(const bt::TileGrid &tg, const bt::Ray &r, int &ix, int &iy) {
  bool leaves;
  STEP
  return leaves;
}
int main() {
  const float big = 3.4e38f, inf = INFINITY;
  const float v[] = {0.0f, 1.0f, -1.0f, 0.6f, 17.5f, big, -big, inf, -inf, NAN, 1e-25f, -1e-25f};
  const float w[] = {10.0f, 1e-3f, inf};
  const int n = sizeof(v) / sizeof(v[0]);
  long bad = 0, walks = 0;
  for (int a = 0; a < n * n * n * n; a++)
    for (float wx : w)
      for (float gx0 : {0.0f, -big}) {
        bt::TileGrid tg = {gx0, 0.0f, wx, 10.0f, gx0 + 4 * wx, 50.0f, 4, 5};
        bt::Ray r;
        r.o = float3{v[a % n], v[a / n % n], 0.0f};
        r.d = float3{v[a / (n * n) % n], v[a / (n * n * n)], 0.0f};
        auto inv = [](float d) { return 1.0f / (fabsf(d) > 1e-20f ? d : copysignf(1e-20f, d)); };
        r.inv = float3{inv(r.d.x), inv(r.d.y), inv(r.d.z)};
        for (int start = 0; start < 20; start++, walks++) {
          int ix = start % 4, iy = start / 4, steps = 0;
          while (!leave(tg, r, ix, iy) && ++steps <= 20) {}
          bad += steps > 20;
        }
      }
  printf("%ld %ld\n", bad, walks);
  return 0;
}
"""


def test_every_ray_leaves_the_grid(tmp_path):
    try:
        nvcc = build_lib.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "walk.cu", tmp_path / "walk"
    kernel = open(os.path.join(build_lib.CSRC, "trace.cu")).read()
    begin = kernel.index("float tex = kInf, tey = kInf;", kernel.index("k_trace_tiled("))
    step = kernel[begin:kernel.index("if (leaves || root_reachable", begin)]
    src.write_text(PROGRAM.replace("STEP", step))
    subprocess.run([nvcc, "-std=c++17", f"-I{build_lib.INCLUDE}", f"-I{build_lib.CSRC}", *build_lib.ARCH, str(src),
                    "-o", str(exe)], check=True)
    bad, walks = map(int, subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split())
    assert walks > 2000000 and bad == 0
