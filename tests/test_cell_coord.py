"""The division-free cell coordinate (gs::cell_coord) against the binary32 division it stands for,
on the host: the quotient of every finite distance and voxel edge, bit for bit."""
import os
import subprocess

import pytest

from paper_2206_14735_gb300 import build as gbuild

PROGRAM = r"""
#include <cstdint>
#include <cstdio>
#include <cstring>
#include "gs_device.cuh"
static uint64_t s = 88172645463325252ull;
static uint64_t rnd() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return s; }
static float bits(uint32_t u) { float f; memcpy(&f, &u, 4); return f; }
static uint32_t word(float f) { uint32_t u; memcpy(&u, &f, 4); return u; }
int main(int, char** argv) {
  const int mode = argv[1][0] - '0';
  const float fixed[10] = {0.96f, 0.24f, 0.06f, 0.02f, 0.64f, 0.08f, 1.0f, 0.1f, 3.0f, 16777215.0f};
  long long bad = 0, seen = 0;
  for (int k = 0; k < 400; ++k) {
    float v = fixed[k % 10];
    if (mode == 1) v = ldexpf(1.0f + (rnd() & 0x7fffff) * 0x1p-23f, (int)(rnd() % 40) - 20);
    if (mode == 2) v = bits((uint32_t)(rnd() % 0x7f800000u));  // any positive edge, subnormal ones too
    if (!(v > 0.f)) continue;
    gs::GridDesc g;
    gs::set_voxel(g, 0, v);
    for (int i = 0; i < 20000; ++i) {
      const uint32_t u = (uint32_t)rnd();
      float d = bits(u);                                                          // any value, infinities and NaN
      if (i & 1) d = ldexpf(1.0f + (u & 0x7fffff) * 0x1p-23f, (int)(u >> 23) % 36 - 30);
      if (i % 3 == 0) d = bits(word((float)(u % 4096) * v) + (int)(rnd() % 3) - 1);  // at a cell's edge
      const float a = d / v, b = gs::cell_coord(d, g.div_scale[0], g.div_voxel[0], g.div_recip[0]);
      ++seen;
      if (isnan(a) ? isnan(b) : word(a) == word(b)) continue;
      if (fabsf(a) >= 0x1p100f && fabsf(b) >= 0x1p99f && signbit(a) == signbit(b)) continue;  // far outside any grid
      if (fabsf(a) < 0x1p-90f && fabsf(b) < 0x1p-90f) continue;                            // at the grid's face
      ++bad;
    }
  }
  printf("%lld of %lld differ\n", bad, seen);
  return bad != 0 || seen == 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("cell")
    src = d / "cell.cu"
    src.write_text(PROGRAM)
    exe = d / "cell"
    subprocess.check_call([gbuild.nvcc(), *gbuild.ARCH, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off",
                           "-I", gbuild.INCLUDE, "-I", gbuild.CSRC, str(src), "-o", str(exe)])
    return str(exe)


@pytest.mark.parametrize("mode", [0, 1, 2], ids=["workload edges", "metre-scale edges", "any edge"])
def test_cell_coord_is_the_division(program, mode):
    r = subprocess.run([program, str(mode)], capture_output=True, text=True, env=dict(os.environ))
    assert r.returncode == 0, r.stdout
