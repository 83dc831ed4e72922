"""The cell coordinate without a division (gs::cell_coord) as the device computes it, against __fdiv_rn:
bit for bit on pseudo-random distances of the size that a grid has and at the cells' edges.  Quotients
below 2^-90 (on a grid's face) and from 2^100 on (far outside of it, clamped) may differ and are left
out, as in the host's test."""
import subprocess

import pytest

from paper_2206_14735_gb300 import build as gbuild

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "gs_device.cuh"
__device__ unsigned mix(unsigned x) {
  x ^= x >> 16, x *= 0x7feb352du, x ^= x >> 15, x *= 0x846ca68bu;
  return x ^ (x >> 16);
}
__global__ void compare(gs::GridDesc g, int l, unsigned long long* out) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x, r = mix(i * 4u + l + 1u);
  float d = ldexpf(1.0f + (r & 0x7fffffu) * 0x1p-23f, (int)(r >> 23) % 24 - 16);
  if (i & 1) d = __int_as_float(__float_as_int((float)(r % 4096u) * g.voxel[l]) + (int)(mix(r) % 5u) - 2);
  if (i & 2) d = -d;
  const float a = __fdiv_rn(d, g.voxel[l]), b = gs::cell_coord(d, g.div_scale[l], g.div_voxel[l], g.div_recip[l]);
  if (!(fabsf(a) >= 0x1p-90f && fabsf(a) < 0x1p100f)) return;
  atomicAdd(out, 1ull);
  if (__float_as_int(a) != __float_as_int(b)) atomicAdd(out + 1, 1ull);
}
int main() {
  const float edges[16] = {0.96f, 0.24f, 0.06f, 0.02f, 0.64f, 0.32f, 0.16f, 0.08f,
                           0.1f,  0.03f, 1.0f,  3.0f,  0.7f,  0.005f, 1.9999999f, 1.0000001f};
  unsigned long long *d, h[2] = {0, 1};
  if (cudaMalloc(&d, 16) != cudaSuccess || cudaMemset(d, 0, 16) != cudaSuccess) return 2;
  for (int k = 0; k < 16; ++k) {
    gs::GridDesc g{};
    for (int l = 0; l < gs::kLevels; ++l) gs::set_voxel(g, l, edges[k]);
    for (int l = 0; l < gs::kLevels; ++l) compare<<<4096, 256>>>(g, l, d);
  }
  if (cudaMemcpy(h, d, 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  printf("%llu of %llu differ\n", h[1], h[0]);
  return h[1] != 0 || h[0] < (1ull << 25);
}
"""


def test_device_cell_coord_is_the_division(tmp_path):
    src, exe = tmp_path / "cell.cu", tmp_path / "cell"
    src.write_text(PROGRAM)
    subprocess.check_call([gbuild.nvcc(), *gbuild.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                           gbuild.INCLUDE, "-I", gbuild.CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
