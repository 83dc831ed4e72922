"""The waits of the render kernels' tile groups, on barriers that a ninth warp of the test arrives on
in place of the tensor-core products: no tensor-core instruction is issued, every wait is bounded."""
import subprocess

import pytest

from paper_2206_14735_gb300 import build as gbuild

pytestmark = pytest.mark.gpu


def run_program(tmp_path, source):
    src, exe = tmp_path / "waits.cu", tmp_path / "waits"
    src.write_text(source)
    subprocess.check_call([gbuild.nvcc(), *gbuild.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                           gbuild.INCLUDE, "-I", gbuild.CSRC, str(src), "-o", str(exe)])
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


COMMON = r"""
#include <cstdio>
#include "gs_render_tc.cuh"
using namespace gs;
__device__ void arrive(uint64_t* mbar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(mbar)) : "memory");
}
__device__ void pause(long long cycles) {
  const long long t0 = clock64();
  while (clock64() - t0 < cycles) {
  }
}
"""

CONVERGE = COMMON + r"""
// Lanes reach the wait at different times, before and after its completion; behind it the warp is one.
__global__ void run(unsigned* split) {
  __shared__ TileBars bars;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bars.done, 1);
    tc::mbar_init(&bars.dw, 1);
    tc::fence_mbar_init();
    bars.abort = 0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  if (threadIdx.x >= kTileThreads) {
    for (int k = 0; k < 64; ++k) {
      if (lane == 0) {
        pause(4000 + 911 * (k % 7));
        arrive(&bars.dw);
      }
      __syncwarp();
      group_sync<kTileThreads + 32>(1);  // the group has seen this completion
    }
    return;
  }
  Tile T;
  T.bars = &bars;
  T.g = 0;
  T.w8 = threadIdx.x >> 5;
  T.ph_done = T.ph_dw = 0;
  for (int k = 0; k < 64; ++k) {
    T.dw_pending = true;
    pause((lane * (k + 3) % 32) * 300);
    tiles_free(T);
    if (__activemask() != 0xffffffffu) atomicAdd(split, 1u);
    group_sync<kTileThreads + 32>(1);
  }
  if (bars.abort) atomicAdd(split, 1u);
}
int main() {
  unsigned *d, h = 1;
  if (cudaMalloc(&d, 4) != cudaSuccess || cudaMemset(d, 0, 4) != cudaSuccess) return 2;
  run<<<1, kTileThreads + 32>>>(d);
  if (cudaMemcpy(&h, d, 4, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  printf("%u threads in a divided warp\n", h);
  return h != 0;
}
"""


def test_a_warp_leaves_the_tile_wait_together(tmp_path):
    run_program(tmp_path, CONVERGE)
