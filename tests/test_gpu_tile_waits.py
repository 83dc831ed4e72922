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


DRAIN = COMMON + r"""
// what the group saw: threads with true, with false, whether the late arrival had come, the status word
struct Seen { int good, bad, arrived, status; };
// scenario 0: every product complete; 1: the weight-gradient products never do; 2: a phase wait ran out
// before, its products complete 1 ms late; 3: weight-gradient products 1 ms late, within the wait; 4: a
// wait for the weight-gradient products ran out before, they complete 1 ms late; 5: and so did the wait
// for the next phase's, both come late, one after the other
__global__ void run(int scenario, Seen* out) {
  __shared__ TileBars bars;
  __shared__ volatile int came;
  if (threadIdx.x == 0) {
    tc::mbar_init(&bars.done, 1);
    tc::mbar_init(&bars.dw, 1);
    tc::fence_mbar_init();
    bars.abort = scenario == 2 || scenario >= 4;
    came = 0;
  }
  __syncthreads();
  if (threadIdx.x >= kTileThreads) {  // the ninth warp
    if (threadIdx.x == kTileThreads && scenario >= 2) {
      for (int k = 0; k < (scenario == 5 ? 2 : 1); ++k) {
        pause(2000000);
        came = k + 1;
        __threadfence_block();
        arrive(scenario == 2 ? &bars.done : &bars.dw);
      }
    }
    return;
  }
  Tile T;
  T.bars = &bars;
  T.g = 0;
  T.w8 = threadIdx.x >> 5;
  T.ph_done = scenario == 2 ? 1u : 0u;  // a phase wait flips it, also when it runs out
  T.ph_dw = scenario == 4 ? 1u : 0u;  // a wait flips it, also when it runs out
  T.dw_pending = scenario == 1 || scenario == 3;
  const bool ok = tile_end(T, &out->status, 64);
  group_sync<kTileThreads>(0);  // the caller's barrier
  atomicAdd(ok ? &out->good : &out->bad, 1);
  if (threadIdx.x == 0) out->arrived = came;
}
int main() {
  const int want[6][4] = {{256, 0, 0, 0}, {0, 256, 0, 64}, {0, 256, 1, 64}, {256, 0, 1, 0}, {0, 256, 1, 64}, {0, 256, 2, 64}};
  Seen* d;
  if (cudaMalloc(&d, sizeof(Seen)) != cudaSuccess) return 2;
  for (int s = 0; s < 6; ++s) {
    Seen h;
    cudaMemset(d, 0, sizeof(Seen));
    run<<<1, kTileThreads + 32>>>(s, d);
    if (cudaMemcpy(&h, d, sizeof(Seen), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
    const int got[4] = {h.good, h.bad, h.arrived, h.status};
    printf("%d: %d %d %d %d\n", s, got[0], got[1], got[2], got[3]);
    for (int k = 0; k < 4; ++k)
      if (got[k] != want[s][k]) return 1;
  }
  return 0;
}
"""


def test_a_wait_that_runs_out_is_reported_and_drained(tmp_path):
    run_program(tmp_path, DRAIN)
