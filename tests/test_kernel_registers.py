"""Registers of the gather kernels whose speed is their number of resident blocks: four blocks of 128
threads per SM need at most 128 registers a thread, and none of them may be spilled for it."""
import os
import re
import subprocess

import pytest

from paper_2206_14735_gb300 import build as gbuild

KERNELS = [("gs_paper.cu", "paper_query_kernel"), ("gs_pose.cu", "eikonal_pose_kernelILb0ELb0E")]


@pytest.mark.parametrize("source,kernel", KERNELS, ids=[k for _, k in KERNELS])
def test_four_blocks_per_sm(source, kernel, tmp_path):
    r = subprocess.run([gbuild.nvcc(), *gbuild.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I", gbuild.INCLUDE,
                        "-I", gbuild.CSRC, "-Xptxas", "-v", "-c", os.path.join(gbuild.CSRC, source), "-o",
                        str(tmp_path / "k.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    report = re.search(kernel + r".*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers",
                       r.stdout + r.stderr, re.S)
    assert report, r.stderr
    stores, loads, registers = (int(v) for v in report.groups())
    assert stores == 0 and loads == 0 and registers <= 128, (stores, loads, registers)
