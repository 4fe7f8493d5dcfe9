"""The cooperative launches' way back (launch_cooperative, csrc/grid.cuh), with
launches faked on the host: refused as too large they are made again with half
the CTAs down to one, and any other answer is final."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

PROGRAM = r"""
#include <cstdio>
#include "grid.cuh"
int main() {
  struct { long grid; unsigned fits; cudaError_t otherwise; } cases[] = {
      {304, 304, cudaSuccess}, {304, 303, cudaSuccess}, {304, 32, cudaSuccess}, {7, 1, cudaSuccess},
      {1, 1, cudaSuccess}, {5, 0, cudaSuccess}, {304, 40, cudaErrorLaunchFailure}};
  for (auto &c : cases) {
    unsigned launched = 0;
    int calls = 0;
    const cudaError_t e = emst::launch_cooperative(c.grid, [&](unsigned g) {
      ++calls;
      if (g > c.fits) return cudaErrorCooperativeLaunchTooLarge;
      launched = g;
      return c.otherwise;
    });
    std::printf("%d %u %d\n", (int)e, launched, calls);
  }
}
"""


@pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc")
def test_refused_launches_shrink(tmp_path):
    src, exe = tmp_path / "launches.cu", tmp_path / "launches"
    src.write_text(PROGRAM)
    subprocess.run([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr",
                    "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2207_00514_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True, timeout=300)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    too_large, failed = 720, 719  # cudaErrorCooperativeLaunchTooLarge, cudaErrorLaunchFailure
    assert [tuple(map(int, x.split())) for x in out.splitlines()] == [
        (0, 304, 1), (0, 152, 2), (0, 19, 5), (0, 1, 4), (0, 1, 1), (too_large, 0, 4), (failed, 38, 4)]
