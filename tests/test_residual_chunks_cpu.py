"""Chunks of the true residual (residual_rows in csrc/common.cuh), compiled from the library's own header by nvcc and run
on the CPU for every nx and nu: a chunk fits in the kernel's shared memory and is no shorter than the other kernels'."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2309_06427_gb300", "csrc")

PROGRAM = r'''
#include <cstdio>
#include "common.cuh"
using namespace sspcg;
int main() {
  int bad = 0;
  for (int nx = 1; nx <= kMaxNx; ++nx)
    for (int nu = 0; nu <= kMaxNx; ++nu) {
      const int m = nx + nu, R = residual_rows(nx, nu);
      const bool ok = R >= chunk_rows(nx, nu) && R <= 64 && 2 * R * m + R * nx * ((nx | 1) + (nu | 1)) <= kResFloats &&
                      (R + 1) * nx <= kChunkItems + 2 * kMaxNx;
      if (!ok && bad++ < 20) std::printf("FAIL %d %d %d\n", nx, nu, R);
    }
  std::printf(bad ? "%d failures\n" : "ok\n", bad);
  return bad ? 1 : 0;
}
'''


def test_residual_chunks_fit(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "rows.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "rows"
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", f"-I{CSRC}", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
