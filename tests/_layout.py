"""Sizes of the PCG kernels' shared-memory layouts, from the library's own header (compiled by nvcc for the host)."""
import functools
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2309_06427_gb300", "csrc")
STATIC_SMEM = 4 * 32 * 8 + 16  # static shared memory of the PCG kernels: what a launch may take is the device's limit less this

PROGRAM = r'''
#include <cstdio>
#include <cstdlib>
#include "kernels.h"
using namespace sspcg;
// op nx nu budget (bytes) -> the largest N whose problem fits whole: in the kernel with a thread per row pair (at most
// 512 pairs), in the general kernel; bytes of the former's layout at its N
int main(int, char **v) {
  const int op = std::atoi(v[1]), nx = std::atoi(v[2]), nu = std::atoi(v[3]);
  const long long budget = std::atoll(v[4]);
  int one = -1, general = -1;
  for (int N = 0; N <= 4096; ++N) {
    if (pcg_one_ok(op, false, kRedDf, 0, 0, 512, budget, N, nx, nu)) one = N;
    if (pcg_layout(op, N + 1, N, nx, nu).total * 4 <= budget) general = N;
  }
  std::printf("%d %d %lld\n", one, general, one < 0 ? 0LL : 4LL * pcg_one_layout(op, one, nx, nu).total);
}
'''


@functools.lru_cache(None)
def _program():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    folder = tempfile.mkdtemp()
    src, exe = os.path.join(folder, "sizes.cu"), os.path.join(folder, "sizes")
    with open(src, "w") as f:
        f.write(PROGRAM)
    r = subprocess.run([nvcc, "-std=c++17", "-O1", f"-I{CSRC}", src, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return exe


@functools.lru_cache(None)
def largest(op, nx, nu, budget):
    """(N of the row-pair kernel, N of the general kernel, bytes of the former); op: 0 block form, 1 QP form."""
    out = subprocess.run([_program(), str(op), str(nx), str(nu), str(budget)], capture_output=True, text=True)
    assert out.returncode == 0, out.stderr
    return tuple(int(v) for v in out.stdout.split())
