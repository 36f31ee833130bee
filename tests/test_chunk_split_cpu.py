"""How the build and the steps around the solve cut problems into chunks (csrc/common.cuh), compiled from the library's
own header by nvcc and run on the CPU for a spread of horizons and batch sizes and for every nx and nu:

* the CTAs of a problem take each of its rows once, in chunks no longer than a full one;
* there is a CTA for every problem, and no more than 56 per SM where problems have several;
* a full chunk fits in shared memory."""
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
static int bad = 0;
static void fail(const char *what, long long a, long long b, long long c, long long d) {
  if (bad++ < 20) std::printf("FAIL %s %lld %lld %lld %lld\n", what, a, b, c, d);
}
int main() {
  const int sms = 152;
  for (int full : {1, 4, 9, 15, 64, 213})
    for (int least : {3, 4})
      for (long long nprob : {1LL, 2LL, 40LL, 64LL, 228LL, 456LL, 457LL, 4096LL, 300000LL})
        for (int longest : {0, 1, 2, 3, 20, 64, 65, 128, 513, 4097}) {
          const ChunkSplit s = chunk_split(nprob, sms, longest, full, least);
          if (s.per < 1 || s.share < 1 || s.share > s.per) fail("split", full, nprob, longest, s.per);
          if (s.per > 1 && (long long)s.per * nprob > 56LL * sms) fail("ctas", full, nprob, longest, s.per);
          if (longest > 0 && s.share > cdiv(longest, least)) fail("short chunks", full, nprob, longest, s.share);
          for (int rows : {0, 1, 5, longest / 2, longest}) {
            if (rows > longest) continue;
            const int C = chunk_length(full, rows, s.share);
            if (C < 1 || C > full) fail("length", full, rows, s.share, C);
            long long next = 0;  // chunks in order: part 0, 1, ... per - 1, then part 0 again
            for (int b0 = 0, part = 0; b0 < rows; b0 += C, part = (part + 1) % s.per) {
              int first = part * C;
              while (first < b0) first += s.per * C;
              if (first != b0 || b0 != next) fail("rows", full, rows, s.per, b0);
              next = b0 + C < rows ? b0 + C : rows;
            }
            if (next != rows) fail("cover", full, rows, s.per, next);
          }
        }
  for (int nx = 1; nx <= kMaxNx; ++nx)
    for (int nu = 0; nu <= kMaxNx; ++nu) {
      const int C = chunk_rows(nx, nu);
      if (C < 1 || C * (nx * (nx | 1) + nx * (nu | 1)) > kChunkFloats || C * (nx + nu) > kChunkItems)
        fail("chunk", nx, nu, C, 0);
    }
  std::printf(bad ? "%d failures\n" : "ok\n", bad);
  return bad ? 1 : 0;
}
'''


def test_chunks_cover_their_problems(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "chunks.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "chunks"
    r = subprocess.run([nvcc, "-std=c++17", "-O1", "--expt-relaxed-constexpr", f"-I{CSRC}", str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
