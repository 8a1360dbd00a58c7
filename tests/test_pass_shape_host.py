"""The launch shape of the packed FP32 row pass (csrc/passes.cuh, xpair_shape) on the CPU, for every
transform length: a launch fits the shared memory and its threads the kernel's bound, and on a
grid large enough to fill the GPU a CTA's rows fill its double pencils of four wherever
two planes can share one."""
import os
import shutil
import subprocess

import pytest

from test_ffloat_host import CSRC

DRIVER = r"""
#include <algorithm>
#include <cstddef>
#include <cstdio>
constexpr size_t kPassSmemBudget = 48 * 1024;
constexpr int kPassThreads = 256;
%s
int main(int argc, char**) {
  if (argc > 1) {   // chunks of a pass: budget's chunk, positions, CTAs beside, rows; and what they become
    for (int rows = 0; rows <= 3; ++rows)
      for (int others : {1, 2, 3, 4, 9, 40, 151, 400})
        for (int n : {1, 2, 3, 12, 57, 102, 276, 405, 2025, 6561})
          for (int chunk : {1, 2, 3, 7, 22, 33, 64})
            std::printf("%%d %%d %%d %%d %%lld\n", rows, others, n, chunk, spread_chunk(chunk, n, others, rows, 1200));
    return 0;
  }
  for (int rpp = 2; rpp <= 3; ++rpp)
    for (int M = 1; M <= 4097; M += 2) {
      const XPairShape big = xpair_shape(M, rpp, 100000, rpp), one = xpair_shape(M, rpp, 1, rpp);
      std::printf("%%d %%d %%d %%d %%zu %%d\n", rpp, M, big.yb, big.threads, xpair_smem(M, big.yb * rpp), one.yb);
    }
  return 0;
}
"""


@pytest.fixture(scope="module")
def shapes(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = open(os.path.join(CSRC, "passes.cuh")).read()

    def cut(start, end):
        i = src.index(start)
        return src[i:src.index(end, i)]
    parts = (cut("constexpr int kXPairThreads", "template") + cut("constexpr long long kSpreadCtas", "template") +
             cut("inline size_t xpair_smem", "template"))
    d = tmp_path_factory.mktemp("shape")
    (d / "main.cpp").write_text(DRIVER % parts)
    subprocess.run([cxx, "-std=c++17", "-O1", str(d / "main.cpp"), "-o", str(d / "shape")], check=True)

    def run(*args):
        out = subprocess.run([str(d / "shape"), *args], check=True, capture_output=True, text=True).stdout
        return [tuple(map(int, line.split())) for line in out.splitlines()]
    return run


def test_launches_fit(shapes):
    for rpp, M, yb, threads, smem, one in shapes():
        if yb > 0:
            assert 64 <= threads <= 256 and smem <= 227 * 1024 and yb <= 32, (rpp, M)
        assert one in (0, 1), (rpp, M)


def test_rows_fill_their_double_pencils(shapes):
    for rpp, M, yb, threads, smem, one in shapes():
        if rpp == 2:
            assert (yb > 0) == (M <= 2346), M
            assert yb % 2 == 0, M
        else:
            assert (yb > 0) == (M <= 438 or 877 < M <= 2346), M
            assert yb >= 4 or M > 438, M   # four planes are three whole groups


def test_spread_chunks(shapes):
    """Within the budget's chunk; and, where a pipe bounds the pass, no SM with more pencils than
    that chunk leaves it."""
    for rows, others, n, chunk, got in shapes("spread"):
        assert 1 <= got <= chunk, (rows, others, n, chunk)

        def ctas(c):
            return -(-n // c) * others

        def fullest(c):
            return -(-ctas(c) // 152) * ((c * rows + 1) // 2)
        if chunk < 2 or ctas(chunk) >= 304:
            assert got == chunk
        elif rows:
            assert fullest(got) <= fullest(chunk), (rows, others, n, chunk, got)
