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
int main() {
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
    out = subprocess.run([str(d / "shape")], check=True, capture_output=True, text=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_launches_fit(shapes):
    for rpp, M, yb, threads, smem, one in shapes:
        if yb > 0:
            assert 64 <= threads <= 256 and smem <= 227 * 1024 and yb <= 32, (rpp, M)
        assert one in (0, 1), (rpp, M)


def test_rows_fill_their_double_pencils(shapes):
    for rpp, M, yb, threads, smem, one in shapes:
        if rpp == 2:
            assert (yb > 0) == (M <= 2346), M
            assert yb % 2 == 0, M
        else:
            assert (yb > 0) == (M <= 438 or 877 < M <= 2346), M
            assert yb >= 4 or M > 438, M   # four planes are three whole groups
