"""The plans without composite radices (the float-float passes', make_plan(M, p, false)) through the
general transform of csrc/common.cuh, on the CPU: every length that the runtime-plan test has, and
lengths with high powers of two alone and next to other factors (GaNi transforms as long as an
even grid), full and pruned, the divisions prepared in the plan or not. Every radix of a plan has a
stage: 2, 4, 8, the odd ones up to 15 that are butterflies, or a prime above 13.

Tolerance as in test_fft_plan_host: 2.3e-16 (8 log2 M + M / 2) of the largest output.
"""
import math
import shutil
import subprocess

import pytest

from test_ffloat_host import CSRC, FFT_SHIM_EXTRA, SHIM
from test_fft_plan_host import DRIVER, LENGTHS

ALL = LENGTHS + [10, 14, 20, 24, 26, 32, 36, 40, 48, 68, 80, 96, 100, 112, 128, 136, 144, 160, 192, 208, 240, 256, 272]

SMALL = """double2* res = big ? fft_pencils<double>(a.data(), b.data(), G, ld, plan, W.data(), dir, band)
                     : fft_pencils_small<double>(a.data(), b.data(), G, ld, plan, W.data(), dir);"""
assert SMALL in DRIVER
MAIN = r"""
static bool has_stage(int r, bool big) {
  if (r == 9 || r == 15) return big;
  for (int k : {2, 3, 4, 5, 7, 8, 11, 13}) if (r == k) return true;
  for (int p = 2; p * p <= r; ++p) if (r % p == 0) return false;
  return r > 13;
}
int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    const int M = std::atoi(argv[i]);
    bool ok = true;
    double worst = 0;
    for (int big = 0; big < 2; ++big) {
      FftPlan p{};
      make_plan(M, p, big != 0);
      int prod = 1;
      for (int s = 0; s < p.nrad; ++s) { prod *= p.radix[s]; ok = ok && has_stage(p.radix[s], big != 0); }
      ok = ok && prod == M;
    }
    for (int dir : {-1, 1})
      for (int prepared = 0; prepared < 2; ++prepared)
        for (int N : {0, (M + 1) / 2, (M + 1) / 2 - 1, (M + 4) / 5})
          if (N >= 0) worst = std::fmax(worst, check(M, dir, N, false, prepared != 0));
    std::printf("%.3e %d\n", worst, ok ? 1 : 0);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("ff_plan")
    (d / "cuda_runtime.h").write_text(SHIM + FFT_SHIM_EXTRA)
    check = DRIVER[:DRIVER.index("static bool smooth_odd")].replace(
        SMALL, "double2* res = fft_pencils<double>(a.data(), b.data(), G, ld, plan, W.data(), dir, band);")
    (d / "main.cpp").write_text(check + MAIN)
    exe = d / "ffplancheck"
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", str(d), "-I", CSRC, str(d / "main.cpp"), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)] + [str(m) for m in ALL], check=True, capture_output=True, text=True).stdout
    rows = [line.split() for line in out.splitlines()]
    return {m: (float(r[0]), r[1] == "1") for m, r in zip(ALL, rows)}


@pytest.mark.parametrize("M", ALL)
def test_plan_without_composite_radices(results, M):
    worst, ok = results[M]
    assert ok, M
    assert worst <= 2.3e-16 * (8 * math.log2(max(M, 2)) + M / 2), (M, worst)
