"""The runtime FFT plans of csrc/common.cuh (lengths without a compile-time kernel) on the CPU.

The header is compiled as host C++ (one thread runs every butterfly of a stage, barriers are
no-ops) and its transforms are compared with DFTs summed in long double, FP64 data, for lengths
over every radix: composite 15 and 9, the odd radices 3 to 13, powers of two, primes above 13
alone and next to other factors; forward and inverse, full and with the zero band's pruned first
(zero-padded inverse) and last (truncating forward) stages, at the smallest and a larger padding,
the batched kernel's form without composite radices (radices 3 to 13 alone) and the divisions
prepared in the plan or not.

Tolerance: a mixed-radix FFT's error is below about 8 eps log2(M) of the DFT's norm, and the
direct prime stages add R / 2 terms, at most R / 2 eps: 2.3e-16 (8 log2 M + M / 2) of the largest
output bounds both.
"""
import os
import shutil
import subprocess

import pytest

from test_ffloat_host import CSRC, FFT_SHIM_EXTRA, SHIM

LENGTHS = [1, 3, 5, 7, 9, 11, 13, 15, 17, 19, 21, 25, 27, 31, 33, 37, 39, 49, 51, 53, 55, 63, 65, 75, 77, 85, 89, 91, 93,
           99, 101, 105, 117, 121, 135, 143, 165, 169, 189, 195, 201, 231, 273, 289, 343, 2, 4, 6, 8, 12, 16, 34, 60, 64]

DRIVER = r"""
#include <cstdio>
#include <cstdlib>
#include <cmath>
#include <vector>
#include "common.cuh"
using namespace homb;
typedef long double LD;
static const LD PI = 3.141592653589793238462643383279502884L;
static uint64_t st = 0x9E3779B97F4A7C15ull;
static double urand() { st ^= st << 13; st ^= st >> 7; st ^= st << 17; return (double)(st >> 11) / 4503599627370496.0 - 1.0; }

// N > 0: N frequencies around 0 are nonzero (inverse) or compared (forward)
static double check(int M, int dir, int N, bool big, bool prepared) {
  FftPlan plan{};
  make_plan(M, plan, big);
  if (!prepared) plan.ndiv = 0;
  const int G = 3, ld = M + 1;
  const int half = N > 0 ? (N - 1) / 2 : 0, top = N > 0 ? N - 1 - half : 0;
  std::vector<double2> W(M), a(G * ld), b(G * ld), x;
  for (int j = 0; j < M; ++j) W[j] = double2{(double)std::cos(-2 * PI * j / M), (double)std::sin(-2 * PI * j / M)};
  for (int g = 0; g < G; ++g)
    for (int p = 0; p < M; ++p) {
      const bool zero = N > 0 && dir > 0 && p > half && p < M - top;
      a[g * ld + p] = zero ? double2{0.0, 0.0} : double2{urand(), urand()};
    }
  x = a;
  const FftBand band{half, top, N > 0 ? (dir > 0 ? 1 : 2) : 0};
  double2* res = big ? fft_pencils<double>(a.data(), b.data(), G, ld, plan, W.data(), dir, band)
                     : fft_pencils_small<double>(a.data(), b.data(), G, ld, plan, W.data(), dir);
  double worst = 0, scale = 0;
  for (int g = 0; g < G; ++g)
    for (int k = 0; k < M; ++k) {
      LD sr = 0, si = 0;
      for (int n = 0; n < M; ++n) {
        const LD ang = dir * 2 * PI * (LD)((long long)n * k % M) / M, c = std::cos(ang), s = std::sin(ang);
        sr += x[g * ld + n].x * c - x[g * ld + n].y * s;
        si += x[g * ld + n].x * s + x[g * ld + n].y * c;
      }
      scale = std::fmax(scale, (double)std::sqrt(sr * sr + si * si));
      if (N > 0 && dir < 0 && k > half && k < M - top) continue;
      const LD er = res[g * ld + k].x - sr, ei = res[g * ld + k].y - si;
      worst = std::fmax(worst, (double)std::sqrt(er * er + ei * ei));
    }
  return worst / scale;
}

static bool smooth_odd(int m) {
  for (int r : {3, 5, 7, 11, 13})
    while (m % r == 0) m /= r;
  return m == 1;
}

int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    const int M = std::atoi(argv[i]);
    double worst = 0;
    for (int dir : {-1, 1})
      for (int big = 0; big < 2; ++big)
        for (int prepared = 0; prepared < 2; ++prepared)
          for (int N : {0, (M + 1) / 2, (M + 1) / 2 - 1, (M + 4) / 5})
            if (N >= 0 && (big || smooth_odd(M))) worst = std::fmax(worst, check(M, dir, N, big != 0, prepared != 0));
    std::printf("%.3e\n", worst);
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("fft_plan")
    (d / "cuda_runtime.h").write_text(SHIM + FFT_SHIM_EXTRA)
    (d / "main.cpp").write_text(DRIVER)
    exe = d / "plancheck"
    subprocess.run([cxx, "-std=c++17", "-O1", "-ffp-contract=off", "-I", str(d), "-I", CSRC, str(d / "main.cpp"), "-o",
                    str(exe)], check=True)
    out = subprocess.run([str(exe)] + [str(m) for m in LENGTHS], check=True, capture_output=True, text=True).stdout
    return dict(zip(LENGTHS, (float(v) for v in out.split())))


@pytest.mark.parametrize("M", LENGTHS)
def test_runtime_plan(errors, M):
    import math
    assert errors[M] <= 2.3e-16 * (8 * math.log2(max(M, 2)) + M / 2), (M, errors[M])
