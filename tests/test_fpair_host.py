"""Radix 3 in the packed FP32 pair type (csrc/fpair.cuh) on the CPU: both halves of a pair are rounded
as single FP32 numbers, and the sine term is one FMA into each sum (one rounding, not two)."""
import shutil
import subprocess

import pytest

from test_ffloat_host import CSRC, SHIM
from test_slab_host import SHIM_EXTRA

DRIVER = r"""
#include <cstdio>
#include "common.cuh"
#include "fpair.cuh"
using namespace homb;
static uint64_t st = 0x9E3779B97F4A7C15ull;
static float urand() { st ^= st << 13; st ^= st >> 7; st ^= st << 17; return (float)((double)(st >> 11) / 4503599627370496.0 - 1.0); }
static float part(fpair p, int h) { return h ? p.v.y : p.v.x; }
int main() {
  const float s3 = (float)0.86602540378443864676372317075294;
  long bad = 0;
  for (int it = 0; it < 20000; ++it)
    for (int dir : {-1, 1}) {
      fpair2 v[3], z[3], o[3];
      for (int k = 0; k < 3; ++k) v[k] = mk<fpair>(fpair(urand(), urand()), fpair(urand(), urand()));
      for (int k = 0; k < 3; ++k) z[k] = o[k] = v[k];
      z[1] = mk<fpair>(fpair(0.f), fpair(0.f));
      const fpair2 w[2][3] = {{v[0], v[1], v[2]}, {z[0], z[1], z[2]}};
      dft3<fpair>(v, dir);
      dft3_mid_in0<fpair>(z, dir);
      dft3_skip_out1<fpair>(o, dir);
      for (int h = 0; h < 2; ++h)
        for (int c = 0; c < 2; ++c) {
          const fpair2* x = w[c];
          const fpair2* y = c ? z : v;
          const float ax = part(x[1].x, h) + part(x[2].x, h), ay = part(x[1].y, h) + part(x[2].y, h);
          const float dx = part(x[1].x, h) - part(x[2].x, h), dy = part(x[1].y, h) - part(x[2].y, h);
          const float tx = std::fmaf(-0.5f, ax, part(x[0].x, h)), ty = std::fmaf(-0.5f, ay, part(x[0].y, h));
          const float p = dir * s3;
          const float e[4] = {std::fmaf(-p, dy, tx), std::fmaf(p, dx, ty), std::fmaf(p, dy, tx), std::fmaf(-p, dx, ty)};
          bad += part(y[1].x, h) != e[0] || part(y[1].y, h) != e[1] || part(y[2].x, h) != e[2] || part(y[2].y, h) != e[3];
          if (!c) bad += part(o[2].x, h) != e[2] || part(o[2].y, h) != e[3];
        }
    }
  std::printf("%ld\n", bad);
  return 0;
}
"""


def test_radix3_sine_terms_are_rounded_once(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(SHIM + SHIM_EXTRA)
    (tmp_path / "main.cpp").write_text(DRIVER)
    exe = tmp_path / "fpair"
    subprocess.run([cxx, "-std=c++20", "-O1", "-ffp-contract=off", "-pthread", "-I", str(tmp_path), "-I", CSRC,
                    str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split() == ["0"]
