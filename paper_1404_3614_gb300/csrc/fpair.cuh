// Two FP32 numbers that every operation treats alike, each in one packed instruction
// (add / mul / fma .f32x2). The transforms are templated on their arithmetic type: with fpair
// one lane transforms two pencils at once. The FP32 pipe does a packed FMA in the time of two
// single ones (80.1 against 78.2 TFLOP/s measured), but in one issue slot, and the index
// arithmetic, twiddles and exchanges of a pencil are shared by two; the register FFTs are bound by
// issue. Each half is rounded as the single FP32 operation is.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"

namespace homb {
// in a namespace of its own, as ffloat: found by argument-dependent lookup
namespace fpa {

struct __align__(8) fpair {
  float2 v;
  fpair() = default;
  __device__ __forceinline__ fpair(float a, float b) { v = make_float2(a, b); }
  __device__ __forceinline__ explicit fpair(float a) { v = make_float2(a, a); }
  __device__ __forceinline__ explicit fpair(double a) { v = make_float2((float)a, (float)a); }
  __device__ __forceinline__ explicit fpair(int a) { v = make_float2((float)a, (float)a); }
};
struct __align__(16) fpair2 {
  fpair x, y;
};
__device__ __forceinline__ fpair fp(float2 v) {
  fpair r;
  r.v = v;
  return r;
}
__device__ __forceinline__ fpair operator-(fpair a) { return fpair(-a.v.x, -a.v.y); }
__device__ __forceinline__ fpair operator+(fpair a, fpair b) { return fp(__fadd2_rn(a.v, b.v)); }
__device__ __forceinline__ fpair operator-(fpair a, fpair b) { return a + (-b); }
__device__ __forceinline__ fpair operator*(fpair a, fpair b) { return fp(__fmul2_rn(a.v, b.v)); }
__device__ __forceinline__ fpair fma(fpair a, fpair b, fpair c) { return fp(__ffma2_rn(a.v, b.v, c.v)); }

}  // namespace fpa

using fpa::fpair;
using fpa::fpair2;
template <> struct cplx_t<fpair> { using type = fpair2; };
template <> struct is_fpair<fpair> { static constexpr bool value = true; };

}  // namespace homb
