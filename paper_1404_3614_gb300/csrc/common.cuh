// Shared device helpers: complex arithmetic, the shared-memory FFT engine,
// deterministic block reductions and the launch-argument structures.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <initializer_list>

namespace homb {

template <typename T> struct cplx_t;
template <> struct cplx_t<double> { using type = double2; };
template <> struct cplx_t<float> { using type = float2; };
}  // namespace homb
#include "ffloat.cuh"
namespace homb {
template <> struct cplx_t<ffloat> { using type = ffloat2; };
template <typename T> using cpx = typename cplx_t<T>::type;
template <typename T> struct is_fpair { static constexpr bool value = false; };   // fpair.cuh

template <typename T> __device__ __forceinline__ cpx<T> mk(T x, T y) { cpx<T> r; r.x = x; r.y = y; return r; }
template <typename T> __device__ __forceinline__ cpx<T> add(cpx<T> a, cpx<T> b) { return mk<T>(a.x + b.x, a.y + b.y); }
template <typename T> __device__ __forceinline__ cpx<T> sub(cpx<T> a, cpx<T> b) { return mk<T>(a.x - b.x, a.y - b.y); }
template <typename T> __device__ __forceinline__ cpx<T> scl(cpx<T> a, T s) { return mk<T>(a.x * s, a.y * s); }
// m + c a for a real c
template <typename T> __device__ __forceinline__ cpx<T> axpy(T c, cpx<T> a, cpx<T> m) {
  return mk<T>(fma(c, a.x, m.x), fma(c, a.y, m.y));
}
#if defined(__CUDA_ARCH__) && !defined(HOMB_SCALAR_COMPLEX)
// FP32: real and imaginary part in one packed instruction (the same rounding; the FP32 pipe does
// a packed FMA at the rate of two single ones, 80.1 against 78.2 TFLOP/s, in half the issue
// slots, which bound the FP32 transforms)
template <> __device__ __forceinline__ float2 add<float>(float2 a, float2 b) { return __fadd2_rn(a, b); }
template <> __device__ __forceinline__ float2 sub<float>(float2 a, float2 b) {
  return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
template <> __device__ __forceinline__ float2 scl<float>(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }
template <> __device__ __forceinline__ float2 axpy<float>(float c, float2 a, float2 m) {
  return __ffma2_rn(make_float2(c, c), a, m);
}
#endif
template <typename T> __device__ __forceinline__ cpx<T> conj_(cpx<T> a) { return mk<T>(a.x, -a.y); }
// a * b
template <typename T> __device__ __forceinline__ cpx<T> mul(cpx<T> a, cpx<T> b) {
  return mk<T>(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}
// a * (b or conj b)
template <typename T> __device__ __forceinline__ cpx<T> mulc(cpx<T> a, cpx<T> b, bool conjb) {
  T by = conjb ? -b.y : b.y;
  return mk<T>(fma(a.x, b.x, -a.y * by), fma(a.x, by, a.y * b.x));
}
// A value as stored between transform stages: float-float pairs renormalised there (their
// sums and products do not renormalise, and a low part left to grow through a whole chain
// of stages would make the rounding error grow with the square of its depth); FP32 and FP64
// values pass unchanged.
template <typename T> __device__ __forceinline__ cpx<T> st_norm(cpx<T> v) {
  if constexpr (is_ff<T>::value) {
    cpx<T> r;
    r.x = ff_norm(v.x);
    r.y = ff_norm(v.y);
    return r;
  } else {
    return v;
  }
}
// i * a  (s = +1) or -i * a (s = -1)
template <typename T> __device__ __forceinline__ cpx<T> rot(cpx<T> a, int s) {
  return s > 0 ? mk<T>(-a.y, a.x) : mk<T>(a.y, -a.x);
}

constexpr int kMaxRadices = 24;

// Division by a runtime divisor d >= 1 for numerators n < 2^31 with one high multiply:
// q = (umulhi(n, m) + n) >> s, s = ceil(log2 d), m = floor(2^32 (2^s - d) / d) + 1
// (the round-up method of Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994).
struct FastDiv {
  uint32_t d, m, s;
  __host__ __device__ FastDiv() : d(1), m(1), s(0) {}
  __host__ __device__ explicit FastDiv(uint32_t dd) : d(dd ? dd : 1) {
    uint32_t sh = 0;
    while ((1ull << sh) < d) ++sh;
    s = sh;
    m = (uint32_t)((((uint64_t)1 << 32) * (((uint64_t)1 << sh) - d)) / d + 1);
  }
  __device__ __forceinline__ int div(int n) const {
    return (int)((__umulhi((uint32_t)n, m) + (uint32_t)n) >> s);
  }
};

// Compile-time factorisation of a transform length. big = false: radices 5 then 3 (the
// runtime plan's order); big = true: composite radices done in registers (15, 25, 9,
// then 5 and 3), fewer shared-memory stages for the same length.
__host__ __device__ constexpr int cf_radix(int M, int stage, bool big = false) {
  int m = M, idx = 0;
  const int rs_small[5] = {5, 3, 7, 11, 13};
  const int rs_big[5] = {15, 25, 9, 5, 3};
  for (int i = 0; i < 5; ++i) {
    const int r = big ? rs_big[i] : rs_small[i];
    while (m > 1 && m % r == 0) {
      if (idx == stage) return r;
      m /= r;
      ++idx;
    }
  }
  return 0;
}
__host__ __device__ constexpr int cf_nstages(int M, bool big = false) {
  int n = 0;
  while (cf_radix(M, n, big) != 0) ++n;
  return n;
}
__host__ __device__ constexpr int cf_ns(int M, int stage, bool big = false) {
  int p = 1;
  for (int i = 0; i < stage; ++i) p *= cf_radix(M, i, big);
  return p;
}

// FastDiv's multiplier and shift alone (an aggregate: all zero until set).
struct DivConst {
  uint32_t m, s;
};
__host__ __device__ inline DivConst div_const(uint32_t d) {
  const FastDiv f(d);
  return DivConst{f.m, f.s};
}
__device__ __forceinline__ int div_by(DivConst c, int n) { return (int)((__umulhi((uint32_t)n, c.m) + (uint32_t)n) >> c.s); }

// Factorised plan of one transform length M (Stockham autosort, mixed radix). Inverse
// transforms run the radices in order, forward ones in reverse order, so that the stage with
// the most to skip (the largest radix) is the first of a zero-padded inverse transform and the
// last of a truncating forward one.
constexpr int kPlanDivs = 8;
struct FftPlan {
  int M;
  int nrad;
  int radix[kMaxRadices];
  int sched;   // compile-time lengths in the batched kernel: 0 precision default,
               // 1 radices 5 and 3, 2 composite register radices 15, 25, 9
  int ndiv;    // > 0: the divisions of a stage prepared (plan_divisions), else formed in the kernel
  DivConst nb[kPlanDivs];   // by M / radix[s]
  DivConst nsi[kPlanDivs];  // by the product of the radices before s (inverse order)
  DivConst nsf[kPlanDivs];  // by the product of the radices after s (forward order)
};
__host__ __device__ inline void plan_divisions(FftPlan& p) {
  p.ndiv = 0;
  if (p.nrad > kPlanDivs) return;
  int ns = 1;
  for (int s = 0; s < p.nrad; ++s) {
    p.nb[s] = div_const((uint32_t)(p.M / p.radix[s]));
    p.nsi[s] = div_const((uint32_t)ns);
    ns *= p.radix[s];
  }
  ns = 1;
  for (int s = p.nrad - 1; s >= 0; --s) {
    p.nsf[s] = div_const((uint32_t)ns);
    ns *= p.radix[s];
  }
  p.ndiv = p.nrad;
}

// Radices of a transform of length M: primes above 13 first (their first inverse stage skips
// the zero padding's terms and needs no twiddles), then with `big` the composite register
// radices 15 and 9 (fewer passes through shared memory), then 13, 11, 7, 5, 3 and, for image
// lengths and even grids (the double grid is odd), 8, 4, 2. The batched kernel and float-float
// passes take radices 5, 3, 7, 11, 13 in this order (big = false, see fft_pencils_small and cfft),
// then 8, 4, 2 as well: float-float transforms of an even grid's own length (GaNi) have them, the
// batch has odd grids alone. Without a factor 2 left, every further radix is an odd prime.
inline void make_plan(int M, FftPlan& p, bool big = true) {
  p.M = M;
  p.nrad = 0;
  p.sched = 0;
  int rest[kMaxRadices], nrest = 0;
  auto pull = [&](int& m, int r) {
    while (m % r == 0 && nrest < kMaxRadices) { rest[nrest++] = r; m /= r; }
  };
  int m = M;
  if (big)
    for (int r : {15, 13, 11, 9, 7, 5, 3, 8, 4, 2}) pull(m, r);
  else
    for (int r : {5, 3, 7, 11, 13, 8, 4, 2}) pull(m, r);
  for (int r = 17; m > 1; r += 2) {
    if ((long long)r * r > m) r = m;   // what is left is prime
    while (m % r == 0 && p.nrad < kMaxRadices) { p.radix[p.nrad++] = r; m /= r; }
  }
  for (int i = 0; i < nrest && p.nrad < kMaxRadices; ++i) p.radix[p.nrad++] = rest[i];
  plan_divisions(p);
}

// ---------------------------------------------------------------------------------
// Small DFT butterflies. dir = -1: forward (w = exp(-2 pi i / r)); dir = +1: inverse.
// The constants are cos/sin of 2 pi/3, 2 pi/5, 4 pi/5.
// ---------------------------------------------------------------------------------
// The sine term of radix 3: v1, v2 = t +- i s sin(2 pi/3) d for the sign s of dir. In the packed FP32 types an
// FMA for each part: a packed product would be rounded by itself (the scalar one is contracted into
// the sums) and takes two operations more in fpair. Against 64 bits: FP32 operator at N = 203 in 2D 1.66e-7
// -> 1.61e-7 (1.60e-7 in scalars), N = 113 in 3D 1.64e-7 -> 1.62e-7 (1.62e-7), the same time.
// F = false: the packed product, in the runtime plans, whose other radices round less than before as it
// is (ragged 41 x 33 x 53 cell 1.57e-7 in scalars, 1.51e-7 so) and which the FMAs make slower
// at some lengths (N = 255 in 2D 95 -> 97 us, N = 17 21.0 -> 22.5).
template <typename T> struct sine_fma { static constexpr bool value = is_fpair<T>::value; };
#if defined(__CUDA_ARCH__) && !defined(HOMB_SCALAR_COMPLEX)
template <> struct sine_fma<float> { static constexpr bool value = true; };
#endif
template <typename T, bool F = sine_fma<T>::value>
__device__ __forceinline__ void dft3_sine(cpx<T> t, cpx<T> d, int dir, cpx<T>* v1, cpx<T>* v2) {
  const T s3 = T(0.86602540378443864676372317075294);
  if constexpr (F) {
    const T p = dir > 0 ? s3 : -s3, n = dir > 0 ? -s3 : s3;
    *v1 = mk<T>(fma(n, d.y, t.x), fma(p, d.x, t.y));
    *v2 = mk<T>(fma(p, d.y, t.x), fma(n, d.x, t.y));
  } else {
    const cpx<T> it3 = rot<T>(scl<T>(d, s3), dir > 0 ? 1 : -1);
    *v1 = add<T>(t, it3);
    *v2 = sub<T>(t, it3);
  }
}
template <typename T, bool F = sine_fma<T>::value> __device__ __forceinline__ void dft3(cpx<T>* v, int dir) {
  const T h = T(0.5);
  const cpx<T> t1 = add<T>(v[1], v[2]), d = sub<T>(v[1], v[2]);
  const cpx<T> t2 = axpy<T>(-h, t1, v[0]);
  v[0] = add<T>(v[0], t1);
  dft3_sine<T, F>(t2, d, dir, &v[1], &v[2]);   // forward: V1 = t2 - i s3 d, V2 = t2 + i s3 d
}

template <typename T> __device__ __forceinline__ void dft5(cpx<T>* v, int dir) {
  const T c1 = T(0.30901699437494742410229341718282);    // cos(2 pi/5)
  const T c2 = T(-0.80901699437494742410229341718282);   // cos(4 pi/5)
  const T s1 = T(0.95105651629515357211643933337938);    // sin(2 pi/5)
  const T s2 = T(0.58778525229247312916870595463907);    // sin(4 pi/5)
  cpx<T> a1 = add<T>(v[1], v[4]), b1 = sub<T>(v[1], v[4]);
  cpx<T> a2 = add<T>(v[2], v[3]), b2 = sub<T>(v[2], v[3]);
  cpx<T> m1 = axpy<T>(c1, a1, axpy<T>(c2, a2, v[0]));
  cpx<T> m2 = axpy<T>(c2, a1, axpy<T>(c1, a2, v[0]));
  cpx<T> n1 = axpy<T>(s1, b1, scl<T>(b2, s2));
  cpx<T> n2 = axpy<T>(s2, b1, scl<T>(b2, -s1));
  v[0] = add<T>(v[0], add<T>(a1, a2));
  int s = dir > 0 ? 1 : -1;     // forward: V1 = m1 - i n1
  cpx<T> in1 = rot<T>(n1, s), in2 = rot<T>(n2, s);
  v[1] = add<T>(m1, in1);
  v[4] = sub<T>(m1, in1);
  v[2] = add<T>(m2, in2);
  v[3] = sub<T>(m2, in2);
}

// Compile-time cos / sin from their Taylor series (arguments up to pi / 4); used only for the
// twiddle constants inside the register DFTs.
__host__ __device__ constexpr double ct_sin_red(double x) {
  double term = x, sum = x;
  for (int n = 1; n < 30; ++n) {
    term *= -x * x / ((2.0 * n) * (2.0 * n + 1.0));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr double ct_cos_red(double x) {
  double term = 1.0, sum = 1.0;
  for (int n = 1; n < 30; ++n) {
    term *= -x * x / ((2.0 * n - 1.0) * (2.0 * n));
    sum += term;
  }
  return sum;
}
// cos and sin of 2 pi p / q, reduced in integers to an angle 2 pi n / m of the first octant: there the
// series has no cancellation (from the whole half circle it left 1e-15, seen in FP64 transforms
// of lengths with radices 7 to 13)
struct CtSinCos {
  double c, s;
};
__host__ __device__ constexpr CtSinCos ct_octant(int n, int m) {   // 0 <= 8 n <= m
  const double x = 6.283185307179586476925286766559 * (double)n / (double)m;
  return CtSinCos{ct_cos_red(x), ct_sin_red(x)};
}
__host__ __device__ constexpr CtSinCos ct_quadrant(int n, int m) {   // 0 <= 4 n <= m
  if (8 * n <= m) return ct_octant(n, m);
  const CtSinCos r = ct_octant(m - 4 * n, 4 * m);   // pi / 2 less the angle
  return CtSinCos{r.s, r.c};
}
__host__ __device__ constexpr CtSinCos ct_sincos(int p, int q) {
  int r = p % q;
  if (r < 0) r += q;
  const bool lower = 2 * r > q;   // sin < 0
  if (lower) r = q - r;
  CtSinCos v{1.0, 0.0};
  if (4 * r <= q) {
    v = ct_quadrant(r, q);
  } else {
    v = ct_quadrant(q - 2 * r, 2 * q);   // pi less the angle
    v.c = -v.c;
  }
  if (lower) v.s = -v.s;
  return v;
}
__host__ __device__ constexpr double ct_cos2pi(int p, int q) { return ct_sincos(p, q).c; }
__host__ __device__ constexpr double ct_sin2pi(int p, int q) { return ct_sincos(p, q).s; }

__host__ __device__ constexpr int ct_first_factor(int R) {
  return R % 3 == 0 ? 3 : (R % 5 == 0 ? 5 : R);
}

// Register DFT of compile-time length R (a product of 3s and 5s): Cooley-Tukey with
// R = R1 * R2, inner DFTs over n1 for each n2, constant twiddles w_R^{n2 k1}, outer
// DFTs over n2; output index k1 + R1 k2. dir = -1 forward, +1 inverse.
template <typename T, int R>
__device__ __forceinline__ void dft_reg(cpx<T>* v, int dir);

template <typename T, int R1, int R2>
__device__ __forceinline__ void dft_ct(cpx<T>* v, int dir) {
  constexpr int R = R1 * R2;
  cpx<T> t[R];
#pragma unroll
  for (int n2 = 0; n2 < R2; ++n2) {
    cpx<T> a[R1];
#pragma unroll
    for (int n1 = 0; n1 < R1; ++n1) a[n1] = v[R2 * n1 + n2];
    dft_reg<T, R1>(a, dir);
#pragma unroll
    for (int k1 = 0; k1 < R1; ++k1) {
      if (n2 * k1 == 0) {
        t[n2 * R1 + k1] = a[k1];
      } else {
        const T c = T(ct_cos2pi(n2 * k1, R)), sn = T(ct_sin2pi(n2 * k1, R));
        const T s = dir > 0 ? sn : -sn;    // w = exp(dir * 2 pi i n2 k1 / R)
        t[n2 * R1 + k1] = mk<T>(fma(a[k1].x, c, -a[k1].y * s), fma(a[k1].x, s, a[k1].y * c));
      }
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < R1; ++k1) {
    cpx<T> b[R2];
#pragma unroll
    for (int n2 = 0; n2 < R2; ++n2) b[n2] = t[n2 * R1 + k1];
    dft_reg<T, R2>(b, dir);
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k1 + R1 * k2] = b[k2];
  }
}

// Length 15 by the prime-factor (Good-Thomas) map, 15 = 3 * 5 with coprime factors:
// input n = (5 n1 + 3 n2) mod 15, output k = (10 k1 + 6 k2) mod 15, so that
// w_15^(n k) = w_3^(n1 k1) w_5^(n2 k2) and no twiddle multiplications are needed.
template <typename T, bool F = sine_fma<T>::value>
__device__ __forceinline__ void dft15_pfa(cpx<T>* v, int dir) {
  cpx<T> t[15];
#pragma unroll
  for (int n2 = 0; n2 < 5; ++n2) {
    cpx<T> a[3];
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) a[n1] = v[(5 * n1 + 3 * n2) % 15];
    dft3<T, F>(a, dir);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) t[n2 * 3 + k1] = a[k1];
  }
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cpx<T> b[5];
#pragma unroll
    for (int n2 = 0; n2 < 5; ++n2) b[n2] = t[n2 * 3 + k1];
    dft5<T>(b, dir);
#pragma unroll
    for (int k2 = 0; k2 < 5; ++k2) v[(10 * k1 + 6 * k2) % 15] = b[k2];
  }
}

template <typename T, int R>
__device__ __forceinline__ void dft_reg(cpx<T>* v, int dir) {
  if constexpr (R == 3) {
    dft3<T>(v, dir);
  } else if constexpr (R == 5) {
    dft5<T>(v, dir);
  } else if constexpr (R == 15) {
    dft15_pfa<T>(v, dir);
  } else {
    constexpr int R1 = ct_first_factor(R);
    dft_ct<T, R1, R / R1>(v, dir);
  }
}

// Known zeros of the warp FFTs' transforms of length M = R*R. A zero-padded inverse transform has
// at most N <= (M+1)/2 nonzero inputs: at positions p <= (M-3)/4 and p >= (3M+3)/4 (the y rows
// of the padded slab, the Hermitian x extension, Nh <= (M+3)/4); a truncating forward one
// keeps only the outputs at those positions. In the lane layout p = l + R n of the register
// FFTs, the rows n in [lo, hi] hold only such positions for every lane l: they are never read
// as inputs (inverse) and never computed or stored as outputs (forward).
template <int R> struct ZeroBand {
  static constexpr int M = R * R;
  static constexpr int lo = ((M + 3) / 4 + R - 1) / R;
  static constexpr int hi = ((3 * M - 3) / 4 - (R - 1)) / R;
  static constexpr bool in(int n) { return n >= lo && n <= hi; }
};
static_assert(ZeroBand<15>::lo == 4 && ZeroBand<15>::hi == 10, "zero band of the length-225 transforms");

// DFT3 of (a0, a1, a2) with compile-time zero inputs (Z0, Z1, Z2), same convention as dft3:
// y_k = sum_n a_n w^(n k), w = exp(dir 2 pi i / 3). Inputs marked zero are not read.
template <typename T, bool Z0, bool Z1, bool Z2>
__device__ __forceinline__ void dft3_z(const cpx<T>* a, cpx<T>* y, int dir) {
  const T h = T(0.5);
  const T s3 = (dir > 0 ? T(1) : T(-1)) * T(0.86602540378443864676372317075294);
  if constexpr (!Z0 && Z1 && Z2) {
    y[0] = a[0];
    y[1] = a[0];
    y[2] = a[0];
  } else if constexpr (Z0 && !Z1 && Z2) {   // y1 = w a1, y2 = w^2 a1
    const cpx<T> b = a[1];
    const T mx = -h * b.x, my = -h * b.y;
    y[0] = b;
    y[1] = mk<T>(fma(-s3, b.y, mx), fma(s3, b.x, my));
    y[2] = mk<T>(fma(s3, b.y, mx), fma(-s3, b.x, my));
  } else if constexpr (!Z0 && !Z1 && Z2) {   // y1 = a0 + w a1, y2 = a0 + w^2 a1
    const cpx<T> m = axpy<T>(-h, a[1], a[0]);
    y[0] = add<T>(a[0], a[1]);
    y[1] = mk<T>(fma(-s3, a[1].y, m.x), fma(s3, a[1].x, m.y));
    y[2] = mk<T>(fma(s3, a[1].y, m.x), fma(-s3, a[1].x, m.y));
  } else if constexpr (!Z0 && Z1 && !Z2) {   // y1 = a0 + w^2 a2, y2 = a0 + w a2
    const cpx<T> m = axpy<T>(-h, a[2], a[0]);
    y[0] = add<T>(a[0], a[2]);
    y[1] = mk<T>(fma(s3, a[2].y, m.x), fma(-s3, a[2].x, m.y));
    y[2] = mk<T>(fma(-s3, a[2].y, m.x), fma(s3, a[2].x, m.y));
  } else if constexpr (Z0 && !Z1 && !Z2) {   // y1 = w a1 + w^2 a2, y2 = w^2 a1 + w a2
    const cpx<T> t = add<T>(a[1], a[2]), dd = sub<T>(a[1], a[2]);
    const T mx = -h * t.x, my = -h * t.y;
    y[0] = t;
    y[1] = mk<T>(fma(-s3, dd.y, mx), fma(s3, dd.x, my));
    y[2] = mk<T>(fma(s3, dd.y, mx), fma(-s3, dd.x, my));
  } else {
    y[0] = a[0];
    y[1] = a[1];
    y[2] = a[2];
    dft3<T>(y, dir);
  }
}

// DFT5 of b computing only the outputs in the compile-time mask KEEP (bit k: output k); the
// others are left unchanged. Same convention as dft5.
template <typename T, int KEEP>
__device__ __forceinline__ void dft5_keep(cpx<T>* v, int dir) {
  const T c1 = T(0.30901699437494742410229341718282);    // cos(2 pi/5)
  const T c2 = T(-0.80901699437494742410229341718282);   // cos(4 pi/5)
  const T s1 = T(0.95105651629515357211643933337938);    // sin(2 pi/5)
  const T s2 = T(0.58778525229247312916870595463907);    // sin(4 pi/5)
  const cpx<T> a1 = add<T>(v[1], v[4]), b1 = sub<T>(v[1], v[4]);
  const cpx<T> a2 = add<T>(v[2], v[3]), b2 = sub<T>(v[2], v[3]);
  const int s = dir > 0 ? 1 : -1;
  cpx<T> o[5];
  if constexpr ((KEEP & 0x12) != 0) {   // outputs 1, 4
    const cpx<T> m1 = axpy<T>(c1, a1, axpy<T>(c2, a2, v[0]));
    const cpx<T> n1 = axpy<T>(s1, b1, scl<T>(b2, s2));
    const cpx<T> in1 = rot<T>(n1, s);
    o[1] = add<T>(m1, in1);
    o[4] = sub<T>(m1, in1);
  }
  if constexpr ((KEEP & 0x0c) != 0) {   // outputs 2, 3
    const cpx<T> m2 = axpy<T>(c2, a1, axpy<T>(c1, a2, v[0]));
    const cpx<T> n2 = axpy<T>(s2, b1, scl<T>(b2, -s1));
    const cpx<T> in2 = rot<T>(n2, s);
    o[2] = add<T>(m2, in2);
    o[3] = sub<T>(m2, in2);
  }
  if constexpr ((KEEP & 1) != 0) v[0] = add<T>(v[0], add<T>(a1, a2));
#pragma unroll
  for (int k = 1; k < 5; ++k)
    if ((KEEP >> k) & 1) v[k] = o[k];
}

// Length-15 DFT (prime-factor map as dft15_pfa) with the inputs of the zero band (4..10) known
// to be zero: they are not read, and the first-layer DFT3s take their reduced forms.
template <typename T>
__device__ __forceinline__ void dft15_zin(cpx<T>* v, int dir) {
  cpx<T> t[15];
  {
    const cpx<T> a[3] = {v[0], v[0], v[0]};   // n2 = 0: inputs 0, 5, 10
    dft3_z<T, false, true, true>(a, t + 0, dir);
  }
  {
    const cpx<T> a[3] = {v[3], v[3], v[13]};   // n2 = 1: inputs 3, 8, 13
    dft3_z<T, false, true, false>(a, t + 3, dir);
  }
  {
    const cpx<T> a[3] = {v[1], v[11], v[1]};   // n2 = 2: inputs 6, 11, 1
    dft3_z<T, true, false, false>(a, t + 6, dir);
  }
  {
    const cpx<T> a[3] = {v[14], v[14], v[14]};   // n2 = 3: inputs 9, 14, 4
    dft3_z<T, true, false, true>(a, t + 9, dir);
  }
  {
    const cpx<T> a[3] = {v[12], v[2], v[2]};   // n2 = 4: inputs 12, 2, 7
    dft3_z<T, false, false, true>(a, t + 12, dir);
  }
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cpx<T> b[5];
#pragma unroll
    for (int n2 = 0; n2 < 5; ++n2) b[n2] = t[n2 * 3 + k1];
    dft5<T>(b, dir);
#pragma unroll
    for (int k2 = 0; k2 < 5; ++k2) v[(10 * k1 + 6 * k2) % 15] = b[k2];
  }
}

// Length-15 DFT (prime-factor map) computing only the outputs outside the zero band (0..3,
// 11..14); the band's outputs are left undefined.
template <typename T, bool F = sine_fma<T>::value>
__device__ __forceinline__ void dft15_zout(cpx<T>* v, int dir) {
  cpx<T> t[15];
#pragma unroll
  for (int n2 = 0; n2 < 5; ++n2) {
    cpx<T> a[3];
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) a[n1] = v[(5 * n1 + 3 * n2) % 15];
    dft3<T, F>(a, dir);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) t[n2 * 3 + k1] = a[k1];
  }
  // outputs k = (10 k1 + 6 k2) mod 15 outside 4..10: k1 = 0: k2 in {0, 2, 3} (0, 12, 3);
  // k1 = 1: k2 in {1, 3} (1, 13); k1 = 2: k2 in {1, 2, 4} (11, 2, 14)
  cpx<T> b[5];
#pragma unroll
  for (int n2 = 0; n2 < 5; ++n2) b[n2] = t[n2 * 3 + 0];
  dft5_keep<T, 0x0d>(b, dir);
  v[0] = b[0];
  v[12] = b[2];
  v[3] = b[3];
#pragma unroll
  for (int n2 = 0; n2 < 5; ++n2) b[n2] = t[n2 * 3 + 1];
  dft5_keep<T, 0x0a>(b, dir);
  v[1] = b[1];
  v[13] = b[3];
#pragma unroll
  for (int n2 = 0; n2 < 5; ++n2) b[n2] = t[n2 * 3 + 2];
  dft5_keep<T, 0x16>(b, dir);
  v[11] = b[1];
  v[2] = b[2];
  v[14] = b[4];
}

// Inputs a zero-padded inverse transform of N <= (M + 1) / 2 frequencies knows to be zero in
// a first stage of odd radix R, and outputs a truncating forward one drops in a last stage:
// q = LO .. R - 1 - LO (positions q M / R + j around the middle of the pencil).
template <int R> struct RadixBand {
  static constexpr int lo = R / 4 + 1, hi = R - 1 - lo;
  static constexpr bool in(int q) { return q >= lo && q <= hi; }
};
// whether those positions hold nothing when the frequencies 0 .. half and -top .. -1 are stored
__device__ __forceinline__ bool radix_band_free(int R, int nb, int M, int half, int top) {
  const int lo = R / 4 + 1;
  return lo * nb > half && (R - lo) * nb <= M - top;
}

// Odd radix R in registers from the sums a_q = v_q + v_{R-q} and differences b_q = v_q - v_{R-q}
// (DFT of a_q with cosines, of b_q with sines: a quarter of the products of the direct sum):
// V_s, V_{R-s} = v_0 + sum_q a_q cos(2 pi q s / R) +- i DIR sum_q b_q sin(2 pi q s / R).
// ZI: the inputs of RadixBand are zero (not read); ZO: its outputs are not needed (undefined).
template <typename T, int R, int DIR, bool ZI = false, bool ZO = false>
__device__ __forceinline__ void dft_odd(cpx<T>* v) {
  constexpr int H = (R - 1) / 2, LO = RadixBand<R>::lo;
  constexpr int QN = ZI ? (LO < H ? LO : H) : H;   // pairs with a nonzero input
  constexpr int SN = ZO ? (LO < H ? LO : H) : H;   // pairs with a needed output
  cpx<T> a[QN], b[QN];
#pragma unroll
  for (int q = 1; q <= QN; ++q) {
    if (ZI && RadixBand<R>::in(q)) {   // only v_{R-q}
      a[q - 1] = v[R - q];
      b[q - 1] = mk<T>(-v[R - q].x, -v[R - q].y);
    } else {
      a[q - 1] = add<T>(v[q], v[R - q]);
      b[q - 1] = sub<T>(v[q], v[R - q]);
    }
  }
  const cpx<T> v0 = v[0];
  cpx<T> t0 = v0;
#pragma unroll
  for (int q = 0; q < QN; ++q) t0 = add<T>(t0, a[q]);
  v[0] = t0;
#pragma unroll
  for (int s = 1; s <= SN; ++s) {
    cpx<T> m = v0, n;
#pragma unroll
    for (int q = 1; q <= QN; ++q) {
      const T c = T(ct_cos2pi(q * s, R)), sn = T(DIR * ct_sin2pi(q * s, R));
      m = axpy<T>(c, a[q - 1], m);
      if (q == 1) n = scl<T>(b[0], sn);
      else n = axpy<T>(sn, b[q - 1], n);
    }
    if (!(ZO && RadixBand<R>::in(s))) v[s] = mk<T>(m.x - n.y, m.y + n.x);
    v[R - s] = mk<T>(m.x + n.y, m.y - n.x);
  }
}

// Radix 9 = 3 x 3 with its middle inputs 3..5 zero (ZI) or its middle outputs 3..5 not needed (ZO)
template <typename T, bool F = sine_fma<T>::value> __device__ __forceinline__ void dft3_mid_in0(cpx<T>* v, int dir);
template <typename T, bool F = sine_fma<T>::value> __device__ __forceinline__ void dft3_skip_out1(cpx<T>* v, int dir);
template <typename T, int DIR, bool ZI, bool ZO>
__device__ __forceinline__ void dft9_band(cpx<T>* v) {
  cpx<T> t[9];
#pragma unroll
  for (int n2 = 0; n2 < 3; ++n2) {
    cpx<T> a[3] = {v[n2], v[3 + n2], v[6 + n2]};
    if (ZI) dft3_mid_in0<T, false>(a, DIR);
    else dft3<T, false>(a, DIR);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      if (n2 * k1 == 0) {
        t[n2 * 3 + k1] = a[k1];
      } else {
        const T c = T(ct_cos2pi(n2 * k1, 9)), s = T(DIR * ct_sin2pi(n2 * k1, 9));
        t[n2 * 3 + k1] = mk<T>(fma(a[k1].x, c, -a[k1].y * s), fma(a[k1].x, s, a[k1].y * c));
      }
    }
  }
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cpx<T> b[3] = {t[k1], t[3 + k1], t[6 + k1]};
    if (ZO) dft3_skip_out1<T, false>(b, DIR);
    else dft3<T, false>(b, DIR);
    v[k1] = b[0];
    if (!ZO) v[3 + k1] = b[1];
    v[6 + k1] = b[2];
  }
}

// Power-of-two radices 2, 4, 8 (image lengths and even grids; the double grid is odd)
template <typename T, int R, int DIR>
__device__ __forceinline__ void dft_pow2(cpx<T>* v) {
  if constexpr (R == 2) {
    const cpx<T> a = v[0];
    v[0] = add<T>(a, v[1]);
    v[1] = sub<T>(a, v[1]);
  } else {
    constexpr int Hh = R / 2;
    cpx<T> e[Hh], o[Hh];
#pragma unroll
    for (int k = 0; k < Hh; ++k) {
      e[k] = v[2 * k];
      o[k] = v[2 * k + 1];
    }
    dft_pow2<T, Hh, DIR>(e);
    dft_pow2<T, Hh, DIR>(o);
#pragma unroll
    for (int k = 0; k < Hh; ++k) {
      cpx<T> w = o[k];
      if (4 * k == R) {
        w = rot<T>(w, DIR);
      } else if (k > 0) {
        const T c = T(ct_cos2pi(k, R)), s = T(DIR * ct_sin2pi(k, R));
        w = mk<T>(fma(o[k].x, c, -o[k].y * s), fma(o[k].x, s, o[k].y * c));
      }
      v[k] = add<T>(e[k], w);
      v[k + Hh] = sub<T>(e[k], w);
    }
  }
}

template <typename T, int R, int DIR, bool ZI, bool ZO>
__device__ __forceinline__ void dft_radix(cpx<T>* v) {
  if constexpr (R % 2 == 0) dft_pow2<T, R, DIR>(v);
  else if constexpr (R == 3 && ZI) dft3_mid_in0<T, false>(v, DIR);
  else if constexpr (R == 3 && ZO) dft3_skip_out1<T, false>(v, DIR);
  else if constexpr (R == 3) dft3<T, false>(v, DIR);
  else if constexpr (R == 9) dft9_band<T, DIR, ZI, ZO>(v);
  else if constexpr (R == 15 && ZI) dft15_zin<T>(v, DIR);
  else if constexpr (R == 15 && ZO) dft15_zout<T, false>(v, DIR);
  else if constexpr (R == 15) dft15_pfa<T, false>(v, DIR);
  else if constexpr (R == 5 && !ZI && !ZO) dft5<T>(v, DIR);
  else dft_odd<T, R, DIR, ZI, ZO>(v);
}

// One Stockham stage of radix R over G pencils (strides ld) of runtime length M.
template <typename T, int R, int DIR, bool ZI, bool ZO>
__device__ __forceinline__ void stage_radix(const cpx<T>* __restrict__ a, cpx<T>* __restrict__ b, int G, int ld, int M,
                                            int Ns, DivConst dnb, DivConst dns, const cpx<T>* W) {
  const int nb = M / R;
  const int step = nb / Ns;   // M / (Ns R)
  for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
    const int g = div_by(dnb, t);
    const int j = t - g * nb;
    const cpx<T>* src = a + (size_t)g * ld + j;
    cpx<T> v[R];
#pragma unroll
    for (int q = 0; q < R; ++q)
      if (!(ZI && RadixBand<R>::in(q))) v[q] = src[q * nb];
    int base = j * R;
    if (Ns > 1) {
      const int c = div_by(dns, j);
      const int k = j - c * Ns;
      base = c * Ns * R + k;
      const int kw = k * step;
#pragma unroll
      for (int q = 1; q < R; ++q) v[q] = mulc<T>(v[q], W[q * kw], DIR > 0);
    }
    dft_radix<T, R, DIR, ZI, ZO>(v);
    cpx<T>* dst = b + (size_t)g * ld + base;
#pragma unroll
    for (int q = 0; q < R; ++q)
      if (!(ZO && RadixBand<R>::in(q))) dst[q * Ns] = st_norm<T>(v[q]);
  }
}

// A stage of any larger prime radix R (twice: the callers synchronise in between). First the
// twiddled inputs' sums x_q + x_{R-q} and differences x_q - x_{R-q}, in place at q and R - q;
// then each thread forms kPrimeTile output pairs (s, R - s) of one butterfly from them:
// R / 2 terms of two real products a complex output instead of R terms of eight, one load of a
// sum and a difference for kPrimeTile pairs. qn, sn: pairs with a nonzero input / a needed output.
constexpr int kPrimeTile = 4;
template <typename T, int DIR>
__device__ __forceinline__ void stage_prime_sums(cpx<T>* a, int G, int ld, int M, int R, int Ns, int qn,
                                                 DivConst dnb, DivConst dns, const cpx<T>* W) {
  const int nb = M / R;
  const int step = nb / Ns;
  for (int t = threadIdx.x; t < G * nb * qn; t += blockDim.x) {
    const int gj = t / qn;
    const int q = t - gj * qn + 1;
    const int g = div_by(dnb, gj);
    const int j = gj - g * nb;
    cpx<T>* p = a + (size_t)g * ld + j;
    cpx<T> x = p[q * nb], y = p[(R - q) * nb];
    if (Ns > 1) {
      const int k = j - div_by(dns, j) * Ns;
      x = mulc<T>(x, W[q * k * step], DIR > 0);
      y = mulc<T>(y, W[(R - q) * k * step], DIR > 0);
    }
    p[q * nb] = st_norm<T>(add<T>(x, y));
    p[(R - q) * nb] = st_norm<T>(sub<T>(x, y));
  }
}
template <typename T, int DIR>
__device__ __forceinline__ void stage_prime_out(const cpx<T>* __restrict__ a, cpx<T>* __restrict__ b, int G, int ld,
                                                int M, int R, int Ns, int qn, int sn, DivConst dnb, DivConst dns,
                                                const cpx<T>* W) {
  const int nb = M / R;
  const int ntile = (sn + kPrimeTile) / kPrimeTile;   // s = 0 .. sn
  const int nbf = G * nb;
  for (int t = threadIdx.x; t < nbf * ntile; t += blockDim.x) {
    const int tile = t / nbf;
    const int gj = t - tile * nbf;
    const int g = div_by(dnb, gj);
    const int j = gj - g * nb;
    const cpx<T>* p = a + (size_t)g * ld + j;
    const int s0 = tile * kPrimeTile;
    const cpx<T> x0 = p[0];
    cpx<T> m[kPrimeTile], n[kPrimeTile];
    int ws[kPrimeTile];
#pragma unroll
    for (int u = 0; u < kPrimeTile; ++u) {
      m[u] = x0;
      n[u] = mk<T>(T(0), T(0));
      ws[u] = 0;
    }
    for (int q = 1; q <= qn; ++q) {
      const cpx<T> sa = p[q * nb], sb = p[(R - q) * nb];
#pragma unroll
      for (int u = 0; u < kPrimeTile; ++u) {
        ws[u] += s0 + u;
        if (ws[u] >= R) ws[u] -= R;
        const cpx<T> w = W[ws[u] * nb];   // cos, -sin of 2 pi q s / R
        m[u] = axpy<T>(w.x, sa, m[u]);
        n[u] = axpy<T>(w.y, sb, n[u]);
      }
    }
    const int c = div_by(dns, j);
    const int k = j - c * Ns;
    cpx<T>* d = b + (size_t)g * ld + c * Ns * R + k;
#pragma unroll
    for (int u = 0; u < kPrimeTile; ++u) {
      const int s = s0 + u;
      if (s > sn || 2 * s >= R) continue;
      // n holds - sum b sin: V_s = m + i DIR sum b sin
      const cpx<T> in = DIR > 0 ? mk<T>(n[u].y, -n[u].x) : mk<T>(-n[u].y, n[u].x);
      d[s * Ns] = st_norm<T>(add<T>(m[u], in));
      if (s > 0) d[(R - s) * Ns] = st_norm<T>(sub<T>(m[u], in));
    }
  }
}

// The frequencies around 0 that a pencil holds (0 .. half and -top .. -1) and which side of the
// transform they bound: prune bit 1, zero-padded inputs (the first stage skips its known
// zeros); bit 2, truncated outputs (the last stage skips what is dropped).
struct FftBand {
  int half, top, prune;
};

// the pairs (q, R - q), q <= h, of rows of `stride` positions with one inside the band
__device__ __forceinline__ int pairs_in_band(int h, int stride, FftBand band) {
  const int up = band.half / stride, dn = (band.top + stride - 1) / stride;
  const int n = up > dn ? up : dn;
  return n < h ? n : h;
}

// G pencils of length M at a + g*ld (ping-pong with b, same strides) by the runtime plan, in
// direction DIR. The CTA runs all stages; returns the buffer holding the result. Ends with
// __syncthreads().
// Bound by instruction issue (FP32, float-float) or the FP64 pipe: so the index divisions by
// runtime lengths are multiplications prepared in the plan, radices 15 and 9 halve the passes
// through shared memory, radices 5 to 13 and primes use the real symmetry, and zero padding and
// dropped outputs are skipped. Against radices 3, 5, 7 with divisions and direct sums: FP32
// operator of a 41 x 33 x 53 cell (lengths 81, 65, 105) 298 -> 92 us, mixed bounds of 16 balls at
// N = 51 (length 105) 176 -> 72 ms, FP64 3D operators at lengths with primes 4 to 7 times.
template <typename T, int DIR>
__device__ __forceinline__ cpx<T>* fft_plan_run(cpx<T>* a, cpx<T>* b, int G, int ld, const FftPlan& plan,
                                                const cpx<T>* W, FftBand band) {
  const int M = plan.M;
  int Ns = 1;
  cpx<T>* src = a;
  cpx<T>* dst = b;
  for (int i = 0; i < plan.nrad; ++i) {
    const int s = DIR > 0 ? i : plan.nrad - 1 - i;
    const int R = plan.radix[s];
    const int nb = M / R;
    DivConst dnb, dns;
    if (plan.ndiv > 0) {
      dnb = plan.nb[s];
      dns = DIR > 0 ? plan.nsi[s] : plan.nsf[s];
    } else {
      dnb = div_const((uint32_t)nb);
      dns = div_const((uint32_t)Ns);
    }
    const bool free_ = radix_band_free(R, nb, M, band.half, band.top);
    const bool zi = DIR > 0 && (band.prune & 1) && i == 0 && free_;
    const bool zo = DIR < 0 && (band.prune & 2) && i == plan.nrad - 1 && free_;
#define HOMB_STAGE(RR)                                                                                        \
  case RR:                                                                                                    \
    if (DIR > 0 && zi) stage_radix<T, RR, DIR, (DIR > 0), false>(src, dst, G, ld, M, Ns, dnb, dns, W);        \
    else if (DIR < 0 && zo) stage_radix<T, RR, DIR, false, (DIR < 0)>(src, dst, G, ld, M, Ns, dnb, dns, W);   \
    else stage_radix<T, RR, DIR, false, false>(src, dst, G, ld, M, Ns, dnb, dns, W);                          \
    break;
    switch (R) {
      case 2: stage_radix<T, 2, DIR, false, false>(src, dst, G, ld, M, Ns, dnb, dns, W); break;
      case 4: stage_radix<T, 4, DIR, false, false>(src, dst, G, ld, M, Ns, dnb, dns, W); break;
      case 8: stage_radix<T, 8, DIR, false, false>(src, dst, G, ld, M, Ns, dnb, dns, W); break;
      HOMB_STAGE(3)
      HOMB_STAGE(5)
      HOMB_STAGE(7)
      HOMB_STAGE(11)
      HOMB_STAGE(13)
      default:
        if constexpr (!is_ff<T>::value) {   // float-float plans hold no composite radix
          if (R == 9) {
            if (DIR > 0 && zi) stage_radix<T, 9, DIR, (DIR > 0), false>(src, dst, G, ld, M, Ns, dnb, dns, W);
            else if (DIR < 0 && zo) stage_radix<T, 9, DIR, false, (DIR < 0)>(src, dst, G, ld, M, Ns, dnb, dns, W);
            else stage_radix<T, 9, DIR, false, false>(src, dst, G, ld, M, Ns, dnb, dns, W);
            break;
          }
          if (R == 15) {
            if (DIR > 0 && zi) stage_radix<T, 15, DIR, (DIR > 0), false>(src, dst, G, ld, M, Ns, dnb, dns, W);
            else if (DIR < 0 && zo) stage_radix<T, 15, DIR, false, (DIR < 0)>(src, dst, G, ld, M, Ns, dnb, dns, W);
            else stage_radix<T, 15, DIR, false, false>(src, dst, G, ld, M, Ns, dnb, dns, W);
            break;
          }
        }
        {
          int qn = (R - 1) / 2, sn = (R - 1) / 2;
          if (DIR > 0 && (band.prune & 1) && i == 0)   // pairs with a position <= half or >= M - top
            qn = pairs_in_band(qn, nb, band);
          if (DIR < 0 && (band.prune & 2) && i == plan.nrad - 1)
            sn = pairs_in_band(sn, Ns, band);
          stage_prime_sums<T, DIR>(src, G, ld, M, R, Ns, qn, dnb, dns, W);
          __syncthreads();
          stage_prime_out<T, DIR>(src, dst, G, ld, M, R, Ns, qn, sn, dnb, dns, W);
        }
        break;
    }
#undef HOMB_STAGE
    __syncthreads();
    cpx<T>* t = src; src = dst; dst = t;
    Ns *= R;
  }
  return src;
}

template <typename T>
__device__ cpx<T>* fft_pencils(cpx<T>* a, cpx<T>* b, int G, int ld, const FftPlan& plan, const cpx<T>* W, int dir,
                               FftBand band = FftBand{0, 0, 0}) {
  return dir > 0 ? fft_plan_run<T, 1>(a, b, G, ld, plan, W, band) : fft_plan_run<T, -1>(a, b, G, ld, plan, W, band);
}

// The batched kernel's form of fft_pencils, for plans of radices 3 to 13 alone. A batch has no
// FP64 refinement, so its bounds at a loose tolerance carry the rounding of its FP32 CG: with
// the order of operations of fft_pencils they moved by 1.2e-9, and by 6e-7 where a cell
// stops at its FP32 floor (cells of one odd N, tolerance 1e-4). So this form keeps its
// arithmetic operation by operation (stages in the plan's order, radices 7 to 13 as direct
// sums, a direction known at run time only, which leaves no products to contract) and takes
// only the multiplications for its divisions.
template <typename T, int R>
__device__ __forceinline__ void dft_direct(cpx<T>* v, const cpx<T>* W, int M, int dir) {
  cpx<T> o[R];
  const int step = M / R;
#pragma unroll
  for (int s = 0; s < R; ++s) {
    cpx<T> acc = v[0];
#pragma unroll
    for (int q = 1; q < R; ++q) acc = add<T>(acc, mulc<T>(v[q], W[((q * s) % R) * step], dir > 0));
    o[s] = acc;
  }
#pragma unroll
  for (int s = 0; s < R; ++s) v[s] = o[s];
}
template <typename T, int R>
__device__ __forceinline__ void stage_small(const cpx<T>* __restrict__ src, cpx<T>* __restrict__ dst, int j, int Ns,
                                            int M, DivConst dns, const cpx<T>* W, int dir) {
  const int nb = M / R;
  const int c = div_by(dns, j);
  const int k = j - c * Ns;
  cpx<T> v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = src[j + q * nb];
  const int tstep = k * (nb / Ns);
  if (k) {
#pragma unroll
    for (int q = 1; q < R; ++q) v[q] = mulc<T>(v[q], W[q * tstep], dir > 0);
  }
  if (R == 3) dft3<T>(v, dir);
  else if (R == 5) dft5<T>(v, dir);
  else dft_direct<T, R>(v, W, M, dir);
  const int base = c * Ns * R + k;
#pragma unroll
  for (int q = 0; q < R; ++q) dst[base + q * Ns] = st_norm<T>(v[q]);
}
template <typename T>
__device__ cpx<T>* fft_pencils_small(cpx<T>* a, cpx<T>* b, int G, int ld, const FftPlan& plan, const cpx<T>* W, int dir) {
  const int M = plan.M;
  int Ns = 1;
  cpx<T>* src = a;
  cpx<T>* dst = b;
  for (int s = 0; s < plan.nrad; ++s) {
    const int R = plan.radix[s];
    const int nb = M / R;
    const bool have = plan.ndiv > 0;
    const DivConst dnb = have ? plan.nb[s] : div_const((uint32_t)nb), dns = have ? plan.nsi[s] : div_const((uint32_t)Ns);
    for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
      const int g = div_by(dnb, t);
      const int j = t - g * nb;
      const cpx<T>* sp = src + (size_t)g * ld;
      cpx<T>* dp = dst + (size_t)g * ld;
      switch (R) {
        case 3: stage_small<T, 3>(sp, dp, j, Ns, M, dns, W, dir); break;
        case 5: stage_small<T, 5>(sp, dp, j, Ns, M, dns, W, dir); break;
        case 7: stage_small<T, 7>(sp, dp, j, Ns, M, dns, W, dir); break;
        case 11: stage_small<T, 11>(sp, dp, j, Ns, M, dns, W, dir); break;
        default: stage_small<T, 13>(sp, dp, j, Ns, M, dns, W, dir); break;
      }
    }
    __syncthreads();
    cpx<T>* t = src; src = dst; dst = t;
    Ns *= R;
  }
  return src;
}

// ---------------------------------------------------------------------------------
// Compile-time length M (product of radices 3 and 5): every divisor is a constant.
// ---------------------------------------------------------------------------------
template <typename T, int M, int R, int Ns>
__device__ __forceinline__ void cbfly(const cpx<T>* __restrict__ src, cpx<T>* __restrict__ dst, int j,
                                      const cpx<T>* W, int dir) {
  constexpr int nb = M / R;
  const int k = j % Ns;
  cpx<T> v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = src[j + q * nb];
  if (Ns > 1) {
    constexpr int step = M / (Ns * R);
#pragma unroll
    for (int q = 1; q < R; ++q) v[q] = mulc<T>(v[q], W[q * k * step], dir > 0);
  }
  dft_reg<T, R>(v, dir);
  const int base = (j / Ns) * Ns * R + k;
#pragma unroll
  for (int q = 0; q < R; ++q) dst[base + q * Ns] = st_norm<T>(v[q]);
}

// Radix-3 butterflies of a first stage whose middle inputs are all zero (a zero-padded
// spectrum), and of a last stage whose middle outputs are not needed (a truncated one).
template <typename T, bool F>
__device__ __forceinline__ void dft3_mid_in0(cpx<T>* v, int dir) {   // v[1] == 0
  const T h = T(0.5);
  const cpx<T> a = v[0], c = v[2];
  const cpx<T> t2 = axpy<T>(-h, c, a);
  v[0] = add<T>(a, c);
  if constexpr (F) {
    dft3_sine<T, F>(t2, mk<T>(-c.x, -c.y), dir, &v[1], &v[2]);
  } else {   // the order of a float-float product's factors is part of its rounding
    const T s3 = T(0.86602540378443864676372317075294);
    const cpx<T> it3 = rot<T>(mk<T>(-s3 * c.x, -s3 * c.y), dir > 0 ? 1 : -1);
    v[1] = add<T>(t2, it3);
    v[2] = sub<T>(t2, it3);
  }
}
template <typename T, bool F>
__device__ __forceinline__ void dft3_skip_out1(cpx<T>* v, int dir) {   // v[1] left undefined
  const T h = T(0.5);
  const cpx<T> t1 = add<T>(v[1], v[2]), d = sub<T>(v[1], v[2]);
  const cpx<T> t2 = axpy<T>(-h, t1, v[0]);
  v[0] = add<T>(v[0], t1);
  dft3_sine<T, F>(t2, d, dir, &v[1], &v[2]);
}

// prune bit 1: the first stage (radix 3, stride nb = M/3) reads only inputs j and j + 2 nb
// (the inputs j + nb are zero padding); bit 2: the last stage (radix 3) writes only outputs
// base and base + 2 Ns (the outputs base + Ns are truncated away); bits 4 and 8: the same for
// a radix-15 first / last stage and its zero band (q = 4..10 of the 15 inputs / outputs,
// positions 4 M/15 .. 11 M/15 - 1). The caller checks that the padding / truncation covers
// those positions.
template <typename T, int M, int S, bool BIG>
__device__ __forceinline__ cpx<T>* cfft_from(cpx<T>* a, cpx<T>* b, int G, const cpx<T>* W, int dir,
                                             int prune = 0) {
  if constexpr (S >= cf_nstages(M, BIG)) {
    return a;
  } else {
    constexpr int R = cf_radix(M, S, BIG);
    constexpr int Ns = cf_ns(M, S, BIG);
    constexpr int nb = M / R;
    constexpr bool last = S + 1 == cf_nstages(M, BIG);
    if constexpr (R == 3 && S == 0 && !last) {
      if (prune & 1) {
        for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
          const int g = t / nb;
          const int j = t - g * nb;
          const cpx<T>* src = a + g * M;
          cpx<T> v[3] = {src[j], mk<T>(T(0), T(0)), src[j + 2 * nb]};
          dft3_mid_in0<T>(v, dir);
          cpx<T>* dst = b + g * M;
#pragma unroll
          for (int q = 0; q < 3; ++q) dst[3 * j + q] = st_norm<T>(v[q]);   // Ns = 1: base = 3 j
        }
        __syncthreads();
        return cfft_from<T, M, S + 1, BIG>(b, a, G, W, dir, prune);
      }
    }
    if constexpr (R == 15 && S == 0 && !last) {
      if (prune & 4) {   // radix-15 first stage: inputs j + nb q, q in the zero band, are zero
        for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
          const int g = t / nb;
          const int j = t - g * nb;
          const cpx<T>* src = a + g * M;
          cpx<T> v[15];
#pragma unroll
          for (int q = 0; q < 15; ++q)
            if (!ZeroBand<15>::in(q)) v[q] = src[j + q * nb];
          dft15_zin<T>(v, dir);
          cpx<T>* dst = b + g * M;
#pragma unroll
          for (int q = 0; q < 15; ++q) dst[15 * j + q] = st_norm<T>(v[q]);   // Ns = 1: base = 15 j
        }
        __syncthreads();
        return cfft_from<T, M, S + 1, BIG>(b, a, G, W, dir, prune);
      }
    }
    if constexpr (R == 15 && last && S > 0) {
      if (prune & 8) {   // radix-15 last stage: outputs base + Ns q, q in the zero band, not needed
        for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
          const int g = t / nb;
          const int j = t - g * nb;
          const cpx<T>* src = a + g * M;
          const int k = j % Ns;
          cpx<T> v[15];
#pragma unroll
          for (int q = 0; q < 15; ++q) v[q] = src[j + q * nb];
          if (k) {
            constexpr int step = M / (Ns * R);
#pragma unroll
            for (int q = 1; q < 15; ++q) v[q] = mulc<T>(v[q], W[q * k * step], dir > 0);
          }
          dft15_zout<T>(v, dir);
          cpx<T>* dst = b + g * M;
          const int base = (j / Ns) * Ns * R + k;
#pragma unroll
          for (int q = 0; q < 15; ++q)
            if (!ZeroBand<15>::in(q)) dst[base + q * Ns] = st_norm<T>(v[q]);
        }
        __syncthreads();
        return b;
      }
    }
    if constexpr (R == 3 && last && S > 0) {
      if (prune & 2) {
        for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
          const int g = t / nb;
          const int j = t - g * nb;
          const cpx<T>* src = a + g * M;
          const int k = j % Ns;
          cpx<T> v[3] = {src[j], src[j + nb], src[j + 2 * nb]};
          if (k) {
            constexpr int step = M / (Ns * R);
            v[1] = mulc<T>(v[1], W[k * step], dir > 0);
            v[2] = mulc<T>(v[2], W[2 * k * step], dir > 0);
          }
          dft3_skip_out1<T>(v, dir);
          cpx<T>* dst = b + g * M;
          const int base = (j / Ns) * Ns * R + k;
          dst[base] = st_norm<T>(v[0]);
          dst[base + 2 * Ns] = st_norm<T>(v[2]);
        }
        __syncthreads();
        return b;
      }
    }
    for (int t = threadIdx.x; t < G * nb; t += blockDim.x) {
      const int g = t / nb;
      const int j = t - g * nb;
      cbfly<T, M, R, Ns>(a + g * M, b + g * M, j, W, dir);
    }
    __syncthreads();
    return cfft_from<T, M, S + 1, BIG>(b, a, G, W, dir, prune);
  }
}

// G contiguous pencils of compile-time length M (stride M), ping-pong between a and b.
// FP32 uses the composite register radices (fewer shared-memory passes, and no twiddle products
// inside a prime-factor radix 15); FP64 keeps radices 3 and 5, which need the fewest FP64
// operations, and so does float-float, whose composite radices leave a chunk of pencils too few
// butterflies for a CTA's threads (radix 25 at length 125: 55 of 256) and take 255 registers a
// thread (the float-float operator at N = 63: 1.68 ms; 0.69 ms with radices 5 and two CTAs an SM),
// except at M = 225 = 15 * 15, where the radix-15 stages with the zero band pruned (bits 4 and 8)
// need fewer operations.
constexpr int kBandM64 = 225;
template <typename T, int M>
__device__ __forceinline__ cpx<T>* cfft(cpx<T>* a, cpx<T>* b, int G, const cpx<T>* W, int dir, int prune = 0) {
  return cfft_from<T, M, 0, (sizeof(T) == 4 || is_fpair<T>::value || M == kBandM64)>(a, b, G, W, dir, prune);
}

// Prune bits valid for a length-M transform whose spectrum is nonzero (inverse) or needed
// (forward) only at [0, lo) and (M - lo, M): the middle third of a radix-3 first / last
// stage, [M/3, 2M/3), must lie inside [lo, M - lo].
__host__ __device__ inline bool prune3_ok(int M, int lo) {
  return M % 3 == 0 && M / 3 >= lo && 2 * (M / 3) - 1 <= M - lo;
}

// Deterministic block sum of one double per thread (fixed tree order).
__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    for (int w = 0; w < nw; ++w) s += red[w];
  }
  return s;  // valid in thread 0 only
}

// Frequency of storage index i in FFT order for odd length n.
__device__ __forceinline__ int sfreq(int i, int n) { return i <= (n - 1) / 2 ? i : i - n; }
// The Nyquist frequency k = -n/2 of an even axis: the conforming spaces E_N, J_N of general
// grids exclude it (Def. FD_proj_E: G^E_{N,0}, G^J_{N,0} vanish there), so every N-grid
// field keeps it at zero. Never true on odd axes.
__device__ __forceinline__ bool nyquist(int k, int n) { return (n & 1) == 0 && k == -(n >> 1); }

// Per-side CG scalars (device memory), one slot per right-hand side.
struct CgScalars {
  double rr[3];
  double pq[3];
  double alpha[3];
  double beta[3];
  double tol2[3];    // stop when r.r <= tol2 (per right-hand side)
  double rr_min[3];  // smallest r.r seen (divergence guard of the FP32 inner solves)
  int min_iter[3];   // iteration of the last new minimum of r.r (stagnation guard)
  int active[3];     // 1 while the solve runs
  int iters[3];
  int status[3];     // 0 converged, 1 running / max_iter, 2 stopped by a guard, -2 breakdown
  int guard;         // 1: an FP32 inner solve; breakdown and divergence stop it (status 2)
  int fault;         // 1: a bounded device wait of an operator pass gave up
};

}  // namespace homb
