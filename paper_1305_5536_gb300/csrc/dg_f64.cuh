// dg_f64.cuh -- FP64 building blocks for the narrow FP64 pipe of sm_103a.
//
// The chip executes two FP64 operations per SM and cycle (a warp-wide DADD, DMUL,
// DFMA or DSETP holds a sub-partition's pipe for 64 cycles), so the FP64 kernels are
// bound by the number of FP64 instructions.  What can run elsewhere does: seeds come
// from the special-function unit (rcp.approx / rsqrt.approx on the high word),
// comparisons, exponents and tables from the integer pipe.
//   rcpv     1/x: one cubically convergent step r (1 + e + e^2), e = 1 - x r, from the
//            ~20-bit seed: 3 FP64 operations, within about 1 ulp.
//   rsqrt64, sqrt64: one cubic (Householder) step y (1 + e/2 + 3e^2/8), e = 1 - x y^2:
//            5 FP64 operations.
//   pow_m1   x^z and x^z - 1 by log2 and exp2 with a table of 2^(i/64) and Taylor
//            polynomials on the remainders (|ln| <= 0.0055): about 22 operations;
//            x^z - 1 keeps its relative accuracy near x = 1.
#pragma once

#include <cuda_runtime.h>

namespace dgk {

// x > 0 and not NaN (+inf is positive), without a comparison on the FP64 pipe.
__device__ __forceinline__ bool posv(double x) {
  return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool posv(float x) { return x > 0.0f; }

// a > b for positive a and b (or a NaN on neither side).
__device__ __forceinline__ bool gt_pos(double a, double b) {
  return __double_as_longlong(a) > __double_as_longlong(b);
}
__device__ __forceinline__ bool gt_pos(float a, float b) { return a > b; }

// x < 0 by the sign bit (-0 counts as negative).
__device__ __forceinline__ bool negv(double x) { return __double2hiint(x) < 0; }
__device__ __forceinline__ bool negv(float x) { return x < 0.0f; }

// Running maximum and minimum of a few values.  FP64 compares the integer images that
// order like the doubles: no comparison on the FP64 pipe.
template <class T>
struct Extremes {
  T hi, lo;
  __device__ __forceinline__ explicit Extremes(T x) : hi(x), lo(x) {}
  __device__ __forceinline__ void add(T x) {
    hi = x > hi ? x : hi;
    lo = x < lo ? x : lo;
  }
  __device__ __forceinline__ void add(T x, T y) { add(x); add(y); }
  __device__ __forceinline__ T max() const { return hi; }
  __device__ __forceinline__ T min() const { return lo; }
};
template <>
struct Extremes<double> {
  long long hi, lo;
  __device__ __forceinline__ static long long image(long long b) {
    return b ^ (long long)((unsigned long long)(b >> 63) >> 1);
  }
  __device__ __forceinline__ explicit Extremes(double x) {
    hi = lo = image(__double_as_longlong(x));
  }
  __device__ __forceinline__ void add(double x) {
    const long long k = image(__double_as_longlong(x));
    hi = k > hi ? k : hi;
    lo = k < lo ? k : lo;
  }
  __device__ __forceinline__ void add(double x, double y) { add(x); add(y); }
  __device__ __forceinline__ double max() const { return __longlong_as_double(image(hi)); }
  __device__ __forceinline__ double min() const { return __longlong_as_double(image(lo)); }
};

// x is neither zero, subnormal, infinite nor NaN.  For every such x the refinements below
// stay in range (a reciprocal below 2^-1022 comes out as zero).
__device__ __forceinline__ bool normal(double x) {
  return ((((unsigned)__double2hiint(x) >> 20) & 0x7ffu) - 1u) < 2046u;
}

// 1/x; 1/0 = inf, 1/inf = 0, NaN.  Subnormal operands count as zero and subnormal results
// are zero.  (A branch to CUDA's own division, root and power for these breaks the chains
// of the solvers into blocks: 3D Euler 64^3 4499 -> 4786 us, 2D MHD 512^2 2964 -> 3029.)
__device__ __forceinline__ double rcpv(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  const double y = fma(r, fma(e, e, e), r);
  return normal(x) ? y : r;
}

// 1/sqrt(x); 1/0 = inf, 1/inf = 0, NaN.  Subnormal operands count as zero.
__device__ __forceinline__ double rsqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  const double s = fma(y * e, fma(0.375, e, 0.5), y);
  return normal(x) ? s : y;
}

// sqrt(x); zero, infinite, NaN and subnormal operands are returned as they are, a negative
// one gives a NaN.
__device__ __forceinline__ double sqrt64(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y;
  const double e = fma(-t, y, 1.0);
  const double s = fma(t * e, fma(0.375, e, 0.5), t);
  return normal(x) ? s : x;
}

// FP32: three-operand minimum and maximum (a NaN operand is passed over, as by the
// comparisons of the general form).
template <>
struct Extremes<float> {
  float hi, lo;
  __device__ __forceinline__ explicit Extremes(float x) { hi = lo = x; }
  __device__ __forceinline__ void add(float x, float y) {
    asm("max.f32 %0, %1, %2, %3;" : "=f"(hi) : "f"(hi), "f"(x), "f"(y));
    asm("min.f32 %0, %1, %2, %3;" : "=f"(lo) : "f"(lo), "f"(x), "f"(y));
  }
  __device__ __forceinline__ float max() const { return hi; }
  __device__ __forceinline__ float min() const { return lo; }
};

// The same operations of the FP32 path: one special-function instruction each (1 to 2
// ulp).  The flushing forms leave out the scaling that subnormal operands would need
// (3 more instructions a call): the averages are flushed when they are converted.
__device__ __forceinline__ float rcpv(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sqrtv(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// A root whose operand may be subnormal: a square of velocities (from 1e-19 on), a fourth
// power of them (from 3e-10 on).
__device__ __forceinline__ float sqrts(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrtp(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2v(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float lg2v(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double sqrtv(double x) { return sqrt64(x); }
__device__ __forceinline__ double sqrts(double x) { return sqrt64(x); }
__device__ __forceinline__ double rsqrtp(double x) { return rsqrt64(x); }

// The smallest normal number of a type: slopes below it count as zero.
template <class T>
struct Tiny;
template <>
struct Tiny<double> {
  static constexpr double v = 2.2250738585072014e-308;
};
template <>
struct Tiny<float> {
  static constexpr float v = 1.17549435e-38f;
};

// 2^(i/64), i = 0 .. 64, rounded to FP64.
__device__ const double kExp2Tab[65] = {
    0x1.0000000000000p+0, 0x1.02c9a3e778061p+0, 0x1.059b0d3158574p+0,
    0x1.0874518759bc8p+0, 0x1.0b5586cf9890fp+0, 0x1.0e3ec32d3d1a2p+0,
    0x1.11301d0125b51p+0, 0x1.1429aaea92de0p+0, 0x1.172b83c7d517bp+0,
    0x1.1a35beb6fcb75p+0, 0x1.1d4873168b9aap+0, 0x1.2063b88628cd6p+0,
    0x1.2387a6e756238p+0, 0x1.26b4565e27cddp+0, 0x1.29e9df51fdee1p+0,
    0x1.2d285a6e4030bp+0, 0x1.306fe0a31b715p+0, 0x1.33c08b26416ffp+0,
    0x1.371a7373aa9cbp+0, 0x1.3a7db34e59ff7p+0, 0x1.3dea64c123422p+0,
    0x1.4160a21f72e2ap+0, 0x1.44e086061892dp+0, 0x1.486a2b5c13cd0p+0,
    0x1.4bfdad5362a27p+0, 0x1.4f9b2769d2ca7p+0, 0x1.5342b569d4f82p+0,
    0x1.56f4736b527dap+0, 0x1.5ab07dd485429p+0, 0x1.5e76f15ad2148p+0,
    0x1.6247eb03a5585p+0, 0x1.6623882552225p+0, 0x1.6a09e667f3bcdp+0,
    0x1.6dfb23c651a2fp+0, 0x1.71f75e8ec5f74p+0, 0x1.75feb564267c9p+0,
    0x1.7a11473eb0187p+0, 0x1.7e2f336cf4e62p+0, 0x1.82589994cce13p+0,
    0x1.868d99b4492edp+0, 0x1.8ace5422aa0dbp+0, 0x1.8f1ae99157736p+0,
    0x1.93737b0cdc5e5p+0, 0x1.97d829fde4e50p+0, 0x1.9c49182a3f090p+0,
    0x1.a0c667b5de565p+0, 0x1.a5503b23e255dp+0, 0x1.a9e6b5579fdbfp+0,
    0x1.ae89f995ad3adp+0, 0x1.b33a2b84f15fbp+0, 0x1.b7f76f2fb5e47p+0,
    0x1.bcc1e904bc1d2p+0, 0x1.c199bdd85529cp+0, 0x1.c67f12e57d14bp+0,
    0x1.cb720dcef9069p+0, 0x1.d072d4a07897cp+0, 0x1.d5818dcfba487p+0,
    0x1.da9e603db3285p+0, 0x1.dfc97337b9b5fp+0, 0x1.e502ee78b3ff6p+0,
    0x1.ea4afa2a490dap+0, 0x1.efa1bee615a27p+0, 0x1.f50765b6e4540p+0,
    0x1.fa7c1819e90d8p+0, 0x1.0000000000000p+1};

// x^z for positive normal x and |z| <= 1/2; returns x^z - 1 and, in w, x^z (zero and
// subnormal x as the smallest normal number).
//   x = 2^(e+1) h, h in [1/2, 1);  k = 64 (1 + log2 h) to the nearest integer (FP32);
//   r = h 2^((64-k)/64) - 1, |r| < 0.0056;  log2 x = (64 e + k)/64 + log2(1 + r);
//   z log2 x = n/64 + f, |f| <= 1/128;  x^z = 2^(n/64) 2^f.
// log2(1 + r) and 2^f - 1 by Taylor polynomials of degree 7 and 6 (truncation
// 2e-17 and 5e-18 relative): the table-driven scheme of Tang (ACM TOMS 1989, 1990).
__device__ __forceinline__ double pow_m1(double x, double z, double& w) {
  const int hx = __double2hiint(x), lx = __double2loint(x);
  const int e = (hx >> 20) - 1023;
  const float m = __int_as_float(0x3f800000 | ((hx & 0x000fffff) << 3) | ((unsigned)lx >> 29));
  int k = __float2int_rn(64.0f * lg2v(m));
  k = k < 0 ? 0 : (k > 64 ? 64 : k);
  const double h = __hiloint2double((hx & 0x000fffff) | 0x3fe00000, lx);
  const double r = fma(h, __ldg(&kExp2Tab[64 - k]), -1.0);
  double q = 0.2060992915555662;
  q = fma(q, r, -0.2404491734814939);
  q = fma(q, r, 0.28853900817779266);
  q = fma(q, r, -0.36067376022224085);
  q = fma(q, r, 0.4808983469629878);
  q = fma(q, r, -0.7213475204444817);
  q = fma(q, r, 1.4426950408889634);
  // integers to FP64 by the 1.5 * 2^52 shift
  constexpr double shift = 6755399441055744.0;
  const double nk = __hiloint2double(0x43380000 + ((64 * e + k) >> 31), 64 * e + k) - shift;
  const double y = fma(z * 0.015625, nk, z * (q * r));
  const double ys = fma(y, 64.0, shift);
  const int n = __double2loint(ys);
  const double f = fma(ys - shift, -0.015625, y);
  double p = 0.0001540353039338161;
  p = fma(p, f, 0.0013333558146428443);
  p = fma(p, f, 0.009618129107628477);
  p = fma(p, f, 0.05550410866482158);
  p = fma(p, f, 0.24022650695910072);
  p = fma(p, f, 0.6931471805599453);
  p *= f;
  const double t0 = __ldg(&kExp2Tab[n & 63]);
  const double t = __hiloint2double(__double2hiint(t0) + ((n >> 6) << 20), __double2loint(t0));
  w = fma(t, p, t);
  return fma(t, p, t - 1.0);
}

}  // namespace dgk
