// dg_dual.cuh -- forward-mode dual numbers for the device and the dual versions
// of the 2D Euler building blocks used by the adjoint kernels: conserved ->
// primitive conversion and the min/max limiter.  A Dn<T, N> carries a value and N tangents; branches are decided on
// values (the derivative of the active branch).
#pragma once

#include "dg_physics.cuh"

namespace dgk {

template <class T, int N>
struct Dn {
  T v;
  T d[N];
  Dn() = default;
  // a constant (zero tangents), so that code written for a scalar type T (its
  // T(0.5), T(1) ...) also runs on Dn<T, N>
  __host__ __device__ Dn(T a) : v(a) {
#pragma unroll
    for (int i = 0; i < N; ++i) d[i] = T(0);
  }
};

template <class T, int N>
__device__ __forceinline__ Dn<T, N> dconst(T a) {
  Dn<T, N> r;
  r.v = a;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = T(0);
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator+(const Dn<T, N>& a, const Dn<T, N>& b) {
  Dn<T, N> r;
  r.v = a.v + b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] + b.d[i];
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator-(const Dn<T, N>& a, const Dn<T, N>& b) {
  Dn<T, N> r;
  r.v = a.v - b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] - b.d[i];
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator-(const Dn<T, N>& a) {
  Dn<T, N> r;
  r.v = -a.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = -a.d[i];
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator*(const Dn<T, N>& a, const Dn<T, N>& b) {
  Dn<T, N> r;
  r.v = a.v * b.v;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * b.v + a.v * b.d[i];
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator/(const Dn<T, N>& a, const Dn<T, N>& b) {
  Dn<T, N> r;
  T ib = T(1) / b.v;
  r.v = a.v * ib;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = (a.d[i] - r.v * b.d[i]) * ib;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator+(const Dn<T, N>& a, T b) {
  Dn<T, N> r = a;
  r.v += b;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator+(T b, const Dn<T, N>& a) { return a + b; }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator-(const Dn<T, N>& a, T b) {
  Dn<T, N> r = a;
  r.v -= b;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator-(T b, const Dn<T, N>& a) {
  Dn<T, N> r = -a;
  r.v += b;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator*(const Dn<T, N>& a, T b) {
  Dn<T, N> r;
  r.v = a.v * b;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * b;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator*(T b, const Dn<T, N>& a) { return a * b; }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator/(const Dn<T, N>& a, T b) { return a * (T(1) / b); }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> operator/(T a, const Dn<T, N>& b) {
  Dn<T, N> r;
  T ib = T(1) / b.v;
  r.v = a * ib;
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = -r.v * b.d[i] * ib;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> dsqrt(const Dn<T, N>& a) {
  Dn<T, N> r;
  r.v = sqrts(a.v);
  T k = r.v > T(0) ? T(0.5) / r.v : T(0);
#pragma unroll
  for (int i = 0; i < N; ++i) r.d[i] = a.d[i] * k;
  return r;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> dabs(const Dn<T, N>& a) { return a.v < T(0) ? -a : a; }

// What the scalar device physics needs besides arithmetic, so that its templates
// (hlld_flux, fast_speed, phys_flux2d) instantiate on Dn<T, N>: comparisons of
// the values (branches follow the value: the derivative of the active branch),
// |x|, the square root, and the solver tolerances of the scalar type.
template <class T, int N>
__device__ __forceinline__ bool operator<(const Dn<T, N>& a, const Dn<T, N>& b) { return a.v < b.v; }
template <class T, int N>
__device__ __forceinline__ bool operator>(const Dn<T, N>& a, const Dn<T, N>& b) { return a.v > b.v; }
template <class T, int N>
__device__ __forceinline__ bool operator<=(const Dn<T, N>& a, const Dn<T, N>& b) { return a.v <= b.v; }
template <class T, int N>
__device__ __forceinline__ bool operator>=(const Dn<T, N>& a, const Dn<T, N>& b) { return a.v >= b.v; }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> fabs(const Dn<T, N>& a) { return dabs(a); }
template <class T, int N>
__device__ __forceinline__ Dn<T, N>& operator*=(Dn<T, N>& a, const Dn<T, N>& b) {
  a = a * b;
  return a;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N>& operator+=(Dn<T, N>& a, const Dn<T, N>& b) {
  a = a + b;
  return a;
}
template <class T, int N>
__device__ __forceinline__ Dn<T, N> sqrtv(const Dn<T, N>& a) { return dsqrt(a); }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> sqrts(const Dn<T, N>& a) { return dsqrt(a); }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> rcpv(const Dn<T, N>& a) { return T(1) / a; }
template <class T, int N>
__device__ __forceinline__ Dn<T, N> rsqrtp(const Dn<T, N>& a) { return T(1) / dsqrt(a); }
template <class T, int N>
__device__ __forceinline__ bool posv(const Dn<T, N>& a) { return posv(a.v); }
template <class T, int N>
__device__ __forceinline__ bool negv(const Dn<T, N>& a) { return a.v < T(0); }
template <class T, int N>
__device__ __forceinline__ bool gt_pos(const Dn<T, N>& a, const Dn<T, N>& b) { return a.v > b.v; }
template <class T, int N>
struct Tiny<Dn<T, N>> {
  static constexpr T v = Tiny<T>::v;
};
template <class T, int N>
struct Prec<Dn<T, N>> {
  static constexpr int newton_max = Prec<T>::newton_max;
  static constexpr T hlld_degenerate = Prec<T>::hlld_degenerate;
};

// Primitive (rho, u, v, p) of conserved (rho, mx, my, E) in 2D, dual.
template <class T, int N>
__device__ __forceinline__ void dprims2d(const Gas<T>& G, const Dn<T, N>* c, Dn<T, N>* W) {
  Dn<T, N> inv = T(1) / c[0];
  Dn<T, N> vx = c[1] * inv, vy = c[2] * inv;
  W[0] = c[0];
  W[1] = vx;
  W[2] = vy;
  W[3] = G.gm1 * (c[3] - T(0.5) * (c[1] * vx + c[2] * vy));
}

// Dual min/max limiter of one 2D Euler cell (Sec. 2.5): c0/s its averages and
// derivative coefficients, cn[k] the averages of its 4 face neighbours; s is
// replaced by the limited coefficients.
template <class T, int N>
__device__ void dlimit_cell2d(const Gas<T>& G, const T* hh, const Dn<T, N>* c0,
                              const Dn<T, N> (*cn)[4], Dn<T, N>* s) {
  typedef Dn<T, N> D;
  D W[4], Wn[4][4];
  dprims2d<T, N>(G, c0, W);
#pragma unroll
  for (int k = 0; k < 4; ++k) dprims2d<T, N>(G, cn[k], Wn[k]);
  const D inv = T(1) / W[0];
  D gr[2], gvx[2], gvy[2], gp[2];
  const D v2h = T(0.5) * (W[1] * W[1] + W[2] * W[2]);
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    gr[d] = s[d];
    gvx[d] = (s[2 + d] - W[1] * gr[d]) * inv;
    gvy[d] = (s[4 + d] - W[2] * gr[d]) * inv;
    gp[d] = G.gm1 * (s[6 + d] - v2h * gr[d] - W[0] * (W[1] * gvx[d] + W[2] * gvy[d]));
  }
  D alpha[4];
  const D* grads[4] = {gr, gvx, gvy, gp};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    D hi = W[q], lo = W[q];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (Wn[k][q].v > hi.v) hi = Wn[k][q];
      if (Wn[k][q].v < lo.v) lo = Wn[k][q];
    }
    D a0 = dabs(grads[q][0] * hh[0]), a1 = dabs(grads[q][1] * hh[1]);
    D amax = a1.v > a0.v ? a1 : a0;
    if (!(amax.v > T(0))) {
      alpha[q] = dconst<T, N>(T(1));
    } else {
      D up = hi - W[q], dn = W[q] - lo;
      D m = up.v < dn.v ? up : dn;
      D psi = m / amax;
      alpha[q] = psi.v < T(1) ? psi : dconst<T, N>(T(1));
    }
  }
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    D r = alpha[0] * gr[d], ux = alpha[1] * gvx[d], uy = alpha[2] * gvy[d], pp = alpha[3] * gp[d];
    s[d] = r;
    s[2 + d] = W[0] * ux + W[1] * r;
    s[4 + d] = W[0] * uy + W[2] * r;
    s[6 + d] = pp * G.inv_gm1 + v2h * r + W[0] * (W[1] * ux + W[2] * uy);
  }
}

}  // namespace dgk
