// dg_physics.cuh -- device physics of the P1 DG step (sm_103a).
//
// Inline device functions, templated on the arithmetic type T (double for the
// FP64 path, float for the FP32 path):
//   * gas constants and the fast magnetosonic speed (Sec. 2.1),
//   * the exact Riemann solver of the Euler equations (Sec. 2.3; Newton iteration
//     on the pressure function with the adaptive PVRS/TRRS/TSRS first guess of
//     Toro's textbook, sampled at x/t = 0),
//   * the HLLD solver of Miyoshi & Kusano (2005) for planar ideal MHD and with two
//     transverse components for 3D MHD (Sec. 2.3),
//   * the min/max slope limiter of one cell on primitive variables (Sec. 2.5).
// Face solvers work in the face frame: normal velocity u, transverse velocities,
// and return fluxes in that frame.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "dg_f64.cuh"

namespace dgk {

enum : unsigned {
  ERR_NONPHYS = 1u,   // rho <= 0 or p <= 0 at an evaluated state
  ERR_VACUUM = 2u,    // the exact solver met a vacuum-generating pair
  ERR_NEWTON = 4u,    // Newton iteration for p* did not converge
  ERR_TIMEOUT = 8u,   // a bounded device wait (grid barrier, TMA completion) ran out
};

template <class T> struct Prec;
template <> struct Prec<double> {
  static constexpr int newton_max = 50;
  static constexpr double hlld_degenerate = 1e-8;
};
template <> struct Prec<float> {
  static constexpr int newton_max = 20;
  static constexpr float hlld_degenerate = 1e-8f;
};

// Powers in the exact solver (positive bases only).  FP64: the accurate pow.
// FP32: the __powf intrinsic (exp2 of e * log2 x on the special-function unit),
// a few ulp for the exponents used here, ~10x fewer instructions than powf.
__device__ __forceinline__ double rpow(double x, double e) { return pow(x, e); }
__device__ __forceinline__ float rpow(float x, float e) { return __powf(x, e); }

// Conversions between the FP64 cell averages and the arithmetic type.  For the
// FP32 path they are done with integer operations on the IEEE-754 bit patterns,
// because GB300 executes FP64<->FP32 conversions on its narrow FP64 pipe.  The
// word-level rules are plain functions of the bit patterns (host and device), so
// that they can be checked on the CPU:
//   f32_bits_of_f64(hi, lo): rebias the exponent (1023 -> 127), keep the top 23
//     mantissa bits rounded to nearest (ties away from zero).  Magnitudes below
//     the smallest normal float become a zero of the same sign; magnitudes that
//     round to 2^128 or above become an infinity of the same sign; infinities stay
//     infinities and every NaN becomes the quiet NaN 0x7fc00000 (with its sign).
//   f64_words_of_f32(u): exact widening; subnormal floats become a zero of the
//     same sign, infinities and NaNs keep their class (a NaN keeps its payload).
__host__ __device__ __forceinline__ unsigned f32_bits_of_f64(unsigned h0, unsigned l0) {
  const unsigned mag = h0 & 0x7fffffffu;                   // magnitude before rounding
  const unsigned lo = l0 + 0x10000000u;                     // round at the float's last bit
  const unsigned hi = mag + (lo < l0 ? 1u : 0u);            // magnitude, with the carry
  unsigned r = ((hi - (896u << 20)) << 3) | (lo >> 29);
  r = hi < (897u << 20) ? 0u : r;                           // below the float range: zero
  r = hi >= (1151u << 20) ? 0x7f800000u : r;                // rounds to 2^128 or above: inf
  const bool special = mag >= 0x7ff00000u;                  // the double is inf or NaN
  const bool nan = mag > 0x7ff00000u || (mag == 0x7ff00000u && l0 != 0u);
  r = special ? (nan ? 0x7fc00000u : 0x7f800000u) : r;
  return r | (h0 & 0x80000000u);
}
__host__ __device__ __forceinline__ void f64_words_of_f32(unsigned u, unsigned& hi,
                                                          unsigned& lo) {
  const unsigned m = u & 0x7fffffffu;
  const unsigned e = m >= 0x7f800000u ? (0x7ff00000u | ((m & 0x007fffffu) >> 3))  // inf / NaN
                                      : ((m >> 3) + (896u << 20));
  const bool tiny = m < 0x00800000u;
  hi = (u & 0x80000000u) | (tiny ? 0u : e);
  lo = tiny ? 0u : m << 29;
}

template <class T> struct Cvt;
template <> struct Cvt<double> {
  __device__ __forceinline__ static double to_tc(double x) { return x; }
  __device__ __forceinline__ static double to_f64(double x) { return x; }
};
template <> struct Cvt<float> {
  // On the two 32-bit halves: masking the sign of the 64-bit pattern would be
  // compiled as a double absolute value, an FP64-pipe instruction.
  __device__ __forceinline__ static float to_tc(double x) {
    return __int_as_float((int)f32_bits_of_f64((unsigned)__double2hiint(x),
                                               (unsigned)__double2loint(x)));
  }
  __device__ __forceinline__ static double to_f64(float f) {
    unsigned hi, lo;
    f64_words_of_f32((unsigned)__float_as_int(f), hi, lo);
    return __hiloint2double((int)hi, (int)lo);
  }
};

// A Courant signal speed sp of a cell with density rho and pressure p that a time
// step can be taken from: finite and non-negative, and the state itself finite
// (an infinite density has zero velocity and sound speed, so sp alone would pass).
template <class T>
__device__ __forceinline__ bool courant_ok(T sp, T rho, T p) {
  const T inf = T(INFINITY);
  return sp >= T(0) && sp < inf && rho < inf && p < inf;
}

// x / 2 without the FP64 pipe: the exponent field lowered by one (integer work on
// the high word).  Exact for finite |x| >= 2^-1021; infinities and NaNs are
// returned as they are; smaller magnitudes (including zero) give a zero of the
// sign of x.
__device__ __forceinline__ double half_f64(double x) {
  const int h = __double2hiint(x), l = __double2loint(x);
  const int e = h & 0x7ff00000;
  const bool keep = e == 0x7ff00000, big = e > 0x00100000 && !keep;
  return __hiloint2double(keep ? h : (big ? h - 0x00100000 : (h & (int)0x80000000)),
                          keep || big ? l : 0);
}

// Constants of the equation of state p_gas = (gamma - 1) rho u.
template <class T>
struct GasConst {
  T g, gm1, gp1, inv_gm1;
  T z;        // (g-1)/(2g)
  T inv_z;    // 2g/(g-1)
  T g6;       // (g-1)/(g+1)
  T shk1;     // (g+1)/(2g)
  T inv_g;    // 1/g
  T two_gm1;  // 2/(g-1)
  T two_gp1;  // 2/(g+1)
  __host__ __device__ void set(double gamma) {
    g = T(gamma);
    gm1 = T(gamma - 1.0);
    gp1 = T(gamma + 1.0);
    inv_gm1 = T(1.0 / (gamma - 1.0));
    z = T((gamma - 1.0) / (2.0 * gamma));
    inv_z = T(2.0 * gamma / (gamma - 1.0));
    g6 = T((gamma - 1.0) / (gamma + 1.0));
    shk1 = T((gamma + 1.0) / (2.0 * gamma));
    inv_g = T(1.0 / gamma);
    two_gm1 = T(2.0 / (gamma - 1.0));
    two_gp1 = T(2.0 / (gamma + 1.0));
  }
};
template <class T>
struct Gas : GasConst<T> {};
// FP64 carries the FP32 constants too: the exact solver's first guess is FP32.
template <>
struct Gas<double> : GasConst<double> {
  GasConst<float> lo;
  __host__ __device__ void set(double gamma) {
    GasConst<double>::set(gamma);
    lo.set(gamma);
  }
};

// Square of the fast magnetosonic speed along a direction with normal field bn; ir =
// 1/rho.
template <class T>
__device__ __forceinline__ T fast_speed2(const Gas<T>& G, T ir, T p, T b2, T bn) {
  const T a2 = G.g * p * ir;
  const T s = a2 + b2 * ir;
  T disc = s * s - T(4) * a2 * (bn * bn * ir);
  disc = negv(disc) ? T(0) : disc;
  return T(0.5) * (s + sqrts(disc));
}
template <class T>
__device__ __forceinline__ T fast_speed(const Gas<T>& G, T rho, T p, T b2, T bn) {
  return sqrtv(fast_speed2(G, rcpv(rho), p, b2, bn));
}

// ----------------------------------------------------------------------------
// Exact Riemann solver (Euler).  NT transverse velocity components.
// Output F[0] mass, F[1] normal momentum, F[2..1+NT] transverse momenta,
// F[2+NT] energy -- all in the face frame.
// ----------------------------------------------------------------------------
// Adaptive PVRS / two-rarefaction / two-shock first guess of the star-region pressure
// (Toro's choice) in FP64, for states outside the FP32 range; at least the floor 1e-10
// min(pL, pR).
__device__ __forceinline__ double exact_guess(const Gas<double>& G, double rL, double pL, double cL,
                                              double rR, double pR, double cR, double du,
                                              double pfloor) {
  double pv = 0.5 * (pL + pR) - 0.125 * du * (rL + rR) * (cL + cR);
  pv = pv > 0.0 ? pv : 0.0;
  const double pmin = pL < pR ? pL : pR, pmax = pL < pR ? pR : pL;
  double p;
  if (pmax / pmin <= 2.0 && pmin <= pv && pv <= pmax) {
    p = pv;
  } else if (pv < pmin) {
    const double num = cL + cR - 0.5 * G.gm1 * du;
    const double den = cL / rpow(pL, G.z) + cR / rpow(pR, G.z);
    p = rpow((num > 0.0 ? num : 0.0) / den, G.inv_z);
  } else {
    const double gL = sqrt(G.two_gp1 / rL / (G.g6 * pL + pv));
    const double gR = sqrt(G.two_gp1 / rR / (G.g6 * pR + pv));
    p = (gL * pL + gR * pR - du) / (gL + gR);
  }
  return p > pfloor ? p : pfloor;
}

// ----------------------------------------------------------------------------
// The exact Riemann solver of the FP32 path.  It computes the solution of
// exact_flux (Toro's exact solver: Newton iteration for p* on f_L + f_R + du = 0
// from the adaptive PVRS / TRRS / TSRS guess, sampled at x/t = 0) with the
// arithmetic arranged for the FP32 pipes:
//   * per side, the constants of the pressure function are formed once:
//       shock       f = (p - pK) q,  q = A_K^(1/2) y,  y = (p + B_K)^(-1/2),
//                   f' = q (1 - (p - pK) / (2 (p + B_K))) = q (1 - (p - pK) y^2 / 2)
//                   (two roots, so that density times pressure need not be in range: in
//                   cgs units it is 1e-40 in diffuse interstellar gas),
//       rarefaction f = 2 cK / (g - 1) ((p/pK)^z - 1),  f' = (p/pK)^z cK / (g p),
//     with A_K = 2 / ((g + 1) rho_K), B_K = (g - 1) / (g + 1) pK, z = (g - 1) / (2g);
//     divisions become approximate reciprocals, square roots reciprocal square
//     roots, powers exp2(e log2 x) (all within a few ulp);
//   * both branches of f are evaluated and one is selected, so that lanes of a
//     warp on different branches (near-equal states put p on either side of pK
//     at random) do not serialise;
//   * Newton converges quadratically: accepting the update p_n after a step of
//     relative size delta leaves an error of about k delta^2 (k <= 1/2 for these
//     pressure functions), so steps below 2e-4 are accepted (error < 2e-8, below
//     the FP32 evaluation noise of f), and f_K(p*) for u* is taken from the last
//     iteration's linearisation f_K(p) + f_K'(p)(p* - p) (error O(delta^2) again);
//   * the sampling picks the side of the contact by select and mirrors the right
//     side onto the left (u -> -u), so the unperturbed / shock-star /
//     rarefaction-star choice is a select; only the transonic rarefaction fan,
//     which is rare, is a branch.
// ----------------------------------------------------------------------------

// The first guess and Newton iteration above: p* and the last linearisation, taken at
// p0 (f_K, f_K' there).
struct Star32 {
  float p, p0, fL, fR, dfL, dfR;
  bool conv;
};
__device__ __forceinline__ Star32 star_f32(const GasConst<float>& G, float rL, float pL, float ipL,
                                           float cL, float rR, float pR, float ipR, float cR,
                                           float du) {
  constexpr float accept = 2e-4f;
  const float AL = rsqrtp(0.5f * G.gp1 * rL), AR = rsqrtp(0.5f * G.gp1 * rR);  // A_K^(1/2)
  const float BL = G.g6 * pL, BR = G.g6 * pR;
  const float CL = G.two_gm1 * cL, CR = G.two_gm1 * cR;          // 2 cK / (g - 1)
  const float DL = cL * G.inv_g, DR = cR * G.inv_g;              // cK / g
  // first guess (Toro's adaptive choice)
  const float pmin = fminf(pL, pR), pmax = fmaxf(pL, pR);
  float pv = 0.5f * (pL + pR) - 0.125f * du * (rL + rR) * (cL + cR);
  pv = fmaxf(pv, 0.0f);
  float p = pv;
  if (!(pmax <= 2.0f * pmin && pmin <= pv && pv <= pmax)) {
    if (pv < pmin) {  // two rarefactions
      const float num = fmaxf(cL + cR - 0.5f * G.gm1 * du, 0.0f);
      const float den = cL * ex2v(-G.z * lg2v(pL)) + cR * ex2v(-G.z * lg2v(pR));
      p = ex2v(G.inv_z * lg2v(num * rcpv(den)));
    } else {  // two shocks
      const float gL = AL * rsqrtp(BL + pv), gR = AR * rsqrtp(BR + pv);
      p = (gL * pL + gR * pR - du) * rcpv(gL + gR);
    }
  }
  const float pfloor = 1e-10f * pmin;
  if (!(p > pfloor)) p = pfloor;
  Star32 S = {p, p, 0.0f, 0.0f, 1.0f, 1.0f, false};
  for (int it = 0; it < Prec<float>::newton_max; ++it) {
    const float rp = rcpv(p);
    {
      const float dp = p - pL;
      const float y = rsqrtp(p + BL), q = AL * y;
      const float fs = dp * q, dfs = q * (1.0f - 0.5f * dp * y * y);
      const float qr = ex2v(G.z * lg2v(p * ipL));
      const float fr = CL * (qr - 1.0f), dfr = qr * DL * rp;
      const bool sh = p > pL;
      S.fL = sh ? fs : fr;
      S.dfL = sh ? dfs : dfr;
    }
    {
      const float dp = p - pR;
      const float y = rsqrtp(p + BR), q = AR * y;
      const float fs = dp * q, dfs = q * (1.0f - 0.5f * dp * y * y);
      const float qr = ex2v(G.z * lg2v(p * ipR));
      const float fr = CR * (qr - 1.0f), dfr = qr * DR * rp;
      const bool sh = p > pR;
      S.fR = sh ? fs : fr;
      S.dfR = sh ? dfs : dfr;
    }
    float pn = p - (S.fL + S.fR + du) * rcpv(S.dfL + S.dfR);
    if (!(pn > pfloor)) pn = pfloor;
    S.p0 = p;
    const bool done = 2.0f * fabsf(pn - p) < accept * (pn + p);
    p = pn;
    if (done) { S.conv = true; break; }
  }
  S.p = p;
  return S;
}

template <int NT>
__device__ __forceinline__ void exact_flux_f32(const Gas<float>& G, float rL, float uL, float pL,
                                               const float* vtL, float rR, float uR, float pR,
                                               const float* vtR, float* F, unsigned& err) {
  if (!(rL > 0.0f && pL > 0.0f && rR > 0.0f && pR > 0.0f)) {
    err |= ERR_NONPHYS;
    for (int q = 0; q < 3 + NT; ++q) F[q] = 0.0f;
    return;
  }
  const float ipL = rcpv(pL), ipR = rcpv(pR);
  const float aL = G.g * pL * rcpv(rL), aR = G.g * pR * rcpv(rR);
  const float cL = sqrts(aL), cR = sqrts(aR);
  const float du = uR - uL;
  if (G.two_gm1 * cL + G.two_gm1 * cR <= du) err |= ERR_VACUUM;
  const Star32 S = star_f32(G, rL, pL, ipL, cL, rR, pR, ipR, cR, du);
  if (!S.conv) err |= ERR_NEWTON;
  const float p = S.p;
  // u* from the pressure functions at p*, by the last linearisation
  const float dps = p - S.p0;
  const float us = 0.5f * (uL + uR) + 0.5f * ((S.fR + S.dfR * dps) - (S.fL + S.dfL * dps));
  // sample at x/t = 0 on the side of the contact that x/t = 0 lies on, the right
  // side mirrored onto the left (velocities negated)
  const bool left = us >= 0.0f;
  const float sg = left ? 1.0f : -1.0f;
  const float rK = left ? rL : rR, pK = left ? pL : pR, cK = left ? cL : cR;
  const float ipK = left ? ipL : ipR;
  const float w = sg * (left ? uL : uR), ws = sg * us;
  const float pr = p * ipK;
  const bool shock = p > pK;
  const float Ssh = w - cK * sqrtv(G.shk1 * pr + G.z);         // shock speed
  const float rsh = rK * (pr + G.g6) * rcpv(G.g6 * pr + 1.0f);      // behind the shock
  const float lpr = lg2v(pr);
  const float cm = cK * ex2v(G.z * lpr);                           // sound speed behind the fan
  const float rrf = rK * ex2v(G.inv_g * lpr);                      // isentropic star density
  const bool unpert = shock ? Ssh >= 0.0f : w - cK >= 0.0f;
  const bool fan = !shock && !unpert && !(ws - cm < 0.0f);
  float rho = unpert ? rK : (shock ? rsh : rrf);
  float u = unpert ? w : ws;
  float pp = unpert ? pK : p;
  if (fan) {
    const float c = G.two_gp1 * (cK + 0.5f * G.gm1 * w);
    const float lc = lg2v(c * rcpv(cK));
    u = c;
    rho = rK * ex2v(G.two_gm1 * lc);
    pp = pK * ex2v(G.inv_z * lc);
  }
  u *= sg;
  float vt[NT > 0 ? NT : 1];
  float kin = u * u;
#pragma unroll
  for (int a = 0; a < NT; ++a) {
    vt[a] = left ? vtL[a] : vtR[a];
    kin += vt[a] * vt[a];
  }
  const float E = pp * G.inv_gm1 + 0.5f * rho * kin;
  const float mu = rho * u;
  F[0] = mu;
  F[1] = mu * u + pp;
#pragma unroll
  for (int a = 0; a < NT; ++a) F[2 + a] = mu * vt[a];
  F[2 + NT] = u * (E + pp);
}

// ----------------------------------------------------------------------------
// The exact Riemann solver of the FP64 path: the same solution, to FP64 accuracy, with
// as few FP64 operations as the narrow pipe asks for:
//   * the adaptive first guess and the Newton iteration run in FP32 (p within about
//     5e-7; an FP64 guess takes its place where a state leaves the FP32 range);
//   * one FP64 evaluation of f_L, f_R and their derivatives there, one Halley step (the
//     curvature from FP32): the step is cubic, so an update of relative size below 2e-6
//     is accepted (error left below 1e-17), else the evaluation is repeated;
//   * the pressure functions at p* for u* by their second-order Taylor expansion about
//     the last point (error of order 1e-18), and p/p_K^z at p* likewise;
//   * one power per side, (p/p_K)^z = w: the isentropic density is rho_K (p/p_K) / w^2;
//   * a shock speed whose sign FP32 decides (margin 1e-5 of it) is not formed in FP64.
// About 200 FP64 operations a solve instead of above 2000 (pow in three or more Newton
// evaluations, a re-evaluation and the sampling): 3D Euler 64^3 step 29.0 -> 5.3 ms, 2D
// Euler 64^2 step 772 -> 154 us.
// ----------------------------------------------------------------------------
// Pressure function of one side at p: f, f' and, for p <= pK, w = (p/pK)^z (0 where the
// side is a shock at p); x = p/pK.
__device__ __forceinline__ void side_f64(const Gas<double>& G, double p, double ip, double rK,
                                         double pK, double x, double cK, double& f, double& df,
                                         double& w) {
  if (gt_pos(p, pK)) {
    const double Ai = (0.5 * G.gp1) * rK, dp = p - pK;  // 1 / A_K
    const double q = rsqrt64(fma(G.g6, pK, p) * Ai);
    f = dp * q;
    df = fma(-0.5 * f, q * q * Ai, q);
    w = 0.0;
  } else {
    const double wm1 = pow_m1(x, G.z, w);
    f = (G.two_gm1 * cK) * wm1;
    df = (cK * G.inv_g) * (w * ip);
  }
}

// p f''/f' of one side at x = p/pK (FP32): for a shock, f'' = -q (p + 4 B + 3 pK) /
// (4 (p + B)^2) and f' = q (p + 2 B + pK) / (2 (p + B)); here B in units of pK.  By
// r = 1/x, a product of bounded factors (x^2 leaves the FP32 range from x = 1.8e19 on);
// -1/2 for the strongest shocks, also where x itself leaves that range (r = 0).
__device__ __forceinline__ float curvature_f32(const GasConst<float>& G, float x) {
  const float B = G.g6;
  const float r = rcpv(x);
  const float sh = -0.25f * fmaf(4.0f * B + 3.0f, r, 1.0f) *
                   rcpv(fmaf(B, r, 1.0f) * fmaf(0.5f + B, r, 0.5f));
  return x > 1.0f ? sh : -G.shk1;
}

struct Star64 {
  double p;       // p*
  double step;    // p* - (point of the last evaluation), relative to that point
  double uj;      // f_R(p*) - f_L(p*)
  double wL, wR;  // (p/p_K)^z at the point of the last evaluation (0 on a shock side)
};
__device__ __forceinline__ Star64 star_f64(const Gas<double>& G, double rL, double pL, double ipL,
                                           double cL, double rR, double pR, double ipR, double cR,
                                           double du, unsigned& err) {
  const GasConst<float>& H = G.lo;
  const float pLf = Cvt<float>::to_tc(pL), pRf = Cvt<float>::to_tc(pR);
  const Star32 S = star_f32(H, Cvt<float>::to_tc(rL), pLf, rcpv(pLf), Cvt<float>::to_tc(cL),
                            Cvt<float>::to_tc(rR), pRf, rcpv(pRf), Cvt<float>::to_tc(cR),
                            Cvt<float>::to_tc(du));
  const double pfloor = 1e-10 * (gt_pos(pR, pL) ? pL : pR);
  double p = Cvt<double>::to_tc(Cvt<float>::to_f64(S.p));
  if (!(S.conv && S.p > 1e-30f && S.p < 1e30f))
    p = exact_guess(G, rL, pL, cL, rR, pR, cR, du, pfloor);
  Star64 R;
  bool conv = false;
  for (int it = 0; it < Prec<double>::newton_max; ++it) {
    const double ip = rcpv(p);
    double fL, dfL, fR, dfR;
    const double xL = p * ipL, xR = p * ipR;
    side_f64(G, p, ip, rL, pL, xL, cL, fL, dfL, R.wL);
    side_f64(G, p, ip, rR, pR, xR, cR, fR, dfR, R.wR);
    // relative Newton step, then Halley's correction 1 / (1 + step H), H = p f''/(2 f')
    const double dS = dfL + dfR, idS = rcpv(dS);
    double x = -(fL + fR + du) * idS * ip;
    float xf = Cvt<float>::to_tc(x);
    const float tL = Cvt<float>::to_tc(dfL * idS), tR = 1.0f - tL;  // shares of f'
    const float kL = tL * curvature_f32(H, Cvt<float>::to_tc(xL));
    const float kR = tR * curvature_f32(H, Cvt<float>::to_tc(xR));
    float c = xf * 0.5f * (kL + kR);
    if (!(fabsf(c) < 0.05f)) c = 0.0f;
    x = fma(-x, Cvt<float>::to_f64(c), x);
    double pn = fma(p, x, p);
    if (!(pn > pfloor)) {  // held at the floor: the step that is taken, 0 once it rests there
      pn = pfloor;
      x = fma(pn, ip, -1.0);
      xf = Cvt<float>::to_tc(x);
    }
    R.p = pn;
    R.step = x;
    const double d = pn - p;
    // second order of f_R - f_L: p f'' d x / 2
    R.uj = fma(d, fma(dS * Cvt<float>::to_f64(0.5f * (kR - kL)), x, dfR - dfL), fR - fL);
    p = pn;
    if (fabsf(xf) < 2e-6f) { conv = true; break; }
  }
  if (!conv) err |= ERR_NEWTON;
  return R;
}

template <int NT>
__device__ __forceinline__ void exact_flux_f64(const Gas<double>& G, double rL, double uL,
                                               double pL, const double* vtL, double rR, double uR,
                                               double pR, const double* vtR, double* F,
                                               unsigned& err) {
  if (!(posv(rL) && posv(pL) && posv(rR) && posv(pR))) {
    err |= ERR_NONPHYS;
    for (int q = 0; q < 3 + NT; ++q) F[q] = 0.0;
    return;
  }
  const double ipL = rcpv(pL), ipR = rcpv(pR);
  const double cL = sqrt64(G.g * pL * rcpv(rL)), cR = sqrt64(G.g * pR * rcpv(rR));
  const double du = uR - uL;
  if (!gt_pos(G.two_gm1 * (cL + cR), du)) err |= ERR_VACUUM;
  const Star64 S = star_f64(G, rL, pL, ipL, cL, rR, pR, ipR, cR, du, err);
  const double p = S.p;
  const double us = 0.5 * ((uL + uR) + S.uj);
  // sample at x/t = 0, the right side of the contact mirrored onto the left
  const bool left = us >= 0.0;
  const double rK = left ? rL : rR, pK = left ? pL : pR, cK = left ? cL : cR;
  const double ipK = left ? ipL : ipR, uK = left ? uL : uR;
  const double w = left ? uK : -uK, ws = left ? us : -us;
  const double x = p * ipK;
  const bool shock = gt_pos(p, pK);
  bool unpert, fan = false;
  double q = 1.0;  // (p/pK)^z at p*
  if (shock) {
    // w against the shock's speed m: decided in FP32 where the two differ by 1e-5, some 25
    // times the rounding of both, and neither has left the FP32 range (m = inf fails too)
    const float wf = Cvt<float>::to_tc(w);
    const float m = Cvt<float>::to_tc(cK) * sqrtv(G.lo.shk1 * Cvt<float>::to_tc(x) + G.lo.z);
    unpert = wf >= m;
    if (!(m > 1e-30f && fabsf(wf - m) > 1e-5f * (fabsf(wf) + m)))
      unpert = w - cK * sqrt64(fma(G.shk1, x, G.z)) >= 0.0;
  } else {
    // from the last evaluation by the relative step since then; from 1 (p = pK) where
    // that evaluation was on the shock side, less than a step away from pK
    q = left ? S.wL : S.wR;
    const bool crossed = q == 0.0;
    const double d = crossed ? x - 1.0 : S.step;
    q = crossed ? 1.0 : q;
    q = fma(q, (G.z * d) * fma(0.5 * (G.z - 1.0), d, 1.0), q);
    unpert = w - cK >= 0.0;
    fan = !unpert && !(fma(-cK, q, ws) < 0.0);
  }
  // star density: rho_K (x + g6) / (g6 x + 1) behind a shock, rho_K x / q^2 in the fan's foot
  const double num = shock ? x + G.g6 : x;
  const double den = shock ? fma(G.g6, x, 1.0) : q * q;
  double rho = rK * (num * rcpv(den)), u = ws, pp = p;
  if (unpert) { rho = rK; u = w; pp = pK; }
  if (fan) {
    const double c = G.two_gp1 * fma(0.5 * G.gm1, w, cK);
    const double y = c / cK;
    u = c;
    rho = rK * pow(y, G.two_gm1);
    pp = pK * pow(y, G.inv_z);
  }
  if (!left) u = -u;
  double kin = u * u;
  double vt[NT > 0 ? NT : 1];
#pragma unroll
  for (int a = 0; a < NT; ++a) {
    vt[a] = left ? vtL[a] : vtR[a];
    kin = fma(vt[a], vt[a], kin);
  }
  const double mu = rho * u;
  F[0] = mu;
  F[1] = fma(mu, u, pp);
#pragma unroll
  for (int a = 0; a < NT; ++a) F[2 + a] = mu * vt[a];
  F[2 + NT] = u * fma(0.5 * rho, kin, pp * (G.inv_gm1 + 1.0));
}

template <class T, int NT>
__device__ __forceinline__ void exact_flux(const Gas<T>& G, T rL, T uL, T pL, const T* vtL, T rR,
                                           T uR, T pR, const T* vtR, T* F, unsigned& err) {
  if constexpr (std::is_same<T, float>::value)
    exact_flux_f32<NT>(G, rL, uL, pL, vtL, rR, uR, pR, vtR, F, err);
  else
    exact_flux_f64<NT>(G, rL, uL, pL, vtL, rR, uR, pR, vtR, F, err);
}

// ----------------------------------------------------------------------------
// HLLD solver with NT transverse components (1: planar MHD, 2: 3D MHD): per side
// (rho, u, p) with u normal, v[] and bt[] the transverse velocity and field; bn the
// common normal field.  Output in the face frame: F[0] mass, F[1] normal momentum,
// F[2 ..] transverse momenta, F[2+NT] energy, F[3+NT ..] transverse field fluxes (the
// normal-field flux is zero).
//
// The flux is that of one state, evaluated once: the outer state of side K, or its
// single- or double-star state with the normal velocity SM and the total pressure of
// the star region (K the side of the contact that x/t = 0 lies on).  By the solver's
// own jump relations this equals F_K + S_K (U*_K - U_K) + S*_K (U**_K - U*_K), without
// forming the four vectors of both sides.  On a degenerate side, where the transverse
// star state is set equal to the outer one, the field flux of that sum differs by
// bt (u_K - SM), which is added.  Bound by the FP64 pipe (about 165 operations, 400 with
// the four vectors and IEEE divisions: 2D MHD 512^2 step 2.83 -> 1.45 ms) and in FP32 by
// issue (about 190 instructions, 358 before).
// ----------------------------------------------------------------------------
template <class T, int NT>
__device__ __forceinline__ void hlld_core(const Gas<T>& G, T rL, T uL, const T* vL, T pL,
                                          const T* btL, T rR, T uR, const T* vR, T pR,
                                          const T* btR, T bn, T* F, unsigned& err) {
  if (!(posv(rL) && posv(pL) && posv(rR) && posv(pR))) {
    err |= ERR_NONPHYS;
    for (int q = 0; q < 3 + 2 * NT; ++q) F[q] = T(0);
    return;
  }
  const T bn2 = bn * bn;
  T b2L = bn2, b2R = bn2;
#pragma unroll
  for (int a = 0; a < NT; ++a) {
    b2L += btL[a] * btL[a];
    b2R += btR[a] * btR[a];
  }
  const T pTL = pL + T(0.5) * b2L, pTR = pR + T(0.5) * b2R;
  const T c2L = fast_speed2(G, rcpv(rL), pL, b2L, bn), c2R = fast_speed2(G, rcpv(rR), pR, b2R, bn);
  const T cmax = sqrtv(gt_pos(c2L, c2R) ? c2L : c2R);
  const bool lt = uL < uR;
  const T SL = (lt ? uL : uR) - cmax, SR = (lt ? uR : uL) + cmax;
  const T dL = SL - uL, dR = SR - uR;
  const T mL = rL * dL, mR = rR * dR;  // mass fluxes through the fast waves
  // contact speed and total pressure of the star region, as corrections of the left
  // state (small jumps lose nothing to cancellation): jK = SM - uK
  const T du = uR - uL;
  const T jL = (mR * du - (pTR - pTL)) * rcpv(mR - mL), jR = jL - du;
  const T SM = uL + jL;
  const T pTs = pTL + mL * jL;
  // single-star transverse states of both sides
  T vsL[NT], bsL[NT], vsR[NT], bsR[NT];
  const T eL = dL - jL, eR = dR - jR;  // S - SM
  const T iL = rcpv(eL), iR = rcpv(eR);
  const T rsL = mL * iL, rsR = mR * iR;
  bool degL, degR;
  {
    const T dd = mL * eL - bn2;
    degL = fabs(dd) < Prec<T>::hlld_degenerate * (mL * dL + bn2);
    const T k = jL * rcpv(dd);
    const T tv = bn * k, tb = mL * k;  // tb + 1 = (m d - bn^2) / dd
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      vsL[a] = degL ? vL[a] : vL[a] - btL[a] * tv;
      bsL[a] = degL ? btL[a] : btL[a] + btL[a] * tb;
    }
  }
  {
    const T dd = mR * eR - bn2;
    degR = fabs(dd) < Prec<T>::hlld_degenerate * (mR * dR + bn2);
    const T k = jR * rcpv(dd);
    const T tv = bn * k, tb = mR * k;
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      vsR[a] = degR ? vR[a] : vR[a] - btR[a] * tv;
      bsR[a] = degR ? btR[a] : btR[a] + btR[a] * tb;
    }
  }
  const T yL = rsqrtp(rsL), yR = rsqrtp(rsR);
  const T sqL = rsL * yL, sqR = rsR * yR;  // sqrt(rho*)
  const T abn = fabs(bn);
  // the side and the region
  const bool left = !negv(SM);
  const bool outer = left ? !negv(SL) : negv(SR);
  const bool single = left ? !negv(SM - abn * yL) : !posv(SM + abn * yR);
  const T rK = left ? rL : rR, uK = left ? uL : uR, pTK = left ? pTL : pTR;
  const T pK = left ? pL : pR, b2K = left ? b2L : b2R;
  T vK[NT], bK[NT], v[NT], b[NT];
#pragma unroll
  for (int a = 0; a < NT; ++a) {
    vK[a] = left ? vL[a] : vR[a];
    bK[a] = left ? btL[a] : btR[a];
    v[a] = left ? vsL[a] : vsR[a];
    b[a] = left ? bsL[a] : bsR[a];
  }
  T v2 = uK * uK, vB = uK * bn;
#pragma unroll
  for (int a = 0; a < NT; ++a) {
    v2 += vK[a] * vK[a];
    vB += vK[a] * bK[a];
  }
  const T EK = pK * G.inv_gm1 + T(0.5) * (rK * v2 + b2K);
  T r, u, E, pT, extra[NT], vBf;
  if (outer) {
    r = rK; u = uK; E = EK; pT = pTK; vBf = vB;
#pragma unroll
    for (int a = 0; a < NT; ++a) { v[a] = vK[a]; b[a] = bK[a]; extra[a] = T(0); }
  } else {
    r = left ? rsL : rsR;
    u = SM;
    pT = pTs;
    T vBs = SM * bn;
#pragma unroll
    for (int a = 0; a < NT; ++a) vBs += v[a] * b[a];
    const T dK = left ? dL : dR, iK = left ? iL : iR, jK = left ? jL : jR;
    E = (dK * EK - pTK * uK + pTs * SM + bn * (vB - vBs)) * iK;
    const bool deg = left ? degL : degR;
#pragma unroll
    for (int a = 0; a < NT; ++a) extra[a] = deg ? -b[a] * jK : T(0);
    vBf = vBs;
    if (!single) {  // between the Alfven waves
      const T sg = bn > T(0) ? T(1) : (bn < T(0) ? T(-1) : T(0));
      const T inv = rcpv(sqL + sqR);
      T vBss = SM * bn;
#pragma unroll
      for (int a = 0; a < NT; ++a) {
        // v** - v*_L, and b** - b*_L = sqrt(rho*_L) sign(bn) (v** - v*_L)
        const T q = (sqR * (vsR[a] - vsL[a]) + (bsR[a] - bsL[a]) * sg) * inv;
        v[a] = vsL[a] + q;
        b[a] = bsL[a] + sqL * sg * q;
        vBss += v[a] * b[a];
      }
      E += (left ? -sqL : sqR) * (vBs - vBss) * sg;
      vBf = vBss;
    }
  }
  const T m = r * u;
  F[0] = m;
  F[1] = m * u + pT - bn2;
  F[2 + NT] = (E + pT) * u - bn * vBf;
#pragma unroll
  for (int a = 0; a < NT; ++a) {
    F[2 + a] = m * v[a] - bn * b[a];
    F[3 + NT + a] = b[a] * u - v[a] * bn + extra[a];
  }
}

// Planar MHD: F[0] mass, F[1] normal and F[2] transverse momentum, F[3] energy, F[4]
// transverse field.
template <class T>
__device__ __forceinline__ void hlld_flux(const Gas<T>& G, T rL, T uL, T vL, T pL, T btL, T rR,
                                          T uR, T vR, T pR, T btR, T bn, T* F, unsigned& err) {
  hlld_core<T, 1>(G, rL, uL, &vL, pL, &btL, rR, uR, &vR, pR, &btR, bn, F, err);
}

// 3D MHD: F[0] mass, F[1] normal, F[2], F[3] transverse momenta, F[4] energy, F[5],
// F[6] transverse field.
template <class T>
__device__ __forceinline__ void hlld_flux3(const Gas<T>& G, T rL, T uL, T vL, T wL, T pL, T bvL,
                                           T bwL, T rR, T uR, T vR, T wR, T pR, T bvR, T bwR,
                                           T bn, T* F, unsigned& err) {
  const T vl[2] = {vL, wL}, bl[2] = {bvL, bwL}, vr[2] = {vR, wR}, br[2] = {bvR, bwR};
  hlld_core<T, 2>(G, rL, uL, vl, pL, bl, rR, uR, vr, pR, br, bn, F, err);
}

// ----------------------------------------------------------------------------
// Min/max limiter coefficient of one primitive (Sec. 2.5):
//   alpha = min(1, min_faces psi_f), psi_f = (phimax - phi)/dphi_f (dphi_f > 0),
//   (phimin - phi)/dphi_f (dphi_f < 0), 1 (dphi_f = 0), dphi_f = grad phi . (f - s).
// On a Cartesian cell the faces along axis d have dphi = +-a_d with
// a_d = g_d h_d / 2, so min_faces psi = min(phimax - phi, phi - phimin) / max_d |a_d|
// (division is monotone, so this is the same floating-point value).
// ----------------------------------------------------------------------------
template <class T, int DIM>
__device__ __forceinline__ T limiter_alpha(T phi, T phimax, T phimin, const T* grad,
                                           const T* half_h) {
  T amax = fabs(grad[0] * half_h[0]);
#pragma unroll
  for (int d = 1; d < DIM; ++d) {
    const T a = fabs(grad[d] * half_h[d]);
    amax = gt_pos(a, amax) ? a : amax;
  }
  const T up = phimax - phi, dn = phi - phimin;  // both >= 0
  const T m = gt_pos(dn, up) ? up : dn;
  // psi = m / amax < 1
  return gt_pos(amax, m) && !gt_pos(T(Tiny<T>::v), amax) ? m * rcpv(amax) : T(1);
}

}  // namespace dgk
