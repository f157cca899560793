// dg_vjp.cuh -- reverse-mode (vector-Jacobian) products of the 2D Euler fluxes, for
// the adjoint of the DG step: given the adjoint mu of a flux, the adjoints of the
// states it was computed from, in one reverse sweep through the flux's own
// arithmetic (instead of forward-mode dual numbers, one pass per input direction).
//
// Exact Riemann flux (Sec. 2.3; Toro's solver sampled at x/t = 0), face frame,
// primitive states (rho, u, v, p) with u normal, v transverse:
//   p* solves Phi(p) = f_L(p; rho_L, p_L) + f_R(p; rho_R, p_R) + u_R - u_L = 0,
//   u* = (u_L + u_R)/2 + (f_R(p*) - f_L(p*))/2,
//   the sampled state is side K's, its shock- or rarefaction-star state, or the
//   transonic fan, and F = (rho u, rho u^2 + p, rho u v, u (E + p)).
// The reverse sweep goes F -> sampled state -> (p*, u*, side K) -> inputs; p* by the
// implicit-function rule: an adjoint a of p* contributes -a/(f_L' + f_R') dPhi/dx.
// The derivative is that of the branch the sample lies in (the adjoint of the step
// differentiates its active branch, as for the limiter).
#pragma once

#include "dg_physics.cuh"

namespace dgk {

// x^z - 1 and, in w, x^z.
__device__ __forceinline__ float pow_m1v(float x, float z, float& w) {
  w = ex2v(z * lg2v(x));
  return w - 1.0f;
}
__device__ __forceinline__ double pow_m1v(double x, double z, double& w) { return pow_m1(x, z, w); }

// q = (Ai pb)^(-1/2) and 1/pb: in FP32 by two roots, as in star_f32.
__device__ __forceinline__ float shock_q(float pb, float Ai, float& ipb) {
  const float y = rsqrtp(pb);
  ipb = y * y;
  return y * rsqrtp(Ai);
}
__device__ __forceinline__ double shock_q(double pb, double Ai, double& ipb) {
  const double q = rsqrtp(pb * Ai);
  ipb = q * q * Ai;
  return q;
}

// Pressure function of side K (Toro's f_K) and its partial derivatives with
// respect to p, rho_K and p_K (c_K = sqrt(g p_K / rho_K) taken into account); i* are
// reciprocals, qz = (p/p_K)^z on a rarefaction side.
template <class T>
__device__ __forceinline__ void pressure_fn_partials(const Gas<T>& G, T p, T ip, T rK, T irK, T pK,
                                                     T ipK, T cK, T& f, T& df, T& dr, T& dpk,
                                                     T& qz) {
  if (gt_pos(p, pK)) {  // shock: f = (p - pK) q, q = (Ai (p + B))^(-1/2), 1/Ai = 2/((g+1) rho_K)
    const T Ai = T(0.5) * G.gp1 * rK;
    T ipb;
    const T q = shock_q(p + G.g6 * pK, Ai, ipb);
    f = (p - pK) * q;
    df = q - T(0.5) * f * ipb;
    dpk = -q - T(0.5) * f * G.g6 * ipb;
    qz = T(1);
  } else {  // rarefaction: f = 2 cK/(g-1) ((p/pK)^z - 1)
    const T m1 = pow_m1v(p * ipK, G.z, qz);
    const T C = G.two_gm1 * cK;
    f = C * m1;
    df = cK * G.inv_g * (qz * ip);
    dpk = C * (T(0.5) * m1 - G.z * qz) * ipK;
  }
  dr = -T(0.5) * f * irK;
}

// p* of the exact solver: FP32 by its Newton iteration, FP64 by the FP32 guess and
// Halley steps (dg_physics.cuh).
__device__ __forceinline__ float vjp_pstar(const Gas<float>& G, float rL, float pL, float ipL,
                                           float cL, float rR, float pR, float ipR, float cR,
                                           float du, unsigned& err) {
  const Star32 S = star_f32(G, rL, pL, ipL, cL, rR, pR, ipR, cR, du);
  if (!S.conv) err |= ERR_NEWTON;
  return S.p;
}
__device__ __forceinline__ double vjp_pstar(const Gas<double>& G, double rL, double pL, double ipL,
                                            double cL, double rR, double pR, double ipR, double cR,
                                            double du, unsigned& err) {
  return star_f64(G, rL, pL, ipL, cL, rR, pR, ipR, cR, du, err).p;
}

// Adjoint of the exact-solver flux: mu (mass, normal momentum, transverse momentum,
// energy) -> aL, aR, the adjoints of (rho, u, v, p) of the two sides.  Divisions are
// products with a few reciprocals and (p/p_K)^z is formed once per side (the star
// density behind a rarefaction is rho_K (p/p_K) / qz^2).
template <class T>
__device__ void exact_flux_vjp(const Gas<T>& G, T rL, T uL, T vL, T pL, T rR, T uR, T vR, T pR,
                               const T* mu, T* aL, T* aR, unsigned& err) {
#pragma unroll
  for (int i = 0; i < 4; ++i) { aL[i] = T(0); aR[i] = T(0); }
  if (!(posv(rL) && posv(pL) && posv(rR) && posv(pR))) {
    err |= ERR_NONPHYS;
    return;
  }
  const T irL = rcpv(rL), irR = rcpv(rR), ipL = rcpv(pL), ipR = rcpv(pR);
  const T cL = sqrts(G.g * pL * irL), cR = sqrts(G.g * pR * irR);
  const T du = uR - uL;
  if (G.two_gm1 * (cL + cR) <= du) err |= ERR_VACUUM;
  const T p = vjp_pstar(G, rL, pL, ipL, cL, rR, pR, ipR, cR, du, err);
  const T ip = rcpv(p);
  T fL, dfL, fLr, fLp, qL, fR, dfR, fRr, fRp, qR;
  pressure_fn_partials(G, p, ip, rL, irL, pL, ipL, cL, fL, dfL, fLr, fLp, qL);
  pressure_fn_partials(G, p, ip, rR, irR, pR, ipR, cR, fR, dfR, fRr, fRp, qR);
  const T us = T(0.5) * (uL + uR) + T(0.5) * (fR - fL);
  // sample on the side of the contact, the right side mirrored onto the left
  const bool left = T(0) <= us;
  const T sg = left ? T(1) : T(-1);
  const T rK = left ? rL : rR, uK = left ? uL : uR, vK = left ? vL : vR;
  const T pK = left ? pL : pR, cK = left ? cL : cR, qz = left ? qL : qR;
  const T irK = left ? irL : irR, ipK = left ? ipL : ipR;
  const T w = sg * uK, ws = sg * us, pr = p * ipK;
  const bool shock = gt_pos(p, pK);
  bool unpert, fan = false;
  if (shock) {
    unpert = T(0) <= w - cK * sqrtv(G.shk1 * pr + G.z);
  } else {
    unpert = T(0) <= w - cK;
    fan = !unpert && !(T(0) > ws - cK * qz);
  }
  // star density factor rho*/rho_K and its derivative with respect to p/p_K
  const T iden = rcpv(shock ? G.g6 * pr + T(1) : qz * qz);
  const T fac = (shock ? pr + G.g6 : pr) * iden;
  const T dfac = shock ? (T(1) - G.g6 * G.g6) * iden * iden : G.inv_g * iden;
  T rho, uf, pp, c = T(0), xa = T(0), xb = T(0);
  if (unpert) {
    rho = rK; uf = w; pp = pK;
  } else if (!fan) {
    rho = rK * fac; uf = ws; pp = p;
  } else {
    c = G.two_gp1 * (cK + T(0.5) * G.gm1 * w);
    xa = rpow(c / cK, G.two_gm1);
    xb = rpow(c / cK, G.inv_z);
    uf = c;
    rho = rK * xa;
    pp = pK * xb;
  }
  const T u = sg * uf;
  const T k2 = T(0.5) * (u * u + vK * vK);
  const T E = pp * G.inv_gm1 + rho * k2;
  // F -> sampled state
  const T a_rho = u * (mu[0] + mu[1] * u + mu[2] * vK + mu[3] * k2);
  const T a_u = rho * (mu[0] + T(2) * mu[1] * u + mu[2] * vK + mu[3] * (u * u)) + mu[3] * (E + pp);
  const T a_p = mu[1] + mu[3] * u * (G.inv_gm1 + T(1));
  const T a_v = rho * u * (mu[2] + mu[3] * vK);
  const T a_uf = sg * a_u;
  // sampled state -> (rho_K, u_K, p_K, c_K), p*, u*
  T a_rK = T(0), a_uK = T(0), a_pK = T(0), a_ps = T(0), a_us = T(0);
  if (unpert) {
    a_rK = a_rho; a_uK = sg * a_uf; a_pK = a_p;
  } else if (!fan) {
    const T t = a_rho * rK * dfac * ipK;
    a_rK = a_rho * fac;
    a_ps = a_p + t;
    a_pK = -t * pr;
    a_us = sg * a_uf;
  } else {
    const T a_c = a_uf + a_rho * rK * G.two_gm1 * xa / c + a_p * pK * G.inv_z * xb / c;
    const T a_cK = -a_rho * rK * G.two_gm1 * xa / cK - a_p * pK * G.inv_z * xb / cK + a_c * G.two_gp1;
    // c_K = sqrt(g p_K / rho_K)
    a_rK = a_rho * xa - T(0.5) * a_cK * cK * irK;
    a_pK = a_p * xb + T(0.5) * a_cK * cK * ipK;
    a_uK = sg * a_c * T(0.5) * G.gm1 * G.two_gp1;
  }
  // u* = (u_L + u_R)/2 + (f_R - f_L)/2, and p* by Phi(p*; x) = 0
  const T hu = T(0.5) * a_us;
  a_ps += hu * (dfR - dfL);
  const T lam = a_ps * rcpv(dfL + dfR);
  const T wl = -(hu + lam), wr = hu - lam;
  aL[0] = wl * fLr;
  aL[1] = hu + lam;
  aL[3] = wl * fLp;
  aR[0] = wr * fRr;
  aR[1] = hu - lam;
  aR[3] = wr * fRp;
  aL[0] += left ? a_rK : T(0);
  aL[1] += left ? a_uK : T(0);
  aL[2] = left ? a_v : T(0);
  aL[3] += left ? a_pK : T(0);
  aR[0] += left ? T(0) : a_rK;
  aR[1] += left ? T(0) : a_uK;
  aR[2] = left ? T(0) : a_v;
  aR[3] += left ? T(0) : a_pK;
}

// Reverse of the centroid primitives of a 2D Euler state: adjoints (a_rho, a_vx,
// a_vy, a_p) of (rho, vx, vy, p) -> adjoints of the conserved (rho, mx, my, E).
template <class T>
__device__ __forceinline__ void prims2d_vjp(const Gas<T>& G, const T* c, const T* aW, T* ac) {
  const T inv = rcpv(c[0]);
  const T vx = c[1] * inv, vy = c[2] * inv;
  ac[3] = G.gm1 * aW[3];
  ac[1] = aW[1] * inv - G.gm1 * vx * aW[3];
  ac[2] = aW[2] * inv - G.gm1 * vy * aW[3];
  ac[0] = aW[0] - (aW[1] * vx + aW[2] * vy) * inv + T(0.5) * G.gm1 * (vx * vx + vy * vy) * aW[3];
}

// Adjoint of the exact flux through a face along `dir` between conserved states
// cl, cr: mu in lab-frame flux order -> the adjoints of cl and cr.
template <class T>
__device__ __forceinline__ void face_flux2d_vjp(const Gas<T>& G, int dir, const T* cl, const T* cr,
                                                const T* mu, T* acl, T* acr, unsigned& err) {
  const bool xd = dir == 0;
  const T il = rcpv(cl[0]), ir = rcpv(cr[0]);
  const T vxl = cl[1] * il, vyl = cl[2] * il, vxr = cr[1] * ir, vyr = cr[2] * ir;
  const T pl = G.gm1 * (cl[3] - T(0.5) * (cl[1] * vxl + cl[2] * vyl));
  const T pr = G.gm1 * (cr[3] - T(0.5) * (cr[1] * vxr + cr[2] * vyr));
  const T muf[4] = {mu[0], xd ? mu[1] : mu[2], xd ? mu[2] : mu[1], mu[3]};
  T aL[4], aR[4];
  exact_flux_vjp<T>(G, cl[0], xd ? vxl : vyl, xd ? vyl : vxl, pl, cr[0], xd ? vxr : vyr,
                    xd ? vyr : vxr, pr, muf, aL, aR, err);
  // face frame (rho, u_n, u_t, p) -> lab (rho, vx, vy, p)
  const T wl[4] = {aL[0], xd ? aL[1] : aL[2], xd ? aL[2] : aL[1], aL[3]};
  const T wr[4] = {aR[0], xd ? aR[1] : aR[2], xd ? aR[2] : aR[1], aR[3]};
  prims2d_vjp<T>(G, cl, wl, acl);
  prims2d_vjp<T>(G, cr, wr, acr);
}

// Adjoint of the physical fluxes (Fx, Fy) of a 2D Euler state c at a volume
// Gauss point: yx, yy the adjoints of Fx, Fy -> a, the adjoint of c.
template <class T>
__device__ __forceinline__ void phys_flux2d_vjp(const Gas<T>& G, const T* c, const T* yx,
                                                const T* yy, T* a) {
  const T inv = rcpv(c[0]);
  const T u = c[1] * inv, v = c[2] * inv;
  const T p = G.gm1 * (c[3] - T(0.5) * (c[1] * u + c[2] * v));
  const T e = c[3] + p;
  // Fx = (mx, mx u + p, my u, e u), Fy = (my, mx v, my v + p, e v), e = E + p
  T a1 = yx[0] + yx[1] * u + yy[1] * v;
  T a2 = yy[0] + yx[2] * u + yy[2] * v;
  T au = yx[1] * c[1] + yx[2] * c[2] + yx[3] * e;
  T av = yy[1] * c[1] + yy[2] * c[2] + yy[3] * e;
  const T ae = yx[3] * u + yy[3] * v;
  const T ap = yx[1] + yy[2] + ae;
  T a3 = ae + G.gm1 * ap;
  // p = (g - 1)(E - (mx u + my v)/2)
  a1 -= T(0.5) * G.gm1 * u * ap;
  a2 -= T(0.5) * G.gm1 * v * ap;
  au -= T(0.5) * G.gm1 * c[1] * ap;
  av -= T(0.5) * G.gm1 * c[2] * ap;
  // u = mx / rho, v = my / rho
  a[1] = a1 + au * inv;
  a[2] = a2 + av * inv;
  a[0] = -(au * u + av * v) * inv;
  a[3] = a3;
}

}  // namespace dgk
