// Pointwise device functions shared by the line kernels: Euler fluxes (Sec. 2.1), the
// product rules of adiabatic wall patches (Remark adiabatic), the SSPRK stage combination
// (Sec. 4.1) and the filter's energy rebuild (Sec. 4.3.1).
#pragma once
#include <cuda_runtime.h>

#include "fc_internal.h"
#include "fc_line.cuh"

namespace fcx {

__device__ __forceinline__ void flux_xy(double r, double mx, double my, double E, double gam, double* fx, double* fy) {
  const double ir = 1.0 / r;
  const double u = mx * ir, v = my * ir;
  const double p = (gam - 1.0) * (E - 0.5 * (mx * u + my * v));
  fx[0] = mx;
  fx[1] = fma(mx, u, p);
  fx[2] = mx * v;
  fx[3] = u * (E + p);
  fy[0] = my;
  fy[1] = my * u;
  fy[2] = fma(my, v, p);
  fy[3] = v * (E + p);
}

__device__ __forceinline__ void flux_x(double r, double mx, double my, double E, double gam, double* f) {
  const double ir = 1.0 / r;
  const double u = mx * ir, v = my * ir;
  const double p = (gam - 1.0) * (E - 0.5 * (mx * u + my * v));
  f[0] = mx;
  f[1] = fma(mx, u, p);
  f[2] = mx * v;
  f[3] = u * (E + p);
}
__device__ __forceinline__ void flux_y(double r, double mx, double my, double E, double gam, double* f) {
  const double ir = 1.0 / r;
  const double u = mx * ir, v = my * ir;
  const double p = (gam - 1.0) * (E - 0.5 * (mx * u + my * v));
  f[0] = my;
  f[1] = my * u;
  f[2] = fma(my, v, p);
  f[3] = v * (E + p);
}

// ---- product-rule form on adiabatic wall patches (Remark adiabatic)
// Derivatives along one direction of e = (rho, rho u, rho v, E) and of p from those of
// Q = (rho, rho u, rho v, theta): dp = theta drho + rho dtheta (eq. p_T),
// dE = dp / (gamma - 1) + u d(rho u) + v d(rho v) - (u^2 + v^2) / 2 drho (eq. perfect_gas_T).
__device__ __forceinline__ void product_rule(const double* Q, const double* DQ, double gm1, double* De, double& Dp) {
  const double ir = 1.0 / Q[0];
  const double u = Q[1] * ir, v = Q[2] * ir;
  Dp = fma(Q[3], DQ[0], Q[0] * DQ[3]);
  De[0] = DQ[0];
  De[1] = DQ[1];
  De[2] = DQ[2];
  De[3] = fma(-0.5 * fma(u, u, v * v), DQ[0], fma(u, DQ[1], fma(v, DQ[2], Dp / gm1)));
}

// div f(e) (eq. euler 2d equation) by the sum and product rules from the x and y derivatives
// of e (ex, ey) and p (px, py); theta = p / rho; du = (d(rho u) - u drho) / rho
__device__ __forceinline__ void conv_div_product(const double* e, double th, const double* ex, double px,
                                                 const double* ey, double py, double* out) {
  const double ir = 1.0 / e[0];
  const double u = e[1] * ir, v = e[2] * ir, p = e[0] * th;
  const double ux = (ex[1] - u * ex[0]) * ir, vy = (ey[2] - v * ey[0]) * ir;
  out[0] = ex[1] + ey[2];
  out[1] = fma(u, ex[1], fma(e[1], ux, px)) + fma(v, ey[1], e[1] * vy);
  out[2] = fma(u, ex[2], e[2] * ux) + fma(v, ey[2], fma(e[2], vy, py));
  out[3] = fma(e[3] + p, ux + vy, fma(u, ex[3] + px, v * (ey[3] + py)));
}

// a / b from ib = 1 / b: the quotient estimate and one correction with its exact remainder
// (Markstein's scheme: a correctly rounded ib gives a correctly rounded quotient up to rare
// cases within an ulp), three FP64 operations where a division takes about six
__device__ __forceinline__ double div_by(double a, double b, double ib) {
  const double q = a * ib;
  return fma(fma(-q, b, a), ib, q);
}
// theta = p / rho (eq. p_T)
__device__ __forceinline__ double theta_of(double r, double mx, double my, double E, double gam) {
  const double ir = 1.0 / r;
  const double p = (gam - 1.0) * (E - 0.5 * (mx * (mx * ir) + my * (my * ir)));
  return div_by(p, r, ir);
}

// Runge-Kutta stage combination of one component (q: flat index of the component's point)
// from its loaded operands; aux is 0 without Uaux, u0 is read only where c0 != 0
__device__ __forceinline__ void stage_put(const StageCoef& sc, double dt, long long q, double L, double cur, double u0,
                                          double aux) {
  if (sc.rhs_only) {
    sc.out[q] = L;
    return;
  }
  double v = sc.c1 * cur;
  if (sc.c0 != 0.0) v = fma(sc.c0, u0, v);
  if (sc.c2 != 0.0) v = fma(sc.c2, aux, v);
  v = fma(sc.cb * dt, L, v);
  if (sc.out2) sc.out2[q] = fma(sc.db * dt, L, fma(sc.d2, aux, sc.d1 * cur));
  sc.out[q] = v;
}
__device__ __forceinline__ void stage_write1(const StageCoef& sc, double dt, long long q, double L) {
  if (sc.rhs_only)
    stage_put(sc, dt, q, L, 0.0, 0.0, 0.0);
  else
    stage_put(sc, dt, q, L, sc.Ucur[q], sc.c0 != 0.0 ? sc.U0[q] : 0.0, sc.Uaux ? sc.Uaux[q] : 0.0);
}
__device__ __forceinline__ void stage_write(const StageCoef& sc, long long p, long long cs, const double* L4) {
  const double dt = sc.rhs_only ? 0.0 : *sc.dt;
#pragma unroll
  for (int c = 0; c < 4; ++c) stage_write1(sc, dt, p + c * cs, L4[c]);
}

__device__ __forceinline__ double energy_of(double r, double mx, double my, double th, double gam) {
  const double g1 = gam - 1.0;
  return div_by(r * th, g1, 1.0 / g1) + div_by(0.5 * (mx * mx + my * my), r, 1.0 / r);
}

// A^T eta for the x (dir 0) or y (dir 1) flux Jacobian at state e (eq. euler 2d equation)
__device__ __forceinline__ void fluxT(int dir, double r, double mx, double my, double E, double gam, const double* eta,
                                      double* out) {
  const double ir = 1.0 / r;
  const double u = mx * ir, v = my * ir;
  const double g1 = gam - 1.0;
  const double q2 = u * u + v * v;
  const double p = g1 * (E - 0.5 * r * q2);
  const double H = (E + p) * ir;
  const double pr = 0.5 * g1 * q2, pm = -g1 * u, pn = -g1 * v, pE = g1;
  if (dir == 0) {
    // rows c = 0..3 of A_x, columns j: out_j = sum_c A[c][j] eta_c
    out[0] = (-u * u + pr) * eta[1] + (-u * v) * eta[2] + (-u * H + u * pr) * eta[3];
    out[1] = eta[0] + (2.0 * u + pm) * eta[1] + v * eta[2] + (H + u * pm) * eta[3];
    out[2] = pn * eta[1] + u * eta[2] + u * pn * eta[3];
    out[3] = pE * eta[1] + u * (1.0 + pE) * eta[3];
  } else {
    out[0] = (-u * v) * eta[1] + (-v * v + pr) * eta[2] + (-v * H + v * pr) * eta[3];
    out[1] = v * eta[1] + pm * eta[2] + v * pm * eta[3];
    out[2] = eta[0] + u * eta[1] + (2.0 * v + pn) * eta[2] + (H + v * pn) * eta[3];
    out[3] = pE * eta[2] + v * (1.0 + pE) * eta[3];
  }
}

// Jacobian transposes of the filter's pointwise maps: of E rebuilt from the filtered
// (rho, rho u, rho v, theta) at the filtered state ef, and of theta(e)
__device__ __forceinline__ void rebuild_T(const double* lam, const double* ef, double gam, double* o) {
  const double r = ef[0], m = ef[1], nn = ef[2];
  const double th = theta_of(r, m, nn, ef[3], gam);
  const double g1 = gam - 1.0, lE = lam[3], ir = 1.0 / r;
  o[0] = lam[0] + lE * (th / g1 - 0.5 * (m * m + nn * nn) * ir * ir);
  o[1] = lam[1] + lE * m * ir;
  o[2] = lam[2] + lE * nn * ir;
  o[3] = lE * r / g1;
}
__device__ __forceinline__ void rebuild_T(const double* __restrict__ lam, const double* __restrict__ ef, long long p,
                                          long long cs, double gam, double* o) {
  const double l[4] = {lam[p], lam[p + cs], lam[p + 2 * cs], lam[p + 3 * cs]};
  const double f[4] = {ef[p], ef[p + cs], ef[p + 2 * cs], ef[p + 3 * cs]};
  rebuild_T(l, f, gam, o);
}
__device__ __forceinline__ void theta_T(const double* q, const double* e, double gam, double* o) {
  const double r = e[0], m = e[1], nn = e[2], E = e[3];
  const double g1 = gam - 1.0, lt = q[3], ir = 1.0 / r, ir2 = ir * ir;
  o[0] = q[0] + lt * g1 * (-E * ir2 + (m * m + nn * nn) * ir2 * ir);
  o[1] = q[1] + lt * (-g1 * m * ir2);
  o[2] = q[2] + lt * (-g1 * nn * ir2);
  o[3] = lt * g1 * ir;
}
__device__ __forceinline__ void theta_T(const double* q, const double* __restrict__ e, long long p, long long cs,
                                        double gam, double* o) {
  const double f[4] = {e[p], e[p + cs], e[p + 2 * cs], e[p + 3 * cs]};
  theta_T(q, f, gam, o);
}

// (dQ/du)^T a for Q = (rho, rho u, rho v, theta), theta = (gamma - 1) (E / rho - |rho u|^2 / (2 rho^2))
__device__ __forceinline__ void thetaT_add(const double* u, double gam, const double* a, double* out) {
  const double ir = 1.0 / u[0], g1 = gam - 1.0;
  const double m2 = fma(u[1], u[1], u[2] * u[2]);
  out[0] += a[0] + a[3] * g1 * ir * ir * (m2 * ir - u[3]);
  out[1] += a[1] - a[3] * g1 * u[1] * ir * ir;
  out[2] += a[2] - a[3] * g1 * u[2] * ir * ir;
  out[3] += a[3] * g1 * ir;
}

}  // namespace fcx
