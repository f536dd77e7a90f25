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

// theta = p / rho (eq. p_T)
__device__ __forceinline__ double theta_of(double r, double mx, double my, double E, double gam) {
  const Prim q = primitives(r, mx, my, E, gam);
  return q.p / r;
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
  return r * th / (gam - 1.0) + 0.5 * (mx * mx + my * my) / r;
}

}  // namespace fcx
