// Contraction kernels of the discrete adjoint: curvilinear lines (fc_mma.cuh).
#include "fc_mma.cuh"

namespace fcx {

namespace {

// ---- curvilinear patches (slots: 0 = S1x then eta_x, 1 = S1y then eta_y, 2 = partial, 3 = g1;
// fc_kernels.cu has the same passes on the FFT engine). Pointers to G and Jm carry the offset
// from a point's state index to its scratch index.
struct LoadWeighted {  // w psi, w = a metric, 0 on PT_NODIFF points; or a slot of G
  const double* f;
  const double* w;  // null: the slot as it is
  const uint32_t* __restrict__ info;
  long long st;
  __device__ __forceinline__ void raw(long long q, double* v) const {
    const double a = w ? ((info[q] & PT_NODIFF) ? 0.0 : w[q]) : 1.0;
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[q + c * st];
    if (w)
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = a * v[c];
  }
  __device__ __forceinline__ void form(long long, double*) const {}
};
struct LoadQ {  // (rho, rho u, rho v, theta)
  const double* __restrict__ u;
  long long cs;
  double gamma;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = u[q + c * cs];
  }
  __device__ __forceinline__ void form(long long, double* v) const { v[3] = theta_of(v[0], v[1], v[2], v[3], gamma); }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_adj_gen_A(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ Jm,
                                             const double* __restrict__ u, const double* __restrict__ psi, double* G) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const long long off = sh.J[0].gbase - sh.J[0].base, Pg = T.Pg;
#pragma unroll 1
  for (int w = 0; w < 2; ++w)
    mm_round<Cfg, false, false, true, true>(T, p, sh, dyn, LoadWeighted{psi, Jm + off + w * Pg, T.info, T.P},
                                              PutField4{G + off + 4 * w * Pg, Pg});
  if (T.patches[sh.J[0].patch].pform)  // product-rule wall form: D_1 Q at the stage state
    mm_round<Cfg, false, false, true, false>(T, p, sh, dyn, LoadQ{u, T.P, T.gamma},
                                               PutField4{G + off + 12 * Pg, Pg});
}

// pass B (other patches than the product-rule wall form's): eta, then the pointwise part with
// g2 = mu (J2x eta_x + J2y eta_y) into slot 0 for the last round
struct PutEta {
  struct Op {
    double a[4], b[4], u[4], j[4], m;
  };
  const double* __restrict__ Jm;
  const double* __restrict__ u;
  const double* __restrict__ mu;
  double* G;
  long long cs, Pg;
  double gamma;
  int rd;
  __device__ __forceinline__ Op pre(long long q) const {
    Op o;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      o.a[c] = G[(4 * rd + c) * Pg + q];
      o.b[c] = rd == 1 ? G[c * Pg + q] : 0.0;
      o.u[c] = rd == 1 ? u[q + c * cs] : 1.0;
      o.j[c] = rd == 1 ? Jm[q + c * Pg] : 0.0;
    }
    o.m = rd == 1 ? mu[q] : 0.0;
    return o;
  }
  __device__ __forceinline__ void put(long long q, const Op& o, const double* v) const {
    if (rd == 2) {
#pragma unroll
      for (int c = 0; c < 4; ++c) G[(8 + c) * Pg + q] = o.a[c] - v[c];
      return;
    }
    double e[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      e[c] = -(o.a[c] + v[c]);
      G[(4 * rd + c) * Pg + q] = e[c];
    }
    if (rd == 1) {
      double ax[4], ay[4];
      fluxT(0, o.u[0], o.u[1], o.u[2], o.u[3], gamma, o.b, ax);
      fluxT(1, o.u[0], o.u[1], o.u[2], o.u[3], gamma, e, ay);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        G[(8 + c) * Pg + q] = ax[c] + ay[c];
        G[(12 + c) * Pg + q] = o.m * fma(o.j[0], o.b[c], o.j[1] * e[c]);
        G[c * Pg + q] = o.m * fma(o.j[2], o.b[c], o.j[3] * e[c]);
      }
    }
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_adj_gen_B(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ Jm,
                                             const double* __restrict__ u, const double* __restrict__ mu,
                                             const double* __restrict__ psi, double* G) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  if (T.patches[sh.J[0].patch].pform) return;
  const MmPlan p = T.mm[sh.J[0].plan];
  const long long off = sh.J[0].gbase - sh.J[0].base, Pg = T.Pg;
#pragma unroll 1
  for (int rd = 0; rd < 3; ++rd)
    mm_round<Cfg, true, false, true, true>(
        T, p, sh, dyn,
        LoadWeighted{rd == 2 ? G + off : psi, rd == 2 ? nullptr : Jm + off + (2 + rd) * Pg, T.info, rd == 2 ? Pg : T.P},
        PutEta{Jm + off, u, mu, G + off, T.P, Pg, T.gamma, rd});
}

// pass C: acc += dt (partial - D_1^T(g1)); product-rule wall form: dt (partial - (dQ/du)^T D_1^T(g1))
struct PutAcc {
  struct Op {
    double a[4], p[4], u[4];
  };
  const double* __restrict__ u;
  const double* __restrict__ G;
  double* acc;
  long long cs, Pg;
  double gamma, dt;
  bool pf;
  __device__ __forceinline__ Op pre(long long q) const {
    Op o;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      o.a[c] = acc[q + c * cs];
      o.p[c] = G[(8 + c) * Pg + q];
      o.u[c] = pf ? u[q + c * cs] : 1.0;
    }
    return o;
  }
  __device__ __forceinline__ void put(long long q, const Op& o, const double* v) const {
    double x[4] = {v[0], v[1], v[2], v[3]};
    if (pf) {
      double y[4] = {0.0, 0.0, 0.0, 0.0};
      thetaT_add(o.u, gamma, x, y);
#pragma unroll
      for (int c = 0; c < 4; ++c) x[c] = y[c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[q + c * cs] = fma(dt, o.p[c] - x[c], o.a[c]);
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_adj_gen_C(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ u,
                                             const double* __restrict__ G, double* acc,
                                             const double* __restrict__ dtp) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const long long off = sh.J[0].gbase - sh.J[0].base;
  const bool pf = T.patches[sh.J[0].patch].pform != 0;
  mm_round<Cfg, false, false, true, true>(T, p, sh, dyn, LoadWeighted{G + off + 12 * T.Pg, nullptr, T.info, T.Pg},
                                            PutAcc{u, G + off, acc, T.P, T.Pg, T.gamma, *dtp, pf});
}

}  // namespace

void launch_mm_adj_gen_A(const DevTables& T, const MmTiles& t, const double* J, const double* u, const double* psi,
                         double* G, cudaStream_t st) {
  MM_LAUNCH(k_mm_adj_gen_A, mm_tail(t.cmax), J, u, psi, G);
}
void launch_mm_adj_gen_B(const DevTables& T, const MmTiles& t, const double* J, const double* u, const double* mu,
                         const double* psi, double* G, cudaStream_t st) {
  MM_LAUNCH(k_mm_adj_gen_B, mm_tail(t.cmax), J, u, mu, psi, G);
}
void launch_mm_adj_gen_C(const DevTables& T, const MmTiles& t, const double* u, const double* G, double* acc,
                         const double* dt, cudaStream_t st) {
  MM_LAUNCH(k_mm_adj_gen_C, mm_tail(t.cmax), u, G, acc, dt);
}

void set_mm_adj_gen_attributes(unsigned configs) {
  MM_OPT_IN(k_mm_adj_gen_A);
  MM_OPT_IN(k_mm_adj_gen_B);
  MM_OPT_IN(k_mm_adj_gen_C);
}

}  // namespace fcx
