// Contraction kernels of the curvilinear passes (fc_mma.cuh).
#include "fc_mma.cuh"

namespace fcx {

namespace {

// ---- curvilinear patches: passes A (q1), B (q2), C (q1) of the stage (fc_kernels.cu has the
// same passes on the FFT engine, with the scratch slots' meaning). g: a point's scratch index
__device__ __forceinline__ double* slot(double* G, long long Pg, int s, int c) { return G + (4 * s + c) * Pg; }

struct LoadState {  // e, or (rho, rho u, rho v, theta) for the product-rule form
  const double* __restrict__ e;
  long long cs;
  double gamma;
  bool theta;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = e[q + c * cs];
  }
  __device__ __forceinline__ void form(long long, double* v) const {
    if (theta) v[3] = theta_of(v[0], v[1], v[2], v[3], gamma);
  }
};
struct PutSlot {
  using Op = NoOp;
  double* G;  // + the offset from state to scratch index
  long long Pg;
  int s;
  __device__ __forceinline__ NoOp pre(int, long long) const { return {}; }
  __device__ __forceinline__ void put(int c, long long q, NoOp, double v) const { G[(4 * s + c) * Pg + q] = v; }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_gen_A(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ e,
                                         double* __restrict__ G) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const bool pf = T.patches[sh.J[0].patch].pform != 0;
  mm_round<Cfg, false, false, false, false>(T, p, sh, dyn, LoadState{e, T.P, T.gamma, pf},
                                              PutSlot{G + (sh.J[0].gbase - sh.J[0].base), T.Pg, 0});
}

// pass B, three rounds: D2 e, then H_x and H_y from both derivatives; R2 = J2x D2 H_x + J2y D2 H_y
struct LoadB {
  const double* __restrict__ e;
  const double* G;  // + offset
  long long cs, Pg;
  double gamma;
  int rd;
  bool pf;
  __device__ __forceinline__ void raw(long long q, double* v) const {
    const double* f = rd == 0 ? e : G + (rd == 1 ? 4 : 8) * Pg;
    const long long st = rd == 0 ? cs : Pg;
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[q + c * st];
  }
  __device__ __forceinline__ void form(long long, double* v) const {
    if (rd == 0 && pf) v[3] = theta_of(v[0], v[1], v[2], v[3], gamma);
  }
};
struct PutB {
  struct Op {
    double a[4], r[4];  // round 0: e and D1; later: the slot-3 sum so far in r
    double j[4], m;
  };
  const double* __restrict__ e;
  const double* __restrict__ mu;
  const double* __restrict__ Jm;  // + offset
  double* G;                      // + offset
  long long cs, Pg;
  double gamma;
  int rd;
  bool pf;
  __device__ __forceinline__ Op pre(long long q) const {
    Op o;
    if (rd == 0) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        o.a[c] = e[q + c * cs];
        o.r[c] = G[c * Pg + q];
        o.j[c] = Jm[c * Pg + q];
      }
      o.m = mu[q];
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        o.a[c] = o.j[c] = 0.0;
        o.r[c] = rd == 2 || pf ? G[(12 + c) * Pg + q] : 0.0;
      }
      o.j[0] = Jm[(rd == 1 ? 2 : 3) * Pg + q];
      o.m = 0.0;
    }
    return o;
  }
  __device__ __forceinline__ void put(long long q, const Op& o, const double* d2) const {
    if (rd > 0) {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        G[(12 + c) * Pg + q] = rd == 1 && !pf ? o.j[0] * d2[c] : fma(o.j[0], d2[c], o.r[c]);
      return;
    }
    double gx[4], gy[4], hx[4], hy[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      gx[c] = fma(o.j[0], o.r[c], o.j[2] * d2[c]);
      gy[c] = fma(o.j[1], o.r[c], o.j[3] * d2[c]);
    }
    if (pf) {
      const double th = theta_of(o.a[0], o.a[1], o.a[2], o.a[3], gamma);
      const double Q[4] = {o.a[0], o.a[1], o.a[2], th};
      double ex[4], ey[4], px, py, div[4];
      product_rule(Q, gx, gamma - 1.0, ex, px);
      product_rule(Q, gy, gamma - 1.0, ey, py);
      conv_div_product(o.a, th, ex, px, ey, py, div);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        hx[c] = -o.m * ex[c];
        hy[c] = -o.m * ey[c];
        G[(12 + c) * Pg + q] = div[c];
      }
    } else {
      double fx[4], fy[4];
      flux_xy(o.a[0], o.a[1], o.a[2], o.a[3], gamma, fx, fy);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        hx[c] = fma(-o.m, gx[c], fx[c]);
        hy[c] = fma(-o.m, gy[c], fy[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      G[(4 + c) * Pg + q] = hx[c];
      G[(8 + c) * Pg + q] = hy[c];
    }
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_gen_B(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ e,
                                         const double* __restrict__ mu, const double* __restrict__ Jm, double* G) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const bool pf = T.patches[sh.J[0].patch].pform != 0;
  const long long off = sh.J[0].gbase - sh.J[0].base;
#pragma unroll 1
  for (int rd = 0; rd < 3; ++rd)
    mm_round<Cfg, true, false, true, false>(T, p, sh, dyn, LoadB{e, G + off, T.P, T.Pg, T.gamma, rd, pf},
                                              PutB{e, mu, Jm + off, G + off, T.P, T.Pg, T.gamma, rd, pf});
}

// pass C, two rounds: R1 = J1x D1 H_x + J1y D1 H_y; L = -(R1 + R2); stage combination
struct LoadC {
  const double* G;  // + offset
  long long Pg;
  int rd;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = G[(4 + 4 * rd + c) * Pg + q];
  }
  __device__ __forceinline__ void form(long long, double*) const {}
};
struct PutC {
  struct Op {
    double j, r1, r2, cur, u0, aux;
    uint32_t info;
  };
  const double* __restrict__ Jm;  // + offset
  double* G;                      // + offset
  const uint32_t* __restrict__ info;
  StageCoef sc;
  double dt;
  long long cs, Pg;
  int rd;
  __device__ __forceinline__ Op pre(int c, long long q) const {
    Op o;
    o.j = Jm[rd * Pg + q];
    o.r1 = o.r2 = o.cur = o.u0 = o.aux = 0.0;
    o.info = 0;
    if (rd == 1) {
      const long long qc = q + c * cs;
      o.r1 = G[c * Pg + q];
      o.r2 = G[(12 + c) * Pg + q];
      o.info = info[q];
      if (!sc.rhs_only) {
        o.cur = sc.Ucur[qc];
        if (sc.c0 != 0.0) o.u0 = sc.U0[qc];
        if (sc.Uaux) o.aux = sc.Uaux[qc];
      }
    }
    return o;
  }
  __device__ __forceinline__ void put(int c, long long q, const Op& o, double v) const {
    if (rd == 0)
      G[c * Pg + q] = o.j * v;
    else
      stage_put(sc, dt, q + c * cs, (o.info & PT_NODIFF) ? 0.0 : -(fma(o.j, v, o.r1) + o.r2), o.cur, o.u0, o.aux);
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_gen_C(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ Jm,
                                         double* G, StageCoef sc) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const long long off = sh.J[0].gbase - sh.J[0].base;
  const double dt = sc.rhs_only ? 0.0 : *sc.dt;
#pragma unroll 1
  for (int rd = 0; rd < 2; ++rd)
    mm_round<Cfg, false, false, false, false>(T, p, sh, dyn, LoadC{G + off, T.Pg, rd},
                                                PutC{Jm + off, G + off, T.info, sc, dt, T.P, T.Pg, rd});
}

}  // namespace

void launch_mm_gen_A(const DevTables& T, const MmTiles& t, const double* e, double* G, cudaStream_t st) {
  MM_LAUNCH(k_mm_gen_A, 0, e, G);
}
void launch_mm_gen_B(const DevTables& T, const MmTiles& t, const double* e, const double* mu, const double* J,
                     double* G, cudaStream_t st) {
  MM_LAUNCH(k_mm_gen_B, 0, e, mu, J, G);
}
void launch_mm_gen_C(const DevTables& T, const MmTiles& t, const double* J, double* G, const StageCoef& sc,
                     cudaStream_t st) {
  MM_LAUNCH(k_mm_gen_C, 0, J, G, sc);
}

void set_mm_gen_attributes(unsigned configs) {
  MM_OPT_IN(k_mm_gen_A);
  MM_OPT_IN(k_mm_gen_B);
  MM_OPT_IN(k_mm_gen_C);
}

}  // namespace fcx
