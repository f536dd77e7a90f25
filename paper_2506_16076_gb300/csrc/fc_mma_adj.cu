// Contraction kernels of the discrete adjoint: affine lines and the filter's transpose (fc_mma.cuh).
#include "fc_mma.cuh"

namespace fcx {

namespace {

// ---- discrete adjoint (mu, dt frozen), affine lines. q1 (DIR 0): R1 = A_x^T eta_x -
// D_x^T (mu eta_x), eta_x = -D_x^T (N psi); q2: acc += dt (R1 + A_y^T eta_y - D_y^T (mu eta_y)).
// mu eta goes through Y to the second round, which an inviscid tile does not need.
struct LoadMasked {  // psi, 0 on PT_NODIFF points; second round: Y
  const double* f;
  const uint32_t* __restrict__ info;
  long long cs;
  bool second;
  __device__ __forceinline__ void raw(long long q, double* v) const {
    const bool z = !second && (info[q] & PT_NODIFF);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[q + c * cs];
    if (z) v[0] = v[1] = v[2] = v[3] = 0.0;
  }
  __device__ __forceinline__ void form(long long, double*) const {}
};
template <int DIR>
struct PutAdj {
  struct Op {
    double u[4], r[4], a[4], m;
  };
  const double* __restrict__ u;
  const double* __restrict__ mu;
  double* R1;
  double* acc;
  double* Y;
  long long cs;
  double gamma, dt;
  bool visc, second;
  __device__ __forceinline__ Op pre(long long q) const {
    Op o;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      o.u[c] = second ? 1.0 : u[q + c * cs];
      o.r[c] = DIR || second ? R1[q + c * cs] : 0.0;
      o.a[c] = DIR && (second || !visc) ? acc[q + c * cs] : 0.0;
    }
    o.m = visc && !second ? mu[q] : 0.0;
    return o;
  }
  __device__ __forceinline__ void put(long long q, const Op& o, const double* v) const {
    double r[4];
    if (second) {
#pragma unroll
      for (int c = 0; c < 4; ++c) r[c] = o.r[c] - v[c];
    } else {
      const double eta[4] = {-v[0], -v[1], -v[2], -v[3]};
      fluxT(DIR, o.u[0], o.u[1], o.u[2], o.u[3], gamma, eta, r);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        if (DIR) r[c] += o.r[c];
        if (visc) Y[q + c * cs] = o.m * eta[c];
      }
    }
    const bool last = second || !visc;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (DIR && last)
        acc[q + c * cs] = fma(dt, r[c], o.a[c]);
      else
        R1[q + c * cs] = r[c];
    }
  }
};
template <class Cfg, int DIR>
__device__ __forceinline__ void adj_cart(const DevTables& T, const Job* __restrict__ jobs, const double* u,
                                         const double* mu, const double* psi, double* R1, double* acc, double* Y,
                                         const double* dtp, const uint8_t* flags, double2* dyn,
                                         MmShared& sh) {
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  DevTables Tq = T;
  Tq.skip_lines = nullptr;  // the skipped rounds of the forward passes are the ones counted
  const bool visc = tile_viscous<Cfg::NT, DIR == 1>(Tq, sh, p, mu, flags, DIR);
  const double dt = DIR ? *dtp : 0.0;
#pragma unroll 1
  for (int rd = 0; rd < (visc ? 2 : 1); ++rd)
    mm_round<Cfg, DIR == 1, false, true, true>(T, p, sh, dyn, LoadMasked{rd ? Y : psi, T.info, T.P, rd == 1},
                                                 PutAdj<DIR>{u, mu, R1, acc, Y, T.P, T.gamma, dt, visc, rd == 1});
}
template <class Cfg>
__global__ void MM_BOUNDS k_mm_adj_q1(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ u,
                                          const double* __restrict__ mu, const double* __restrict__ psi, double* R1,
                                          double* acc, double* Y, const double* __restrict__ dtp,
                                          const uint8_t* __restrict__ flags) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  adj_cart<Cfg, 0>(T, jobs, u, mu, psi, R1, acc, Y, dtp, flags, dyn, sh);
}
template <class Cfg>
__global__ void MM_BOUNDS k_mm_adj_q2(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ u,
                                          const double* __restrict__ mu, const double* __restrict__ psi, double* R1,
                                          double* acc, double* Y, const double* __restrict__ dtp,
                                          const uint8_t* __restrict__ flags) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  adj_cart<Cfg, 1>(T, jobs, u, mu, psi, R1, acc, Y, dtp, flags, dyn, sh);
}

// transpose of the linearised filter (Sec. 4.3.1): q2 lines, lam (adjoint of the filtered
// state) with the E rebuild's Jacobian at ef (the filter's output) -> MF; q1 lines, MF ->
// out through theta's Jacobian at e (the state the filter was applied to)
struct LoadRebuildT {
  const double* __restrict__ lam;
  const double* __restrict__ ef;
  long long cs;
  double gamma;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = ef[q + c * cs];
  }
  __device__ __forceinline__ void form(long long q, double* v) const {
    const double l[4] = {lam[q], lam[q + cs], lam[q + 2 * cs], lam[q + 3 * cs]};
    double o[4];
    rebuild_T(l, v, gamma, o);
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = o[c];
  }
};
struct PutThetaT {
  struct Op {
    double e[4];
  };
  const double* __restrict__ e;
  double* __restrict__ out;
  long long cs;
  double gamma;
  __device__ __forceinline__ Op pre(long long q) const { return {{e[q], e[q + cs], e[q + 2 * cs], e[q + 3 * cs]}}; }
  __device__ __forceinline__ void put(long long q, const Op& o, const double* v) const {
    double r[4];
    theta_T(v, o.e, gamma, r);
#pragma unroll
    for (int c = 0; c < 4; ++c) out[q + c * cs] = r[c];
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_filterT_q2(DevTables T, const Job* __restrict__ jobs,
                                              const double* __restrict__ lam, const double* __restrict__ ef,
                                              double* __restrict__ MF) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  mm_round<Cfg, true, true, true, true>(T, p, sh, dyn, LoadRebuildT{lam, ef, T.P, T.gamma}, PutField4{MF, T.P});
}
template <class Cfg>
__global__ void MM_BOUNDS k_mm_filterT_q1(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ MF,
                                              const double* __restrict__ e, double* __restrict__ out) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  mm_round<Cfg, false, true, true, true>(T, p, sh, dyn, LoadField{MF, T.P}, PutThetaT{e, out, T.P, T.gamma});
}

}  // namespace

void launch_mm_adj_cart(const DevTables& T, const MmTiles& t, int dir, const double* u, const double* mu,
                        const double* psi, double* R1, double* acc, double* Y, const double* dt, cudaStream_t st) {
  if (dir == 0)
    MM_LAUNCH(k_mm_adj_q1, mm_tail(t.cmax), u, mu, psi, R1, acc, Y, dt, t.visc);
  else
    MM_LAUNCH(k_mm_adj_q2, mm_tail(t.cmax), u, mu, psi, R1, acc, Y, dt, t.visc);
}
void launch_mm_filterT_q2(const DevTables& T, const MmTiles& t, const double* lam, const double* ef, double* MF,
                          cudaStream_t st) {
  MM_LAUNCH(k_mm_filterT_q2, mm_tail(t.cmax), lam, ef, MF);
}
void launch_mm_filterT_q1(const DevTables& T, const MmTiles& t, const double* MF, const double* e, double* out,
                          cudaStream_t st) {
  MM_LAUNCH(k_mm_filterT_q1, mm_tail(t.cmax), MF, e, out);
}

void set_mm_adj_attributes(unsigned configs) {
  MM_OPT_IN(k_mm_adj_q1);
  MM_OPT_IN(k_mm_adj_q2);
  MM_OPT_IN(k_mm_filterT_q1);
  MM_OPT_IN(k_mm_filterT_q2);
}

}  // namespace fcx
