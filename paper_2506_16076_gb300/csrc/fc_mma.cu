// Contraction kernels of the affine passes and of the filter (fc_mma.cuh).
#include "fc_mma.cuh"

namespace fcx {

namespace {

// affine q1 lines: R1 = d/dx (f_x(e) - mu d/dx e); Fy: the points' y fluxes
struct LoadQ1 {
  const double* __restrict__ e;
  const double* __restrict__ mu;
  const double* R1;
  double* __restrict__ Fy;
  long long cs;
  double gamma;
  bool grad, visc;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = e[q + c * cs];
  }
  __device__ __forceinline__ void form(long long q, double* v) const {
    if (grad) return;
    double f[4], fy[4];
    flux_xy(v[0], v[1], v[2], v[3], gamma, f, fy);
#pragma unroll
    for (int c = 0; c < 4; ++c) Fy[q + c * cs] = fy[c];
    if (visc) {
      const double m = mu[q];
#pragma unroll
      for (int c = 0; c < 4; ++c) f[c] = fma(-m, R1[q + c * cs], f[c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[c];
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_cart_q1(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ e,
                                           const double* __restrict__ mu, double* R1, double* __restrict__ Fy,
                                           const uint8_t* __restrict__ flags) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const bool visc = tile_viscous<Cfg::NT, false>(T, sh, p, mu, flags, 0);
  // viscous tiles: the gradient goes through R1 (a round's opening barrier orders it)
#pragma unroll 1
  for (int rd = visc ? 0 : 1; rd < 2; ++rd)
    mm_round<Cfg, false, false, false, false>(T, p, sh, dyn, LoadQ1{e, mu, R1, Fy, T.P, T.gamma, rd == 0, visc},
                                         PutField{R1, T.P});
}

// affine q2 lines: L = -(R1 + d/dy (f_y(e) - mu d/dy e)) and the stage combination; the y
// fluxes come from the q1 pass and become the viscous ones in place
struct PutQ2 {
  struct Op {
    double a, cur, u0, aux;  // gradient round: Fy and mu in a and cur
    uint32_t info;
  };
  const double* __restrict__ mu;
  const double* __restrict__ R1;
  double* Fy;
  const uint32_t* __restrict__ info;
  StageCoef sc;
  double dt;
  long long cs;
  bool grad;
  __device__ __forceinline__ Op pre(int c, long long q) const {
    Op o;
    const long long qc = q + c * cs;
    if (grad) {
      o.a = Fy[qc];
      o.cur = mu[q];
      o.u0 = o.aux = 0.0;
      o.info = 0;
    } else {
      o.a = R1[qc];
      o.info = info[q];
      o.cur = o.u0 = o.aux = 0.0;
      if (!sc.rhs_only) {
        o.cur = sc.Ucur[qc];
        if (sc.c0 != 0.0) o.u0 = sc.U0[qc];
        if (sc.Uaux) o.aux = sc.Uaux[qc];
      }
    }
    return o;
  }
  __device__ __forceinline__ void put(int c, long long q, const Op& o, double v) const {
    const long long qc = q + c * cs;
    if (grad)
      Fy[qc] = fma(-o.cur, v, o.a);
    else
      stage_put(sc, dt, qc, (o.info & PT_NODIFF) ? 0.0 : -(o.a + v), o.cur, o.u0, o.aux);
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_cart_q2(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ mu,
                                           const double* __restrict__ R1, double* Fy,
                                           const uint8_t* __restrict__ flags, StageCoef sc) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  const bool visc = tile_viscous<Cfg::NT, true>(T, sh, p, mu, flags, 1);
  const double dt = sc.rhs_only ? 0.0 : *sc.dt;
#pragma unroll 1
  for (int rd = visc ? 0 : 1; rd < 2; ++rd)
    mm_round<Cfg, true, false, false, false>(T, p, sh, dyn, LoadField{rd == 0 ? sc.Ucur : Fy, T.P},
                                        PutQ2{mu, R1, Fy, T.info, sc, dt, T.P, rd == 0});
}

// filter, q1 lines: (rho, rho u, rho v, theta) filtered into F
struct LoadTheta {
  const double* __restrict__ e;
  long long cs;
  double gamma;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = e[q + c * cs];
  }
  __device__ __forceinline__ void form(long long, double* v) const { v[3] = theta_of(v[0], v[1], v[2], v[3], gamma); }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_filter_q1(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ e,
                                             double* __restrict__ F) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  mm_round<Cfg, false, true, false, false>(T, p, sh, dyn, LoadTheta{e, T.P, T.gamma}, PutField{F, T.P});
}

// filter, q2 lines, and E rebuilt
struct PutEnergy {
  using Op = NoOp;
  double* __restrict__ e;
  long long cs;
  double gamma;
  __device__ __forceinline__ NoOp pre(long long) const { return {}; }
  __device__ __forceinline__ void put(long long q, NoOp, const double* v) const {
    e[q] = v[0];
    e[q + cs] = v[1];
    e[q + 2 * cs] = v[2];
    e[q + 3 * cs] = energy_of(v[0], v[1], v[2], v[3], gamma);
  }
};
template <class Cfg>
__global__ void MM_BOUNDS k_mm_filter_q2(DevTables T, const Job* __restrict__ jobs, const double* __restrict__ F,
                                             double* __restrict__ e) {
  extern __shared__ double2 dyn[];
  __shared__ MmShared sh;
  load_tile(sh, jobs);
  const MmPlan p = T.mm[sh.J[0].plan];
  mm_round<Cfg, true, true, true, false>(T, p, sh, dyn, LoadField{F, T.P}, PutEnergy{e, T.P, T.gamma});
}

// one warp per tile: mu != 0 on one of its lines
__global__ void k_tile_flags(const Job* __restrict__ jobs, int n, const double* __restrict__ mu,
                             uint8_t* __restrict__ flags) {
  const int tile = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  if (tile >= n) return;
  const Job* J = jobs + (size_t)tile * MM_LINES;
  const bool col = J[0].stride != 1;
  bool v = false;
  for (int l = 0; l < (col ? 1 : MM_LINES); ++l) {  // columns: the four lines side by side
    const Job& K = J[col ? (lane & 3) : l];
    for (int t = col ? lane >> 2 : lane; t < K.n; t += col ? 8 : 32) v |= mu[K.base + (long long)t * K.stride] != 0.0;
  }
  v = __any_sync(0xffffffffu, v);
  if (lane == 0) flags[tile] = v;
}

}  // namespace

void launch_tile_flags(const Job* jobs, int n, const double* mu, uint8_t* visc, cudaStream_t st) {
  if (n > 0) k_tile_flags<<<(n + 7) / 8, 256, 0, st>>>(jobs, n, mu, visc);
}
void launch_mm_cart_q1(const DevTables& T, const MmTiles& t, const double* e, const double* mu, double* R1, double* Fy,
                       cudaStream_t st) {
  MM_LAUNCH(k_mm_cart_q1, 0, e, mu, R1, Fy, t.visc);
}
void launch_mm_cart_q2(const DevTables& T, const MmTiles& t, const double* mu, const double* R1, double* Fy,
                       const StageCoef& sc, cudaStream_t st) {
  MM_LAUNCH(k_mm_cart_q2, 0, mu, R1, Fy, t.visc, sc);
}
void launch_mm_filter_q1(const DevTables& T, const MmTiles& t, const double* e, double* F, cudaStream_t st) {
  MM_LAUNCH(k_mm_filter_q1, 0, e, F);
}
void launch_mm_filter_q2(const DevTables& T, const MmTiles& t, const double* F, double* e, cudaStream_t st) {
  MM_LAUNCH(k_mm_filter_q2, 0, F, e);
}

void set_mm_attributes(unsigned configs) {
  MM_OPT_IN(k_mm_cart_q1);
  MM_OPT_IN(k_mm_cart_q2);
  MM_OPT_IN(k_mm_filter_q1);
  MM_OPT_IN(k_mm_filter_q2);
}

}  // namespace fcx
