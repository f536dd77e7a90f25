// FC line operators as exact tensor-core contractions (fc_split.cuh, fc_mmtab.h).
//
// GB300 executes 2 FP64 FMAs per clock and SM but about 1000 FP16 ones through mma.sync
// (profiles/mma_sync_probe.md), so the circulant of a continued line (21 FP16 digit products per
// entry, L^2/2 entries per line) costs less time than the FP64 butterflies of its two FFTs, by a
// factor of 2 at a few hundred points and about as much as them at 1024. What a line still needs
// from the FP64 pipe is its pointwise work: fluxes and stage combination.
//
// A CTA takes MM_LINES lines of one length (16 columns: 4 lines x 4 components): their values
// go to shared memory with lanes along the points, are continued there, and are replaced by
// the FP16 digits of the sums and differences of the two halves. A warp then contracts 16
// output rows of two lines at a time: the right operand's fragments come from shared memory
// (ldmatrix), the left operand is a Toeplitz matrix, so a fragment is three table entries of
// which each 16-column step needs two new ones (read through L1: all warps of an SM share a
// table of 24 bytes per entry). Digits need 12 bytes per point, component and part; 24
// accumulators per lane leave room for 24 warps per SM at 80 registers.
//
// Measured (28M points, affine lines of 48 to 384 points, per pass, FFT kernels -> these): q1 9.6
// -> 3.5 ms, q2 10.0 -> 5.0 ms, filter q1 + q2 17.5 -> 6.4 ms; a 128 x 128 operator with
// L = 155 = 5 x 31: 462 -> 23 us. Largest
// error on white lines 2.4e-16 of the largest value (FP64 FFT: 6e-16 to 9e-16). No pipe is
// full (FP64 and matrix pipes 15% to 39% busy): fixed latencies of the integer chains
// and the barriers between a tile's phases are what is left; 64 registers and 32 warps gained
// 1% in q1 and lost 6% in q2 (spills), quartering the even part (22% fewer matrix
// instructions, twice the live sums) lost 8% and 18%.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fc_internal.h"
#include "fc_line.cuh"
#include "fc_point.cuh"
#include "fc_split.cuh"

namespace fcx {

namespace {

constexpr int NCOL = 4 * MM_LINES;  // columns of a tile: component * MM_LINES + line

constexpr int CONT_PITCH = 24;  // FP16 per column of the end values' digits: 16 and a conflict-free pad

// static shared state of a tile
struct MmShared {
  Job J[MM_LINES];
  uint32_t emax[NCOL];  // high words of the largest magnitudes
  double fac[NCOL];     // value of one unit of a joined sum
  int fexp[NCOL];       // without the lines' scale: 2^fexp
  double tmp[NCOL * 16];  // detrended end values of the columns, 2d <= 16 each
  int cexp[NCOL];         // largest exponent of a column's weighted end values
  int sq[16];             // their weights (MmCont)
  __align__(16) uint16_t cdig[SP_DIGITS * NCOL * CONT_PITCH];  // their digits (FP16)
};

constexpr int LB = 4;  // points of a thread whose loads are in flight together

// pitch of a column's values in shared memory: 4 (mod 16) doubles keep the four lines of a
// row of q2 points in different banks
__host__ __device__ inline int mm_line_pitch(int L) { return L + ((4 - L % 16) + 16) % 16; }

__device__ __forceinline__ void mma16816(float* c, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t* r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

// table entries stay in L1 (every warp of the SM reads them)
__device__ __forceinline__ uint4 ldg_keep(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::evict_last.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ uint2 ldg_keep(const uint2* p) {
  uint2 v;
  asm volatile("ld.global.nc.L1::evict_last.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

// two biased values' digit k as an FP16 pair: the 10-bit fields become 1024 + field by
// setting the exponent bits, then 1536 comes off
__device__ __forceinline__ uint32_t digit_pair(long long a, long long b, int k) {
  const uint32_t fa = (uint32_t)(a >> (SP_BITS * (SP_DIGITS - 1 - k)));
  const uint32_t fb = (uint32_t)(b >> (SP_BITS * (SP_DIGITS - 1 - k)));
  uint32_t w = (__byte_perm(fa, fb, 0x5410) & 0x03ff03ffu) | 0x64006400u;
  __half2 h = __hsub2(*reinterpret_cast<__half2*>(&w), __half2half2(__ushort_as_half(0x6600)));
  return *reinterpret_cast<uint32_t*>(&h);
}

// adds the joined sums of one part over columns kb..ke-1 for the warp's 16 rows from i0 and
// its 8 columns: W[r * 2 + c] is row i0 + g + 8 r, column 2 t + c (g = lane / 4, t = lane % 4)
// (x0: table entry of row i0, column 0)
__device__ __forceinline__ void mm_part(const uint4* __restrict__ lo, const uint2* __restrict__ hi, int x0,
                                        uint32_t dig, int pitch, int kb, int ke, int lane, long long* W) {
  const int g = lane >> 2, t = lane & 3;
  float acc[SP_DIGITS][4];
#pragma unroll
  for (int l = 0; l < SP_DIGITS; ++l)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[l][q] = 0.f;
  const uint4* pl = lo + (x0 + kb + 2 * t - g);
  const uint2* ph = hi + (x0 + kb + 2 * t - g);
  uint32_t Am[SP_DIGITS], A0[SP_DIGITS], Ap[SP_DIGITS];
  auto entry = [&](uint32_t* A, int x) {
    const uint4 a = ldg_keep(pl + x);
    const uint2 b = ldg_keep(ph + x);
    A[0] = a.x;
    A[1] = a.y;
    A[2] = a.z;
    A[3] = a.w;
    A[4] = b.x;
    A[5] = b.y;
  };
  entry(Am, -8);
  // ldmatrix: the 8 columns of two digits, at k and k + 8 each
  const uint32_t slice = (uint32_t)NCOL * pitch;
  uint32_t baddr = dig + (uint32_t)((lane & 7) * pitch + ((lane >> 3) & 1) * 16 + kb * 2) + (lane >> 4) * slice;
#pragma unroll 1
  for (int k0 = 0; k0 < ke - kb; k0 += 16) {
    entry(A0, k0);
    entry(Ap, k0 + 8);
#pragma unroll
    for (int j2 = 0; j2 < SP_DIGITS; j2 += 2) {
      uint32_t b[4];
      ldsm4(b, baddr + j2 * slice);
#pragma unroll
      for (int i = 0; i + j2 < SP_DIGITS; ++i) {
        mma16816(acc[i + j2], A0[i], Am[i], Ap[i], A0[i], b[0], b[1]);
        if (i + j2 + 1 < SP_DIGITS) mma16816(acc[i + j2 + 1], A0[i], Am[i], Ap[i], A0[i], b[2], b[3]);
      }
    }
    baddr += 32;
#pragma unroll
    for (int i = 0; i < SP_DIGITS; ++i) Am[i] = Ap[i];
    sp_carries(acc, k0, ke - kb);
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    int s[SP_DIGITS];
#pragma unroll
    for (int l = 0; l < SP_DIGITS; ++l) s[l] = __float2int_rn(acc[l][q]);
    W[q] += sp_join(s);
  }
}

// the tile's point of a line (absent lines have the first line's addresses: read, never used)
__device__ __forceinline__ long long point(const MmShared& sh, int line, int t) {
  return sh.J[line].base + (long long)t * sh.J[line].stride;
}

// Continuation values of the tile's columns from their detrended end values (eq.
// continuation, as continue_lines): 2d FP64 operations per value, a quarter of a pass's FP64
// work, are one 16-column step of digit products instead (mm_continuation in fc_mmtab.h). A
// column's end values are scaled by the largest of their weighted magnitudes, not by the
// line's, so small second differences keep their bits.
template <int NT>
__device__ __forceinline__ void continuation(const uint4* __restrict__ frag, int C, MmShared& sh, double* ext, int LP) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  constexpr uint32_t pitch = CONT_PITCH * 2, slice = NCOL * pitch;
  for (int u = warp; 16 * (u >> 1) < C; u += NT / 32) {
    const int mb = u >> 1, n0 = 8 * (u & 1);
    const uint4* f = frag + (size_t)mb * SP_DIGITS * 32 + lane;
    uint4 A[SP_DIGITS];
#pragma unroll
    for (int j = 0; j < SP_DIGITS; ++j) A[j] = ldg_keep(f + 32 * j);
    float acc[SP_DIGITS][4];
#pragma unroll
    for (int l = 0; l < SP_DIGITS; ++l)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[l][q] = 0.f;
    const uint32_t addr = (uint32_t)__cvta_generic_to_shared(sh.cdig) +
                          (uint32_t)((n0 + (lane & 7)) * pitch + ((lane >> 3) & 1) * 16) + (lane >> 4) * slice;
#pragma unroll
    for (int j2 = 0; j2 < SP_DIGITS; j2 += 2) {
      uint32_t b[4];
      ldsm4(b, addr + j2 * slice);
#pragma unroll
      for (int i = 0; i + j2 < SP_DIGITS; ++i) {
        mma16816(acc[i + j2], A[i].x, A[i].y, A[i].z, A[i].w, b[0], b[1]);
        if (i + j2 + 1 < SP_DIGITS) mma16816(acc[i + j2 + 1], A[i].x, A[i].y, A[i].z, A[i].w, b[2], b[3]);
      }
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int k = 16 * mb + g + 8 * (q >> 1), col = n0 + 2 * t + (q & 1);
      int s[SP_DIGITS];
#pragma unroll
      for (int l = 0; l < SP_DIGITS; ++l) s[l] = __float2int_rn(acc[l][q]);
      const int e = sh.cexp[col] - 1023 - SP_DATA + SP_UNIT - SP_COEF;
      if (k < C) {
        const double x = sp_double_exp(sp_join(s), e, scalbn(1.0, e));
        ext[col * LP + k] = x;
        atomicMax(&sh.emax[col], sp_hi(x) & 0x7fffffffu);
      }
    }
  }
}

// One round: ld.raw(point, v) loads four values and ld.form(point, v) makes the point's four
// values to transform of them; the continued lines' operator (derivative, or the filter
// with FILT) is applied; ep.put(comp, point, op, value) takes the results, op =
// ep.pre(comp, point) loaded ahead for a batch of eight, or with PT ep.put(point, v[4]) a
// point's four at once (PT ops: ep.pre(point)). All threads of the CTA call it; it begins
// with a barrier. TR (with PT): the transposed operator (eqs. fc_der and filtering of a line
// extended by zeros; the derivative's circulant is odd, its transpose the negative; the
// results at the continuation points are folded back onto the first and last d points).
template <class Cfg, bool COL, bool FILT, bool PT, bool TR, class Load, class Ep>
__device__ __forceinline__ void mm_round(const DevTables& T, const MmPlan& plan, MmShared& sh, double2* dyn, Load ld,
                                         Ep ep) {
  constexpr int NT = Cfg::NT, S = Cfg::S, NW = NT / 32, TS = NT / 4;  // TS: points per step of a line
  // opaque copies: without them the compiler hoists the address arithmetic of both of a
  // kernel's rounds out of their loop (250 registers wanted instead of 160, at that time)
  int tid = threadIdx.x;
  MmPlan p = plan;
  asm volatile("" : "+r"(tid), "+r"(p.H), "+r"(p.Kp), "+r"(p.nx), "+r"(p.Mp));
  const int warp = tid >> 5, lane = tid & 31;
  const int n = sh.J[0].n, C = sh.J[0].C, fcm = sh.J[0].fcm, d = T.d, H = p.H;
  const int LP = mm_line_pitch(S * H);
  double* F = reinterpret_cast<double*>(dyn);  // [NCOL][LP]: the continued lines
  if (tid < NCOL) {
    sh.emax[tid] = 0;
    sh.cexp[tid] = 0;
    if (!TR && fcm >= 0) sh.sq[tid] = T.mmc[C].sq[tid];
  }
  __syncthreads();

  // (1) the lines' values into shared memory, and their maxima. q1 lines: a warp per line
  // (two with 256 threads), lanes along it; q2 lines: 4 neighbouring lines along the lanes
  {
    const int line = COL ? (tid & 3) : (warp & 3);
    const int t0 = COL ? tid >> 2 : (warp >> 2) * 32 + lane;
    const bool have = sh.J[line].n > 0;
    uint32_t hm[4] = {0, 0, 0, 0};
    for (int b = t0; b < n; b += LB * TS) {
      double X[LB][4];
#pragma unroll
      for (int r = 0; r < LB; ++r)  // the batch's loads first (absent points read the line's first one)
        ld.raw(point(sh, line, b + r * TS < n ? b + r * TS : 0), X[r]);
#pragma unroll
      for (int r = 0; r < LB; ++r) {
        const int t = b + r * TS;
        if (t < n) {
          double* v = X[r];
          if (have)
            ld.form(point(sh, line, t), v);
          else
            v[0] = v[1] = v[2] = v[3] = 0.0;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const uint32_t h = sp_hi(v[c]) & 0x7fffffffu;
            hm[c] = h > hm[c] ? h : hm[c];
            F[(c * MM_LINES + line) * LP + t] = v[c];
          }
        }
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (COL) {
        uint32_t h = hm[c];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) {
          const uint32_t g = __shfl_xor_sync(0xffffffffu, h, o);
          h = g > h ? g : h;
        }
        if (lane < MM_LINES) atomicMax(&sh.emax[c * MM_LINES + line], h);
      } else {
        const uint32_t h = __reduce_max_sync(0xffffffffu, hm[c]);
        if (lane == 0) atomicMax(&sh.emax[c * MM_LINES + line], h);
      }
    }
  }
  __syncthreads();

  // (2) continuation (eq. continuation) in the detrended form of continue_lines
  if (!TR && fcm >= 0) {
    for (int it = tid; it < NCOL * 2 * d; it += NT) {
      const int col = it & (NCOL - 1), q = it / NCOL;
      const double* x = F + col * LP;
      const double f0 = x[0], dl = x[1] - f0, fn = x[n - 1], dr = fn - x[n - 2];
      double v;
      if (q < d - 2) {
        v = fma(-(double)(q + 2), dl, x[q + 2] - f0);
      } else if (q < 2 * d - 4) {
        const int j = q - (d - 2);
        v = fma((double)(d - 1 - j), dr, x[n - d + j] - fn);
      } else {
        const int w = q - (2 * d - 4);
        v = w == 0 ? f0 : (w == 1 ? dl : (w == 2 ? fn : dr));
      }
      sh.tmp[col * 16 + q] = v;
      const int e = (int)((sp_hi(v) >> 20) & 0x7ffu);
      if (e > 0) atomicMax(&sh.cexp[col], e + sh.sq[q]);
      if (e == 0x7ff) atomicMax(&sh.emax[col], 0x7ff00000u);
    }
    __syncthreads();
    for (int it = tid; it < NCOL * 16; it += NT) {
      const int col = it & (NCOL - 1), q = it / NCOL;
      const long long x = q < 2 * d ? sp_fixed(sh.tmp[col * 16 + q], sh.cexp[col] - sh.sq[q]) : 0;
#pragma unroll
      for (int k = 0; k < SP_DIGITS; ++k)
        sh.cdig[(k * NCOL + col) * CONT_PITCH + q] = (uint16_t)digit_pair(x + SP_BIAS, 0, k);
    }
    __syncthreads();
    continuation<NT>(T.mmcf + T.mmc[C].first, C, sh, F + n, LP);
    __syncthreads();
  }
  const int te = FILT ? p.fte : p.dte;
  if (tid < NCOL) {
    const uint32_t h = sh.emax[tid], h2 = sh.emax[tid ^ MM_LINES];
    const double sc = FILT ? 1.0 : (TR ? -1.0 : 1.0) * sh.J[tid & (MM_LINES - 1)].scale;
    // a non-finite value spoils its line, and its packed partner's, as in the FFT kernels
    const int e = (int)(h >> 20) - 1023 - SP_DATA + SP_UNIT - te - (S - 1);
    const bool bad = h >= 0x7ff00000u || h2 >= 0x7ff00000u;
    sh.fac[tid] = bad ? __longlong_as_double(0x7ff8000000000000ll) : scalbn(sc, e);
    sh.fexp[tid] = bad ? 1 << 20 : e;  // the filter's factor is a power of two
  }

  // (3) digits of the parts, over the values: all reads come before the first write. A warp
  // per line again, lanes along the pairs (2q, 2q + 1). Digit column of (component, line):
  // 8 (line / 2) + 2 component + line % 2, so that a warp's 8 columns are two lines whole
  const int pitch = (p.Kp + 8) * 2;                         // bytes per column
  const uint32_t part1 = (uint32_t)(SP_DIGITS * NCOL) * pitch;  // bytes per part
  {
    constexpr int R = Cfg::R;  // pairs per thread
    const int line = warp & 3, q0 = (warp >> 2) * 32 + lane;
    double X[R][4][S][2];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            const int k = 2 * (q0 + r * TS) + a;
            X[r][c][s][a] = k < H && (!TR || k + s * H < n) ? F[(c * MM_LINES + line) * LP + k + s * H] : 0.0;
          }
    int ex[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) ex[c] = (int)(sh.emax[c * MM_LINES + line] >> 20);
    __syncthreads();
    char* dig = reinterpret_cast<char*>(dyn) + (8 * (line >> 1) + (line & 1)) * pitch;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int q = q0 + r * TS;
      if (2 * q < p.Kp) {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          long long w[S][2];
#pragma unroll
          for (int a = 0; a < 2; ++a) {
            const long long x0 = sp_fixed(X[r][c][0][a], ex[c]);
            if (S == 2) {
              const long long x1 = sp_fixed(X[r][c][S - 1][a], ex[c]);
              w[0][a] = x0 + x1 + SP_BIAS;
              w[S - 1][a] = x0 - x1 + SP_BIAS;
            } else {
              w[0][a] = x0 + SP_BIAS;
            }
          }
#pragma unroll
          for (int s = 0; s < S; ++s)
#pragma unroll
            for (int k = 0; k < SP_DIGITS; ++k)
              *(uint32_t*)(dig + s * part1 + (k * NCOL + 2 * c) * pitch + 4 * q) = digit_pair(w[s][0], w[s][1], k);
        }
      }
    }
  }
  __syncthreads();

  // (4) contraction and results: a warp takes 16 rows of two lines at a time
  const uint32_t dsh = (uint32_t)__cvta_generic_to_shared(dyn);
  const int tab = FILT ? p.ftab : p.dtab;
  const int g = lane >> 2, t = lane & 3;
  // TR: results at the end points and at the continuation points, past the digits
  double* endv = reinterpret_cast<double*>(reinterpret_cast<char*>(dyn) + S * part1);
  double* extv = endv + NCOL * 16;
  // joined sums y of rows i0 + g (+ 8) of lines l0, l0 + 1, component t: y[r * 2 + c]; the
  // results are at index row + off
  auto emit = [&](int i0, int l0, int off, const long long* y) {
    const double fac[2] = {sh.fac[t * MM_LINES + l0], sh.fac[t * MM_LINES + l0 + 1]};
    auto value = [&](long long w, int c) {
      return FILT ? sp_double_exp(w, sh.fexp[t * MM_LINES + l0 + c], fac[c]) : sp_double(w) * fac[c];
    };
    if constexpr (!PT) {
      const int stride = sh.J[0].stride;
      const long long base[2] = {sh.J[l0].base, sh.J[l0 + 1].base};
      const bool have[2] = {sh.J[l0].n > 0, sh.J[l0 + 1].n > 0};
      typename Ep::Op op[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {  // the operands of the four results in flight
        const int i = i0 + g + 8 * (q >> 1), idx = i + off;
        op[q] = ep.pre(t, base[q & 1] + (long long)(i < H && idx < n ? idx : 0) * stride);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = i0 + g + 8 * (q >> 1), idx = i + off;
        if (i < H && idx < n && have[q & 1])
          ep.put(t, base[q & 1] + (long long)idx * stride, op[q], value(y[q], q & 1));
      }
    } else {
      // the four lanes of a row hold its four components: a 4 x 4 transpose gives each lane
      // one point, row g + 8 (t / 2) of line l0 + t % 2
      const int i = i0 + g + 8 * (t >> 1), idx = i + off, ln = l0 + (t & 1);
      const bool in = i < H && sh.J[ln].n > 0;
      const typename Ep::Op op = ep.pre(point(sh, ln, i < H && idx < n ? idx : 0));
      double z[4], x[4], v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) z[q] = value(y[q], q & 1);
#pragma unroll
      for (int s = 0; s < 4; ++s) {  // x[s]: component t ^ s of this lane's point
        const int d = t ^ s;
        const double snd = d & 2 ? (d & 1 ? z[3] : z[2]) : (d & 1 ? z[1] : z[0]);
        x[s] = s ? __shfl_xor_sync(0xffffffffu, snd, s) : snd;
      }
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int s = c ^ t;
        v[c] = s & 2 ? (s & 1 ? x[3] : x[2]) : (s & 1 ? x[1] : x[0]);
      }
      if (TR && fcm >= 0 && in && (idx < d || idx >= n - d)) {  // completed after the fold
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int col = m * MM_LINES + ln;
          if (idx >= n)
            extv[col * C + idx - n] = v[m];
          else
            endv[col * 16 + (idx < d ? idx : d + idx - (n - d))] = v[m];
        }
      } else if (in && idx < n) {
        ep.put(point(sh, ln, idx), op, v);
      }
    }
  };
  // joined sums of part s for 16 rows from i0 and the two lines from l0, joined every MM_KCHUNK
  // columns (768 threads)
  auto part = [&](int s, int i0, int l0, long long* w) {
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = 0;
#pragma unroll 1
    for (int kb = 0; kb < (NT == 768 ? p.Kp : 1); kb += MM_KCHUNK)
      mm_part(T.mmlo + tab + s * p.nx, T.mmhi + tab + s * p.nx, p.Mp - i0, dsh + s * part1 + 4 * l0 * pitch, pitch, kb,
              NT == 768 && kb + MM_KCHUNK < p.Kp ? kb + MM_KCHUNK : p.Kp, lane, w);
  };
  for (int u = warp; 16 * (u >> 1) < H; u += NW) {
    const int i0 = 16 * (u >> 1), l0 = 2 * (u & 1);
    long long y[4];
    part(0, i0, l0, y);
    if constexpr (S == 2) {
      long long w[4];
      part(1, i0, l0, w);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long a = y[q];
        y[q] = a + w[q];
        w[q] = a - w[q];
      }
      emit(i0, l0, 0, y);
      emit(i0, l0, H, w);
    } else {
      emit(i0, l0, 0, y);
    }
  }
  if constexpr (TR) {
    if (fcm >= 0) {
      __syncthreads();
      const double* ML = T.rp + fcm;
      for (int it = tid; it < NCOL * 2 * d; it += NT) {
        const int col = it & (NCOL - 1), q = it / NCOL;
        const double* M = q < d ? ML + q : ML + C * d + q - d;
        double x = 0.0;
        for (int k = 0; k < C; ++k) x = fma(__ldg(M + k * d), extv[col * C + k], x);
        endv[col * 16 + q] += x;
      }
      __syncthreads();
      for (int it = tid; it < MM_LINES * 2 * d; it += NT) {
        const int ln = it & (MM_LINES - 1), q = it / MM_LINES, idx = q < d ? q : n - d + q - d;
        if (sh.J[ln].n > 0) {
          double v[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) v[m] = endv[(m * MM_LINES + ln) * 16 + q];
          const long long pt = point(sh, ln, idx);
          ep.put(pt, ep.pre(pt), v);
        }
      }
    }
  }
}

__device__ __forceinline__ void load_tile(MmShared& sh, const Job* __restrict__ jobs) {
  if (threadIdx.x < MM_LINES) sh.J[threadIdx.x] = jobs[(size_t)blockIdx.x * MM_LINES + threadIdx.x];
  __syncthreads();
}
// mu != 0 somewhere on the tile's lines (on every thread); lines of an inviscid tile are
// counted as skipped gradient rounds. A step's mu serves its five stages: flags, found once
// per step, replace ten scans of mu, each a chain of memory latencies at the head of a tile
// (7.5k of a tile's 120k cycles).
template <int NT, bool COL>
__device__ __forceinline__ bool tile_viscous(const DevTables& T, const MmShared& sh, const MmPlan& p,
                                             const double* __restrict__ mu, const uint8_t* __restrict__ flags,
                                             int dir) {
  bool visc;
  if (flags) {
    visc = flags[blockIdx.x] != 0;
  } else {
    bool v = false;
    const int n = sh.J[0].n;
    const int line = COL ? (threadIdx.x & 3) : (threadIdx.x >> 5) & 3;
    const int t0 = COL ? threadIdx.x >> 2 : (threadIdx.x & 31) + 32 * (threadIdx.x >> 7);
    for (int t = t0; t < n; t += NT / 2) {  // two loads in flight per thread and step
      const double a = mu[point(sh, line, t)], b = mu[point(sh, line, t + NT / 4 < n ? t + NT / 4 : t)];
      v |= a != 0.0 || b != 0.0;
    }
    v = v && sh.J[line].n > 0;
    visc = __syncthreads_or(v) != 0;
  }
  if (!visc && threadIdx.x < MM_LINES && sh.J[threadIdx.x].n > 0 && T.skip_lines) {
    const int L = p.H * p.S;
    atomicAdd(T.skip_lines + dir, 1ull);
    atomicAdd(T.skip_flops + dir, 4.0 * 5.0 * L * log2((double)L) + 16.0 * T.d * sh.J[0].C + 8.0 * L);
  }
  return visc;
}

// CTA configurations: NT threads (24 warps per SM resident, 80 registers a thread), S parts,
// R pairs of columns per thread in the digits phase
template <int NT_, int S_, int R_>
struct MmCfg {
  static constexpr int NT = NT_, S = S_, R = R_;
};
#define MM_BOUNDS __launch_bounds__(Cfg::NT, 768 / Cfg::NT)

struct NoOp {};
struct PutField {  // results into a field
  using Op = NoOp;
  double* f;
  long long cs;
  __device__ __forceinline__ NoOp pre(int, long long) const { return {}; }
  __device__ __forceinline__ void put(int c, long long q, NoOp, double v) const { f[q + c * cs] = v; }
};
struct PutField4 {
  using Op = NoOp;
  double* f;
  long long cs;
  __device__ __forceinline__ NoOp pre(long long) const { return {}; }
  __device__ __forceinline__ void put(long long q, NoOp, const double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) f[q + c * cs] = v[c];
  }
};
struct LoadField {
  const double* f;
  long long cs;
  __device__ __forceinline__ void raw(long long q, double* v) const {
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = f[q + c * cs];
  }
  __device__ __forceinline__ void form(long long, double*) const {}
};

}  // namespace

// dynamic shared memory: the digits [S][SP_DIGITS][NCOL][Kp + 8] of FP16 (columns padded by
// 16 bytes: conflict-free ldmatrix), over the continued lines [NCOL][pitch] they come from
inline size_t mm_smem(int S, int Kp) {
  const size_t dig = (size_t)S * SP_DIGITS * NCOL * (Kp + 8) * 2;
  const size_t val = (size_t)NCOL * mm_line_pitch(S * Kp) * sizeof(double);
  return dig > val ? dig : val;
}
// TAIL: the transposed operators' end and continuation results
inline size_t mm_tail(int cmax) { return (size_t)NCOL * (16 + cmax) * sizeof(double); }
#define MM_CASE(I, KERNEL, NT, S, R, ...)                                   \
  case I:                                                                   \
    KERNEL<MmCfg<NT, S, R>><<<t.n, NT, sm, st>>>(T, t.jobs, __VA_ARGS__);   \
    break;
#define MM_LAUNCH(KERNEL, TAIL, ...)                          \
  do {                                                        \
    if (t.n <= 0) return;                                     \
    const size_t sm = mm_smem(t.two ? 2 : 1, t.kp) + (TAIL);  \
    switch (mm_config(t)) {                                   \
      MM_CASE(0, KERNEL, 256, 1, 1, __VA_ARGS__)              \
      MM_CASE(1, KERNEL, 256, 2, 1, __VA_ARGS__)              \
      MM_CASE(2, KERNEL, 384, 1, 1, __VA_ARGS__)              \
      MM_CASE(3, KERNEL, 384, 2, 1, __VA_ARGS__)              \
      MM_CASE(4, KERNEL, 384, 1, 2, __VA_ARGS__)              \
      MM_CASE(5, KERNEL, 384, 2, 2, __VA_ARGS__)              \
      MM_CASE(6, KERNEL, 768, 1, 1, __VA_ARGS__)              \
      MM_CASE(7, KERNEL, 768, 2, 1, __VA_ARGS__)              \
      MM_CASE(8, KERNEL, 768, 1, 2, __VA_ARGS__)              \
      MM_CASE(9, KERNEL, 768, 2, 2, __VA_ARGS__)              \
    }                                                         \
  } while (0)

namespace {
template <class K>
void opt_in(unsigned configs, int i, K k) {
  if (configs >> i & 1)
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(mm_smem(2, MM_KMAX) + mm_tail(MM_CMAX)));
}
}  // namespace
#define MM_OPT_IN(KERNEL)                                                                                     \
  opt_in(configs, 0, KERNEL<MmCfg<256, 1, 1>>), opt_in(configs, 1, KERNEL<MmCfg<256, 2, 1>>),                 \
      opt_in(configs, 2, KERNEL<MmCfg<384, 1, 1>>), opt_in(configs, 3, KERNEL<MmCfg<384, 2, 1>>),             \
      opt_in(configs, 4, KERNEL<MmCfg<384, 1, 2>>), opt_in(configs, 5, KERNEL<MmCfg<384, 2, 2>>),             \
      opt_in(configs, 6, KERNEL<MmCfg<768, 1, 1>>), opt_in(configs, 7, KERNEL<MmCfg<768, 2, 1>>),             \
      opt_in(configs, 8, KERNEL<MmCfg<768, 1, 2>>), opt_in(configs, 9, KERNEL<MmCfg<768, 2, 2>>)

}  // namespace fcx
