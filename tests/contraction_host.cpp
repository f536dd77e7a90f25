// Host build of the split-integer contraction (fc_split.cuh, fc_mmtab.h): the tables and
// the arithmetic the GPU kernels use, with the matrix products formed in plain loops.
//
//   contraction_host [filter alpha p] L1 L2 ...
//     for every continued length, the derivative and the filter (filter: only that one, with
//     sigma(z) = exp(-alpha z^p); else alpha = 10, p = 14) of a white line, a nearly
//     constant one and one with a spike against the same circulant in long double; prints
//     "L op kind error/max|x| largest_level_sum" (op 0: derivative, 1: filter; the error also over
//     the largest sigma), or "L none" when lines of this length are left to the FFT kernels.
//
//   contraction_host aligned L1 L2 ...
//     the derivative and the filter of lines whose digits carry the signs of one row's coefficients,
//     so that one level's sum is as large as it can be, summed in FP32 as the matrix
//     instruction does, with the carries between levels; prints "L op level part error/max|x|
//     largest_sum_of_levels_0_to_3".
//
//   contraction_host tables L1 L2 ...
//     prints "L derivative filter": whether the tables exist (alpha = 10, p = 14).
//
//   contraction_host continuation C Q
//     the continuation's digit products (mm_continuation, fragments read back as the matrix
//     instruction does) for a matrix whose columns differ in size, on end values that differ,
//     against long double; prints the error over the largest |coefficient x value|.
//
//   contraction_host quotient
//     quotient_f32 against the FP64 division rounded to FP32, on random quotients and on
//     quotients placed around the rounding midpoints; prints "tested different".
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "../paper_2506_16076_gb300/csrc/fc_mmtab.h"

using namespace fcx;

static double half_value(unsigned h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const double v = e ? std::ldexp(1024.0 + m, e - 25) : 0.0;
  return (h >> 15) & 1 ? -v : v;
}

static int quotients() {
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  long long n = 0, bad = 0;
  auto check = [&](double df, double rg) {
    const volatile double q = df / rg;
    const float a = quotient_f32(df, rg, 1.0 / rg), b = (float)q;
    ++n;
    bad += std::memcmp(&a, &b, 4) != 0;
  };
  for (int k = 0; k < 2000000; ++k) {
    const double rg = std::ldexp(1.0 + U(g), (int)(40 * U(g)) - 20);
    check(U(g) * rg, rg);
    // a quotient a few ulp around the midpoint of two FP32 numbers, and around one of them
    const float f = (float)std::ldexp(0.5 + 0.5 * U(g), -(int)(60 * U(g)));
    const double mid = 0.5 * ((double)f + (double)std::nextafter(f, 2.f));
    for (int u = -3; u <= 3; ++u) {
      check(std::min(rg, std::ldexp(std::nearbyint(std::ldexp(mid, 60)), -60) * rg * (1.0 + u * 1.1e-16)), rg);
      check(std::min(rg, (double)f * rg * (1.0 + u * 1.1e-16)), rg);
    }
    if (k < 1000) {
      check(0.0, rg);
      check(rg, rg);
      check(std::ldexp(rg, -200 - k / 2), rg);
    }
  }
  printf("%lld %lld\n", n, bad);
  return 0;
}

static int continuation(int C, int Q) {
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  std::vector<long double> M((size_t)C * Q);
  std::vector<uint4> lo(5);  // (a table does not start at 0)
  for (int k = 0; k < C; ++k)
    for (int q = 0; q < Q; ++q) M[(size_t)k * Q + q] = std::ldexp((long double)U(g), (int)(14.0 * q / Q));
  const MmCont r = mm_continuation(C, Q, M, lo);
  double worst = 0;
  for (int trial = 0; trial < 200; ++trial) {
    std::vector<double> e(Q);
    int ce = 0;
    for (int q = 0; q < Q; ++q) {
      e[q] = trial == 0 ? 0.0 : std::ldexp(U(g), -(int)(30 * (U(g) + 1.0)) * (trial % 3) - 14 * q / Q);
      const int x = (int)((sp_hi(e[q]) >> 20) & 0x7ffu);
      if (x > 0) ce = std::max(ce, x + r.sq[q]);
    }
    std::vector<long long> f(16, SP_BIAS);
    for (int q = 0; q < Q; ++q) f[q] += sp_fixed(e[q], ce - r.sq[q]);
    for (int k = 0; k < C; ++k) {
      double lev[SP_DIGITS] = {0};
      for (int q = 0; q < 16; ++q) {
        const int i = ((k & 15) >> 3) + 2 * (q >> 3), lane = (k & 7) * 4 + (q & 7) / 2;
        for (int u = 0; u < SP_DIGITS; ++u) {
          const uint4 a = lo[(size_t)r.first + ((k / 16) * SP_DIGITS + u) * 32 + lane];
          const unsigned w = i == 0 ? a.x : i == 1 ? a.y : i == 2 ? a.z : a.w;
          for (int v = 0; u + v < SP_DIGITS; ++v)
            lev[u + v] += half_value(q & 1 ? w >> 16 : w & 0xffff) * ((int)sp_field(f[q], v) - 512);
        }
      }
      int si[SP_DIGITS];
      for (int l = 0; l < SP_DIGITS; ++l) si[l] = (int)lev[l];
      const int x = ce - 1023 - SP_DATA + SP_UNIT - SP_COEF;
      const double got = sp_double_exp(sp_join(si), x, std::scalbn(1.0, x));
      long double ref = 0, top = 0;
      for (int q = 0; q < Q; ++q) {
        ref += M[(size_t)k * Q + q] * e[q];
        top = std::max(top, std::ldexp(std::fabs((long double)e[q]), r.sq[q]));
      }
      if (top > 0) worst = std::max(worst, (double)(std::fabs(got - ref) / top));
      if (trial == 0 && got != 0.0) worst = 1.0;
    }
  }
  printf("%.3e\n", worst);
  return 0;
}

static std::vector<long double> default_sigma(int L) {
  std::vector<long double> sig;
  for (int k = 0; 2 * k <= L; ++k) sig.push_back(expl(-10.0L * powl(2.0L * k / L, 14)));
  return sig;
}

static int tables(int n, char** v) {
  for (int a = 0; a < n; ++a) {
    const int L = std::atoi(v[a]);
    std::vector<uint4> lo;
    std::vector<uint2> hi;
    const std::vector<long double> sig = default_sigma(L);
    const MmPlan p = mm_plan(L, &sig, lo, hi);
    printf("%d %d %d\n", L, p.dtab >= 0, p.ftab >= 0);
  }
  return 0;
}

static int aligned(int n, char** v) {
  std::mt19937_64 g(5);
  const long double PI = 3.14159265358979323846264338327950288L;
  for (int a = 0; a < n; ++a) {
    const int L = std::atoi(v[a]);
    std::vector<uint4> lo;
    std::vector<uint2> hi;
    const std::vector<long double> sig = default_sigma(L);
    const MmPlan p = mm_plan(L, &sig, lo, hi);
    for (int op = 0; op < 2; ++op) {
      const int te = op ? p.fte : p.dte, tab = op ? p.ftab : p.dtab;
      std::vector<long double> c(L);  // the circulant
      for (int m = 0; m < L; ++m) {
        long double s = op ? sig[0] : 0.0L;
        for (int k = 1; 2 * k <= L; ++k) {
          const long double an = 2.0L * PI * ((long long)k * m % L) / L;
          if (op == 0)
            s += 2 * k < L ? -2.0L * (2.0L * PI * k / L) * sinl(an) : 0.0L;
          else
            s += (2 * k < L ? 2.0L : 1.0L) * sig[k] * cosl(an);
        }
        c[m] = s / L;
      }
      auto coef = [&](int s, int at, int* d) {
        const int e = tab + s * p.nx + at;
        const unsigned w[SP_DIGITS] = {lo[e].x, lo[e].y, lo[e].z, lo[e].w, hi[e].x, hi[e].y};
        for (int u = 0; u < SP_DIGITS; ++u) d[u] = (int)half_value(w[u] & 0xffff);
      };
      for (int level = 1; level < 4; ++level)
        for (int part = 0; part < p.S; ++part) {
          const int row = (int)(g() % p.H);
          std::vector<double> x(L, 0.0);
          for (int k = 0; k < p.H; ++k) {
            int d[SP_DIGITS];
            coef(part, k - row + p.Mp, d);
            long long val = 0;
            for (int j = 0; j < SP_DIGITS - 1; ++j) {
              const int big = j ? 511 : 127 * p.S, any = (int)(g() % (2 * big + 1)) - big;
              val += (long long)(j <= level ? (d[level - j] < 0 ? -big : big) : any) << (SP_BITS * (SP_DIGITS - 1 - j));
            }
            const long long h = p.S == 2 ? val / 2 : val;
            x[k] = std::ldexp((double)h, -57);
            if (p.S == 2) x[k + p.H] = std::ldexp((double)(part ? h - val : val - h), -57);
          }
          double top = 0;
          for (double y : x) top = std::max(top, std::fabs(y));
          const int ex = (int)((sp_hi(top) >> 20) & 0x7ff);
          std::vector<long long> W[2];
          double largest = 0;
          for (int s = 0; s < p.S; ++s)
            for (int i = 0; i < p.H; ++i) {
              unsigned long long joined = 0;
              for (int kb = 0; kb < p.Kp; kb += MM_KCHUNK) {
                float acc[SP_DIGITS][1] = {};
                const int nk = std::min(p.Kp - kb, MM_KCHUNK);
                for (int k0 = 0; k0 < nk; k0 += 16) {
                  double step[SP_DIGITS][SP_DIGITS] = {};
                  for (int k = kb + k0; k < std::min(p.H, kb + k0 + 16); ++k) {
                    const long long x0 = sp_fixed(x[k], ex), x1 = p.S == 2 ? sp_fixed(x[k + p.H], ex) : 0;
                    const long long b = (s ? x0 - x1 : x0 + x1) + SP_BIAS;
                    int d[SP_DIGITS];
                    coef(s, k - i + p.Mp, d);
                    for (int u = 0; u < SP_DIGITS; ++u)
                      for (int w = 0; u + w < SP_DIGITS; ++w) step[u][w] += (double)d[u] * ((int)sp_field(b, w) - 512);
                  }
                  for (int w = 0; w < SP_DIGITS; ++w)
                    for (int u = 0; u + w < SP_DIGITS; ++u) {
                      acc[u + w][0] = (float)(acc[u + w][0] + step[u][w]);
                      if (u + w < 4) largest = std::max(largest, (double)std::fabs(acc[u + w][0]));
                    }
                  sp_carries(acc, k0, nk);
                }
                int si[SP_DIGITS];
                for (int l = 0; l < SP_DIGITS; ++l) si[l] = (int)acc[l][0];
                joined += (unsigned long long)sp_join(si);
              }
              W[s].push_back((long long)joined);
            }
          const double fac = std::scalbn(1.0, ex - 1023 - SP_DATA + SP_UNIT - te - (p.S - 1));
          double err = 0;
          for (int i = 0; i < L; ++i) {
            const long long y = p.S == 1 ? W[0][i] : (i < p.H ? W[0][i] + W[1][i] : W[0][i - p.H] - W[1][i - p.H]);
            long double ref = 0;
            for (int j = 0; j < L; ++j) ref += c[((i - j) % L + L) % L] * (long double)x[j];
            err = std::max(err, (double)fabsl((long double)sp_double(y) * fac - ref));
          }
          printf("%d %d %d %d %.3e %.0f\n", L, op, level, part, err / top, largest);
        }
    }
  }
  return 0;
}

int main(int argc, char** argv) {
  if (argc > 2 && !std::strcmp(argv[1], "aligned")) return aligned(argc - 2, argv + 2);
  if (argc > 2 && !std::strcmp(argv[1], "tables")) return tables(argc - 2, argv + 2);
  if (argc == 4 && !std::strcmp(argv[1], "continuation")) return continuation(std::atoi(argv[2]), std::atoi(argv[3]));
  if (argc == 2 && !std::strcmp(argv[1], "quotient")) return quotients();
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  const long double PI = 3.14159265358979323846264338327950288L;
  const bool filter = argc > 4 && !std::strcmp(argv[1], "filter");
  const long double alpha = filter ? std::atof(argv[2]) : 10.0L, pw = filter ? std::atof(argv[3]) : 14.0L;
  for (int a = filter ? 4 : 1; a < argc; ++a) {
    const int L = std::atoi(argv[a]);
    if (!mm_length_ok(L)) {
      printf("%d none\n", L);
      continue;
    }
    std::vector<uint4> lo;
    std::vector<uint2> hi;
    std::vector<long double> sig;
    for (int k = 0; 2 * k <= L; ++k) sig.push_back(expl(-alpha * powl(2.0L * k / L, pw)));
    const double stop = (double)*std::max_element(sig.begin(), sig.end());
    const MmPlan p = mm_plan(L, &sig, lo, hi);
    if (filter && p.ftab < 0) printf("%d none\n", L);
    for (int op = filter; op < (p.ftab < 0 ? 1 : 2); ++op) {
      std::vector<long double> c(L, 0.0L);  // the circulant, by its definition
      for (int m = 0; m < L; ++m) {
        long double s = 0;
        for (int k = 1; 2 * k <= L; ++k) {
          const long double an = 2.0L * PI * ((long long)k * m % L) / L;
          if (op == 0)
            s += 2 * k < L ? -2.0L * (2.0L * PI * k / L) * sinl(an) : 0.0L;
          else
            s += (2 * k < L ? 2.0L : 1.0L) * sig[k] * cosl(an);
        }
        c[m] = (s + (op ? sig[0] : 0.0L)) / L;
      }
      for (int kind = 0; kind < 3; ++kind) {
        std::vector<double> x(L);
        double top = 0;
        for (int i = 0; i < L; ++i) {
          x[i] = kind == 0 ? U(g) : kind == 1 ? 1.4 + 0.01 * std::sin(6.283185307179586 * 3 * i / L) : 1e-3 * U(g);
          if (kind == 2 && i == L / 3) x[i] = 1000.0;
          top = std::max(top, std::fabs(x[i]));
        }
        const int ex = (int)((sp_hi(top) >> 20) & 0x7ff), te = op ? p.fte : p.dte, tab = op ? p.ftab : p.dtab;
        std::vector<long long> W[2];
        double level = 0;
        for (int s = 0; s < p.S; ++s)
          for (int i = 0; i < p.H; ++i) {
            long long joined = 0;
            for (int kb = 0; kb < p.H; kb += MM_KCHUNK) {
            double lev[SP_DIGITS] = {0};
            for (int k = kb; k < std::min(p.H, kb + MM_KCHUNK); ++k) {
              const long long x0 = sp_fixed(x[k], ex), x1 = p.S == 2 ? sp_fixed(x[k + p.H], ex) : 0;
              const long long b = (s ? x0 - x1 : x0 + x1) + SP_BIAS;
              const int at = tab + s * p.nx + k - i + p.Mp;
              const unsigned w[SP_DIGITS] = {lo[at].x, lo[at].y, lo[at].z, lo[at].w, hi[at].x, hi[at].y};
              for (int u = 0; u < SP_DIGITS; ++u)
                for (int v = 0; u + v < SP_DIGITS; ++v)
                  lev[u + v] += half_value(w[u] & 0xffff) * ((int)sp_field(b, v) - 512);
            }
            int si[SP_DIGITS];
            for (int l = 0; l < SP_DIGITS; ++l) {
              si[l] = (int)lev[l];
              level = std::max(level, std::fabs(lev[l]));
            }
            joined = (long long)((unsigned long long)joined + (unsigned long long)sp_join(si));
            }
            W[s].push_back(joined);
          }
        const double fac = std::scalbn(1.0, ex - 1023 - SP_DATA + SP_UNIT - te - (p.S - 1));
        double err = 0;
        for (int i = 0; i < L; ++i) {
          const long long v = p.S == 1 ? W[0][i] : (i < p.H ? W[0][i] + W[1][i] : W[0][i - p.H] - W[1][i - p.H]);
          long double ref = 0;
          for (int j = 0; j < L; ++j) ref += c[((i - j) % L + L) % L] * (long double)x[j];
          err = std::max(err, (double)fabsl((long double)(sp_double(v) * fac) - ref));
        }
        printf("%d %d %d %.3e %.0f\n", L, op, kind, err / top / (op ? stop : 1.0), level);
      }
    }
  }
  return 0;
}
