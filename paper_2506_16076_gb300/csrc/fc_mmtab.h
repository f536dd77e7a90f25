// Host-side builder of the coefficient tables of the tensor-core line contractions
// (fc_mma.cu): per continued length, the digits of the circulant's coefficients in the
// order in which a warp's matrix fragments read them.
//
// Even L = 2H: with u_j = x_j + x_{j+H}, v_j = x_j - x_{j+H} (j < H) and
//   U_i = sum_j (c(i-j) + c(i-j+H)) u_j,  V_i = sum_j (c(i-j) - c(i-j+H)) v_j,
// y_i = (U_i + V_i) / 2 and y_{i+H} = (U_i - V_i) / 2: half the products of the direct
// sum (two parts of H x H). Odd L: one part of L x L. The left operand of part s is the
// Toeplitz matrix t_s(i - k); a table holds r(x) = t_s(off - x) at x = k - i + off, one
// entry per x with the digits of r(x) and r(x+1) side by side (a fragment's register).
//
// Derivative (per index): c(m) = (pi/L) (-1)^m cot(pi m / L) for even L (the Nyquist mode
// has no derivative), (pi/L) (-1)^m / sin(pi m / L) for odd L. Filter: c(m) =
// (1/L) sum_k sigma(2k/L) cos(2 pi k m / L), sigma(z) = exp(-alpha z^p).
#pragma once
#include <algorithm>
#include <cmath>
#include <vector>

#include "fc_internal.h"
#include "fc_split.cuh"
#include "fc_tables.h"

namespace fcx {

// whether lines of continued length L run as contractions: the parts' inner length fits a CTA
inline bool mm_length_ok(int L) { return L >= 16 && ((L % 2 == 0 && L / 2 <= MM_KMAX) || (L % 2 == 1 && L <= MM_KMAX)); }

// FP16 bits of an integer of magnitude below 2048
inline uint16_t mm_half(int v) {
  if (v == 0) return 0;
  const int a = v < 0 ? -v : v;
  int e = 0;
  while ((a >> (e + 1)) != 0) ++e;
  return (uint16_t)((v < 0 ? 0x8000 : 0) | ((e + 15) << 10) | ((a << (10 - e)) & 0x3ff));
}

// balanced base-1024 digits, most significant first
inline void mm_digits(long long q, int* dg) {
  for (int k = SP_DIGITS - 1; k > 0; --k) {
    const long long r = ((q + 512) & 1023) - 512;
    dg[k] = (int)r;
    q = (q - r) / 1024;
  }
  dg[0] = (int)q;
}

// Whether the level sums of one part's digits D[digit][x] stay exact for any data: per level, the
// largest sum over a window of columns between carries (fc_split.cuh; any window of x: a row's
// columns are consecutive entries) of |coefficient digit| times the largest data digit (the first is
// at most 128, 256 for sums of two values), with 2^16 for what carries bring and leave, below 2^24
inline bool mm_sums_exact(const std::vector<int>* D, int S, int H) {
  const int nx = (int)D[0].size();
  const long long B[4] = {128 * S, 512, 512, 512};
  for (int l = 0; l < 4; ++l) {
    const int w = std::min(H, l == 0 ? MM_KCHUNK : (l == 1 ? SP_CARRY2 : SP_CARRY));
    auto at = [&](int x) {
      long long a = 0;
      for (int i = 0; i <= l; ++i) a += std::abs(D[i][x]) * B[l - i];
      return a;
    };
    long long s = 0;
    for (int x = 0; x < nx; ++x) {
      s += at(x) - (x >= w ? at(x - w) : 0);
      if (s + (1 << 16) >= 1 << 24) return false;
    }
  }
  return true;
}

// appends the tables of coefficients c (L values, c(m) = c[m mod L]) to lo / hi (entries
// of digits 0..3 and 4..5) and returns the first entry (-1: their level sums would not be exact); *te: the coefficients were scaled
// by 2^te, which takes the largest to about 2^SP_COEF but leaves the joined sums, and U + V and
// U - V, in 63 bits: with line values below 2^(SP_DATA + 1) each is at most
// sum |c| 2^(te + SP_DATA + 2) units of 2^SP_UNIT. (A broad filter's coefficients are small and
// many, sum |c| about 1: 2^64 or so then, four bits more than the largest of a narrow one gets.)
inline int mm_table(const MmPlan& p, int L, const std::vector<long double>& c, std::vector<uint4>& lo,
                    std::vector<uint2>& hi, int* te) {
  const int H = p.H, S = p.S, nx = p.nx, off = p.Mp;
  auto t = [&](int s, int m) {
    const long double a = c[(size_t)(((m % L) + L) % L)];
    if (S == 1) return a;
    const long double b = c[(size_t)((((m + H) % L) + L) % L)];
    return s ? a - b : a + b;
  };
  long double top = 0, sum = 0;
  for (int s = 0; s < S; ++s)
    for (int m = 0; m < H; ++m) top = std::max(top, std::fabs(t(s, m)));
  for (long double v : c) sum += std::fabs(v);
  *te = SP_COEF;
  if (top > 0)
    *te = std::min(SP_COEF - (int)std::lround(std::log2((double)top)),
                   63 + SP_UNIT - SP_DATA - 2 + (int)std::floor(-0.1 - std::log2((double)sum)));
  std::vector<int> D[2][SP_DIGITS];
  bool exact = false;
  for (int cut = 0; cut < 5 && !exact; ++cut) {  // (broad filters have bits to spare)
    if (cut) --*te;
    exact = true;
    for (int s = 0; s < S; ++s) {
      for (int k = 0; k < SP_DIGITS; ++k) D[s][k].resize(nx + 1);
      for (int x = 0; x <= nx; ++x) {
        int d[SP_DIGITS];
        mm_digits((long long)std::llround(std::ldexp(t(s, off - x), *te)), d);
        for (int k = 0; k < SP_DIGITS; ++k) D[s][k][x] = d[k];
      }
      exact = exact && mm_sums_exact(D[s], S, H);
    }
  }
  if (!exact) return -1;
  const int first = (int)lo.size();
  for (int s = 0; s < S; ++s) {
    auto pair = [&](int k, int x) {
      return (uint32_t)mm_half(D[s][k][x]) | ((uint32_t)mm_half(D[s][k][x + 1]) << 16);
    };
    for (int x = 0; x < nx; ++x) {
      lo.push_back(uint4{pair(0, x), pair(1, x), pair(2, x), pair(3, x)});
      hi.push_back(uint2{pair(4, x), pair(5, x)});
    }
  }
  return first;
}

// MmPlan of length L (mm_length_ok) with its derivative table and, when sig is given
// (sigma(2k/L) >= 0 for k = 0..L/2) and its size is that of FP64 numbers, its filter table
inline MmPlan mm_plan(int L, const std::vector<long double>* sig, std::vector<uint4>& lo, std::vector<uint2>& hi) {
  const long double PI_L = 3.14159265358979323846264338327950288L;
  MmPlan p{};
  p.S = L % 2 == 0 ? 2 : 1;
  p.H = L / p.S;
  p.Kp = (p.H + 15) / 16 * 16;
  p.Mp = p.Kp;
  p.nx = p.Mp + p.Kp;
  // cos(pi j / (2L)), j = 0..2L, which also gives sin(pi m / L) = cos(pi (L - 2m) / (2L))
  const Trig tg(4 * L);
  const std::vector<long double>& cs = tg.c;
  std::vector<long double> c((size_t)L, 0.0L);
  for (int m = 1; 2 * m <= L; ++m) {
    const long double sn = cs[L - 2 * m];  // sin(pi m / L)
    const long double v = (PI_L / L) * (m % 2 ? -1.0L : 1.0L) * (L % 2 == 0 ? cs[2 * m] / sn : 1.0L / sn);
    c[m] = v;
    c[L - m] = -v;
  }
  if (L % 2 == 0) c[L / 2] = 0.0L;
  p.dtab = mm_table(p, L, c, lo, hi, &p.dte);
  p.ftab = -1;
  // 2^(se - 1) < largest sigma <= 2^se
  long double stop = 0;
  bool usable = sig != nullptr;
  if (sig)
    for (long double v : *sig) {
      usable = usable && std::isfinite(v);
      stop = std::max(stop, v);
    }
  int se = 0;
  if (usable && stop > 0 && std::frexp(stop, &se) == 0.5L) --se;
  usable = usable && stop > 0 && std::abs(se) <= 900;
  if (usable) {
    // cosine sums in 128-bit integers (sigma in 2^(se - 58), cosines in 2^-58)
    std::vector<long long> sq((size_t)L / 2 + 1), cq((size_t)L);
    for (int k = 0; 2 * k <= L; ++k) sq[k] = (long long)std::llround(std::ldexp((*sig)[k], 58 - se));
    for (int j = 0; 2 * j <= L; ++j) {
      cq[j] = (long long)std::llround(std::ldexp(cs[4 * j], 58));
      if (j) cq[L - j] = cq[j];
    }
    for (int m = 0; 2 * m <= L; ++m) {
      __int128 a = 0;
      for (int k = 1; 2 * k < L; ++k) a += (__int128)sq[k] * cq[(size_t)((long long)k * m % L)];
      a *= 2;
      a += (__int128)sq[0] * cq[0];
      if (L % 2 == 0) a += (__int128)sq[L / 2] * cq[(size_t)((long long)(L / 2) * m % L)];
      const long double v = std::ldexp((long double)a, se - 116) / L;
      c[m] = v;
      if (m) c[L - m] = v;
    }
    p.ftab = mm_table(p, L, c, lo, hi, &p.fte);
  }
  return p;
}

// The continuation's contraction: ext_k = sum_q M[k][q] e_q over the Q <= 16 detrended end
// values of a line, as digit products of one 16-column step. The columns' coefficients differ
// by four orders of magnitude (second differences 1e4, values 1), so column q carries 2^-sq
// and its value 2^sq. Levels 0 to 3 are exact for any data, as in mm_sums_exact, in the end with
// one bit less of the coefficients (digits up to 512: 16 columns of 3 x 2^18 + 2^16). Fragments of the matrix instruction, 16 rows (continuation points) each:
// [block][digit][lane], a lane's four registers side by side.
inline MmCont mm_continuation(int C, int Q, const std::vector<long double>& M, std::vector<uint4>& lo) {
  MmCont r{};
  r.first = (int)lo.size();
  for (int q = 0; q < Q; ++q) {
    long double top = 0;
    for (int k = 0; k < C; ++k) top = std::max(top, std::fabs(M[(size_t)k * Q + q]));
    int e = 0;
    if (top > 0) std::frexp(top, &e);
    r.sq[q] = e;
  }
  auto digits = [&](int k, int q, int* d) {
    mm_digits((long long)std::llround(std::ldexp(M[(size_t)k * Q + q], SP_COEF - r.sq[q])), d);
  };
  bool exact = true;
  for (int k = 0; k < C; ++k) {
    long long s[4] = {0, 0, 0, 0};
    for (int q = 0; q < Q; ++q) {
      int d[SP_DIGITS];
      digits(k, q, d);
      for (int l = 0; l < 4; ++l)
        for (int i = 0; i <= l; ++i) s[l] += (long long)std::abs(d[i]) * (i == l ? 128 : 512);
    }
    for (int l = 0; l < 4; ++l) exact = exact && s[l] < 1 << 24;
  }
  if (!exact)
    for (int q = 0; q < Q; ++q) ++r.sq[q];
  auto digit = [&](int k, int q, int j) -> uint32_t {
    if (k >= C || q >= Q) return 0;
    int d[SP_DIGITS];
    digits(k, q, d);
    return mm_half(d[j]);
  };
  for (int b = 0; b < (C + 15) / 16; ++b)
    for (int j = 0; j < SP_DIGITS; ++j)
      for (int lane = 0; lane < 32; ++lane) {
        const int g = lane >> 2, t = lane & 3;
        uint32_t a[4];
        for (int i = 0; i < 4; ++i) {
          const int k = 16 * b + g + 8 * (i & 1), q = 2 * t + 8 * (i >> 1);
          a[i] = digit(k, q, j) | (digit(k, q + 1, j) << 16);
        }
        lo.push_back(uint4{a[0], a[1], a[2], a[3]});
      }
  return r;
}

}  // namespace fcx
