// Exact split-integer arithmetic of the tensor-core line contractions (fc_mma.cu).
//
// An FC line operator (derivative or filter of the continued line, eqs. fc_der and
// filtering) is a circulant of length L: y_i = sum_j c(i - j) x_j. Data and coefficients
// are held as fixed-point integers of 60 bits, cut into six balanced base-1024 digits in
// [-512, 511]. A digit is exact in FP16, and the FP16 matrix instruction with FP32
// accumulation adds digit products without rounding while their sums stay below 2^24. The
// products of equal weight (levels i + j = 0..5, 21 of the 36 pairs) share an accumulator.
// Levels 0 to 3 are exact for any data: level 3 hands what exceeds a digit to level 2, and 2
// to 1, every 32 columns, level 1 to 0 every 64 (sp_carries), and a table is used only if its
// digits keep these levels below 2^24 between the carries (mm_sums_exact in fc_mmtab.h: at most
// 2^23.95 for the derivative and the default filter). Levels 4 and 5, which weigh 2^-56 and 2^-66
// of the result's scale, stay below 2^24 for typical data and can reach 2^25.2 and 2^27.4 for data
// whose digits all carry the signs of one row's coefficients; rounding their sums then costs up
// to 2^-48 of that scale (an FP64 transform: 2^-50). The levels are joined in 64-bit integers.
// The dropped levels and the truncation of the data leave an error of a few 2^-57 of the line's
// largest value times the operator's largest coefficient, below the rounding of an FP64
// transform of the same line.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "fc_internal.h"

#ifndef FC_HD
#define FC_HD __host__ __device__ __forceinline__
#endif

namespace fcx {

constexpr int SP_DIGITS = 6;     // digits per value = accumulation levels
constexpr int SP_BITS = 10;      // bits per digit
constexpr int SP_DATA = 56;      // a line's data are scaled so that its largest value lies in [2^56, 2^57)
constexpr int SP_COEF = 60;      // coefficients: the largest is scaled into [2^59.5, 2^60.5], or lower (mm_table)
constexpr int SP_UNIT = 60;      // unit of the joined sums: 2^60 of data x coefficient units
// 512 in every digit position: turns balanced digits into plain bit fields
constexpr long long SP_BIAS = (512ll << 50) | (512ll << 40) | (512ll << 30) | (512ll << 20) | (512ll << 10) | 512ll;

FC_HD uint32_t sp_hi(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2hiint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)(b >> 32);
#endif
}
FC_HD uint32_t sp_lo(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2loint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)b;
#endif
}

// x as a fixed-point integer in units 2^(ex - 1023 - SP_DATA), ex the biased exponent of
// the line's largest magnitude (rounded down; zero and subnormal values are 0)
FC_HD long long sp_fixed(double x, int ex) {
  const uint32_t hi = sp_hi(x), lo = sp_lo(x);
  const int e = (int)((hi >> 20) & 0x7ffu);
  const int d = ex - e;
  if (e == 0 || d > 62 || d < 0) return 0;  // d < 0 only for a non-finite line (its outputs are NaN)
  const long long m = (long long)(((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << (SP_DATA - 52);
  return ((hi >> 31) ? -m : m) >> d;
}

// digit pair: the base-1024 digits number k (0 = most significant) of two biased values,
// as two FP16 integers in one word
FC_HD uint32_t sp_field(long long biased, int k) { return (uint32_t)(biased >> (SP_BITS * (SP_DIGITS - 1 - k))) & 1023u; }

// the multiple of 2^SP_BITS nearest to lo goes over to hi, the next higher level (|lo| < 2^31;
// four FP32 operations, on a pipe that the contraction does not use otherwise)
FC_HD void sp_carry(float& hi, float& lo) {
  const float c = fmaf(lo, 1.f / (1 << SP_BITS), 12582912.f) - 12582912.f;  // 1.5 2^23: rounds to an integer
  lo = fmaf(c, -(float)(1 << SP_BITS), lo);
  hi += c;
}
// columns between carries out of levels 2 and 3, and out of levels 1 and 4
constexpr int SP_CARRY = 32, SP_CARRY2 = 64;
// carries of the level sums s[level][0..N-1] after the 16 columns from k0 of n that are summed before the
// join (which needs none), higher levels first: they do not wait for one another. Measured against
// none: step of a 28M-point array 69.3 -> 70.0 ms, operator of a 128 x 128 box (L = 155) 22.8 -> 23.4 us,
// of a 509 x 333 box 113.1 -> 110.6 us (level 4 every 32 columns as well: half a percent more).
template <int N>
FC_HD void sp_carries(float (&s)[SP_DIGITS][N], int k0, int n) {
  if ((k0 & (SP_CARRY - 16)) == 0 || k0 + 16 >= n) return;
  const bool both = (k0 & (SP_CARRY2 - 16)) == SP_CARRY2 - 16;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int q = 0; q < N; ++q) {
    if (both) sp_carry(s[0][q], s[1][q]);
    sp_carry(s[1][q], s[2][q]);
    sp_carry(s[2][q], s[3][q]);
    if (both) sp_carry(s[3][q], s[4][q]);
  }
}

// joined sum of the six level sums (integers below 2^28) in units 2^SP_UNIT
FC_HD long long sp_join(const int* s) {
  const long long hi = ((long long)s[0] << 20) + ((long long)s[1] << 10) + s[2];
  const long long lo = ((long long)s[3] << 20) + ((long long)s[4] << 10) + s[5];
  return (hi << (80 - SP_UNIT)) + (lo >> (SP_UNIT - 50));
}

// a 64-bit integer as a double, rounded to nearest (ties away from zero), without the FP64 pipe
FC_HD double sp_double(long long v) {
  const uint64_t a = v < 0 ? (uint64_t)(-v) : (uint64_t)v;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  const uint64_t m = a << (lz & 63);
  uint64_t b = ((uint64_t)(1085 - lz) << 52) + (m >> 11) + ((m >> 10) & 1u);
  b = a ? b : 0;
  b |= (uint64_t)v & 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double r;
  memcpy(&r, &b, 8);
  return r;
#endif
}

// v 2^e as a double, without the FP64 pipe while the result is a normal number; else by the
// multiplication with fac = 2^e (NaN for a non-finite line, with e out of every range)
FC_HD double sp_double_exp(long long v, int e, double fac) {
  const uint64_t a = v < 0 ? (uint64_t)(-v) : (uint64_t)v;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  const int x = 1085 - lz + e;  // biased exponent - 1
  if ((unsigned)(x - 1) >= 2040u) return sp_double(v) * fac;
  const uint64_t m = a << (lz & 63);
  uint64_t b = ((uint64_t)x << 52) + (m >> 11) + ((m >> 10) & 1u);
  b = a ? b : 0;
  b |= (uint64_t)v & 0x8000000000000000ull;
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double r;
  memcpy(&r, &b, 8);
  return r;
#endif
}

// The FP64 quotient df / rg rounded to FP32 (0 <= df <= rg, both finite, r = 1 / rg rounded):
// t = df r is within 2.5 ulp of the rounded quotient and rounds to the same FP32 number
// unless its low 29 bits lie that close to the midpoint of two FP32 numbers, where the
// division itself decides (as it does for quotients below 2^-100). The rounding runs on the
// bit pattern: conversions, too, occupy the FP64 pipe.
FC_HD float quotient_f32(double df, double rg, double r) {
  const double t = df * r;
  const uint32_t hi = sp_hi(t), lo = sp_lo(t);
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  const int low = (int)(lo & 0x1fffffffu) - 0x10000000;
  const uint32_t f = (uint32_t)((b >> 29) + ((b >> 28) & 1u)) - (896u << 23);
  float x;
#ifdef __CUDA_ARCH__
  x = __uint_as_float(f);
#else
  memcpy(&x, &f, 4);
#endif
  if (b == 0)
    x = 0.f;
  else if ((low >= -4 && low <= 4) || (hi >> 20) < 1023u - 100u)
    x = (float)(df / rg);
  return x;
}

}  // namespace fcx
