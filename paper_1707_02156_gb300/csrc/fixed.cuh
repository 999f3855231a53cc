// Sums of products in fixed point on the integer pipe, for set-up contractions whose operation count the FP64
// pipe bounds: GB300 does 1.7 FP64 multiply-adds per clock and SM, and 30 of the 32 x 32 + 64 bit integer
// ones.  A value is scaled by a power of two common to the sum's operands, rounded to an integer of at most 57
// bits (tables: 58) and split into a high and a centred low part of 29 bits; a product is then
//   (a_h 2^29 + a_l)(b_h 2^29 + b_l) = a_h b_h 2^58 + (a_h b_l + a_l b_h) 2^29 + a_l b_l,
// whose first two terms are accumulated exactly in two 64-bit sums (three multiply-adds a product; both sums of up
// to 63 products stay below 2^63) and whose last one is left out.  Operands within 2^-4 of the largest are exact,
// smaller ones and a left-out term are good to 2^-58 of the largest product, so that a sum of K products errs by
// about 2^-58 sqrt(K) of it, where FP64 sums round every addition to 2^-53 of the running sum.  (With 54 bits
// and parts of 28, the many small coefficients of a smooth drop added up to errors 15 to 40 % above FP64's.)
#pragma once
#include <cuda_runtime.h>

namespace bie {

constexpr int kFixPart = 29;  // bits of the low part

// v 2^(57 - e) as an integer, rounded to nearest; |v| < 2^(e + 4)
__device__ __forceinline__ long long fix_encode(double v, int e) {
  const long long b = __double_as_longlong(v);
  const int ex = (int)(b >> 52) & 0x7ff;
  const int s = ex - 1018 - e;  // v = m 2^(ex - 1075)
  if (ex == 0 || s < -54) return 0;
  const long long m = (b & 0xfffffffffffffLL) | (1LL << 52);
  const long long f = s >= 0 ? m << s : (m + (1LL << (-s - 1))) >> -s;
  return b < 0 ? -f : f;
}
// the two parts of an integer
__host__ __device__ __forceinline__ int2 fix_split(long long f) {
  const int h = (int)((f + (1LL << (kFixPart - 1))) >> kFixPart);
  return make_int2(h, (int)(f - ((long long)h << kFixPart)));
}
// accumulates a b into the sums of high (h) and cross (x) products
__device__ __forceinline__ void fix_mad(long long& h, long long& x, int2 a, int2 b) {
  h += (long long)a.x * b.x;
  x += (long long)a.x * b.y;
  x += (long long)a.y * b.x;
}
// (h + x 2^-29) 2^extra as an integer, 0 <= extra < 29: the sum in units of 2^(58 - extra) of its products'; half of it
__device__ __forceinline__ long long fix_half(long long h, long long x) { return (h + (x >> kFixPart) + 1) >> 1; }
__device__ __forceinline__ long long fix_sum(long long h, long long x, int extra) {
  return (h << extra) + ((x + (1LL << (kFixPart - 1 - extra))) >> (kFixPart - extra));
}
// r 2^u; zero below the normal numbers, infinite above the largest
__device__ __forceinline__ double fix_decode(long long r, int u) {
  const double d = __ll2double_rn(r);
  const int hi = __double2hiint(d), ex = (hi >> 20 & 0x7ff) + u;
  if (r == 0 || ex <= 0) return 0.0;
  if (ex >= 0x7ff) return __hiloint2double((hi & (int)0x80000000) | 0x7ff00000, 0);
  return __hiloint2double((int)((unsigned)hi + ((unsigned)u << 20)), __double2loint(d));
}
// Exponents over a set of values: the largest fix_magnitude of them gives the smallest e with |v| < 2^e for all, or
// fix_none if all are zero (or below the normal range) and fix_bad with a NaN or an infinity among them.
constexpr int fix_none = -4000, fix_bad = 4000;
__device__ __forceinline__ int fix_magnitude(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ int fix_exponent(int magnitude) {
  const int ex = magnitude >> 20;
  return ex == 0x7ff ? fix_bad : ex == 0 ? fix_none : ex - 1022;
}
__host__ __device__ constexpr int ceil_log2(int n) {
  int b = 0;
  while ((1 << b) < n) ++b;
  return b;
}

}  // namespace bie
