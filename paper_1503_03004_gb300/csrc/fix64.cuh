// Float64 dot products on the integer units.
//
// GB300 issues float64 FMA at about 2 per clock per SM (1.9 measured), but 32 x 32 + 64 -> 64 bit
// integer multiply-adds at about 30 per clock (29 measured).  The float64 path
// therefore forms its inner products in fixed point, an error-free split of each operand into
// integer slices whose products are accumulated exactly (the Ozaki scheme: Ozaki, Ogita, Oishi and
// Rump, "Error-free transformations of matrix multiplication", Numer. Algorithms 59, 2012; here two
// 28-bit slices and 64-bit integer accumulators instead of short floating-point slices):
//   * the entries of an operand that meet in one sum share one exponent e, with |x| < 2^e for all of them;
//   * x 2^(56-e) is rounded to an integer F, |F| <= 2^56, held as F = hi 2^28 + lo with
//     |hi| <= 2^28, -2^27 <= lo < 2^27;
//   * x y 2^(112 - e_x - e_y) = hi hi' 2^56 + (hi lo' + lo hi') 2^28 + lo lo', and the last term,
//     at most 2^54, is dropped: three multiply-adds per product.
// Sums over at most kTerms = 64 products cannot overflow (64 2^56 = 2^62, 128 2^55 = 2^62), and they
// are exact, so they do not depend on the order of the terms.  Errors per product, relative to the
// bound 2^(e_x + e_y): 2^-57 for each operand's rounding and 2^-58 for the dropped term, against
// 2^-54 for the rounding of a float64 operation at that size.
//
// What shares an exponent is therefore a row of the left operand and a column of the right one (the
// entries of one sum), never a block of rows or columns of different size: a row 1e10 times smaller than its
// neighbour keeps its 56 bits.  A factor common to a column of the left operand, as in P T with
// T = B (B G B)^{-1/2}, is taken out of it and put into the row of the right one first (a power of two).
// Only the operands that are bounded alike throughout, the orthonormal U and V in sums over their rows, have
// one exponent per 64 rows.
#pragma once

#include <cuda_runtime.h>

#include <cstring>

namespace sfr {
namespace fx {

constexpr int kTerms = 64;
constexpr int kBad = 1 << 16;  // exponent of a block with a non-finite entry: its products become NaN
constexpr int kZero = -4096;   // exponent of zeros where exponents are added (below every sum of two others)

// Exponent e with |x| < 2^e, from the upper word of the largest |x| (zero and subnormal: -1022).
__host__ __device__ inline int exponent(int hi_word) {
  const int ex = (hi_word & 0x7fffffff) >> 20;
  return ex == 0x7ff ? kBad : ex - 1022;
}

// The same for one finite value, with kZero for zero (and what is below 2^-1042).
__host__ __device__ inline int value_exponent(int hi_word) {
  const int h = hi_word & 0x7fffffff;
  return h ? (h >> 20) - 1022 : kZero;
}

// x in the fixed point of exponent e (|x| < 2^e, rounded to nearest): .x = hi, .y = lo.
__host__ __device__ inline int2 to_fix(double x, int e) {
  long long b;
#ifdef __CUDA_ARCH__
  b = __double_as_longlong(x);
#else
  std::memcpy(&b, &x, sizeof b);
#endif
  int ex = (int)((b >> 52) & 0x7ff);
  unsigned long long mant = (unsigned long long)b & 0xfffffffffffffULL;
  if (ex) mant |= 1ULL << 52; else ex = 1;
  const int s = 1019 + e - ex;  // F = mant 2^-s, s >= -3
  unsigned long long f = 0;
  if (s <= 0) f = s >= -4 ? mant << -s : 0;  // (not finite: 0)
  else if (s < 64) f = ((mant >> (s - 1)) + 1) >> 1;
  const long long F = b < 0 ? -(long long)f : (long long)f;
  int2 r;
  r.x = (int)((F + (1LL << 27)) >> 28);
  r.y = (int)(F - ((long long)r.x << 28));
  return r;
}

// 2^k (NaN for the exponent sum of a kBad block).
__host__ __device__ inline double pow2(int k) {
  long long b;
  if (k > kBad / 2) b = 0x7ff8000000000000LL;
  else if (k > 1023) b = 0x7ff0000000000000LL;
  else if (k >= -1022) b = (long long)(k + 1023) << 52;
  else b = k < -1074 ? 0 : 1LL << (k + 1074);
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double d;
  std::memcpy(&d, &b, sizeof d);
  return d;
#endif
}

// One product added to the accumulators: hh += hi hi', cx += hi lo' + lo hi'.
__host__ __device__ inline void mac(const int2& a, const int2& b, long long& hh, long long& cx) {
  hh += (long long)a.x * b.x;
  cx += (long long)a.x * b.y + (long long)a.y * b.x;
}

template <int X, int Y>
__host__ __device__ inline void mac_block(const int2 (&a)[X], const int2 (&b)[Y], long long (&hh)[X][Y],
                                          long long (&cx)[X][Y]) {
#pragma unroll
  for (int x = 0; x < X; ++x)
#pragma unroll
    for (int y = 0; y < Y; ++y) mac(a[x], b[y], hh[x][y], cx[x][y]);
}

// The accumulated sum in units of 2^(e_x + e_y - 56).
__host__ __device__ inline long long total(long long hh, long long cx) { return hh + ((cx + (1LL << 27)) >> 28); }

// A scale pair for a block pair: the sum T stands for T 2^(e - 56), e = e_x + e_y, formed as
// upper32(T) c1 + lower32(T) c2 in float64.
struct Scale {
  double c1, c2;
  __host__ __device__ explicit Scale(int e) : c1(pow2(e - 24)), c2(pow2(e - 56)) {}
};

// y + T scaled (two float64 operations, each product exact).
__host__ __device__ inline double add_total(long long T, const Scale& s, double y) {
  const double h = (double)(int)(T >> 32), l = (double)(unsigned)T;
#ifdef __CUDA_ARCH__
  return fma(h, s.c1, fma(l, s.c2, y));
#else
  return h * s.c1 + (l * s.c2 + y);
#endif
}

}  // namespace fx
}  // namespace sfr
