// Integer conversions of the emulated FP64 products: the emulated GEMM
// (ozaki_gemm.cu) and the task-graph leaves' 32 x 32 tile products
// (potrf_dag.cu).
#pragma once

#include <cstdint>

namespace bta {
namespace oz {

// Conversions between FP32 and 32-bit integers of magnitude below 2^22 by
// FP32 arithmetic against 1.5 2^23 (the FP32 adder's round to nearest even,
// exact for integers): one add and one integer operation each, on the
// full-rate pipes instead of the conversion unit.
__device__ __forceinline__ int f2i_small(float x) {
  return __float_as_int(x + 12582912.0f) - 0x4B400000;
}
__device__ __forceinline__ float i2f_small(int d) {
  return __int_as_float(d + 0x4B400000) - 12582912.0f;
}

// u * 2^E (negated if neg) rounded to the nearest double, from the integer u > 0 by
// integer operations (the usual case); out-of-range exponents take ldexp.
__device__ __forceinline__ double compose_mag(bool neg, unsigned long long u, int E) {
  int lz = __clzll((long long)u);
  const unsigned long long mag = u;
  u <<= lz;                                   // leading one at bit 63
  unsigned long long m = u >> 11;             // 53 significant bits
  const unsigned long long rem = u & 0x7FFull;
  if (rem > 0x400ull || (rem == 0x400ull && (m & 1ull))) {
    ++m;
    if (m >> 53) { m >>= 1; --lz; }
  }
  const int be = 1023 + (63 - lz) + E;
  if (be <= 0 || be >= 2047) return ldexp(neg ? -(double)mag : (double)mag, E);
  return __longlong_as_double((long long)((neg ? 1ull << 63 : 0ull) |
                                          ((unsigned long long)be << 52) |
                                          (m & ((1ull << 52) - 1))));
}

// X * 2^E rounded to the nearest double.
__device__ __forceinline__ double compose(long long X, int E) {
  if (X == 0) return 0.0;
  return compose_mag(X < 0, X < 0 ? 0ull - (unsigned long long)X : (unsigned long long)X, E);
}

// The 8 signed base-128 digits of v for the row exponent bound er, as integers
// in FP32 (|d_0| <= 128, |d_j| <= 64 otherwise): v = sum_j d_j 2^(er - 1029 - 7 j).
__device__ __forceinline__ void digits(double v, int er, float (&out)[8]) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(v);
  const int E = (int)((bits >> 52) & 0x7FF);
  long long F = 0;   // v 2^(1078 - er): |F| < 2^56
  if (E != 0) {
    const unsigned long long mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const int sh = E - er + 3;   // <= 3
    if (sh >= 0) {
      F = (long long)(mant << sh);
    } else if (sh > -54) {
      F = (long long)((mant + (1ull << (-sh - 1))) >> (-sh));
    }
    if (bits >> 63) F = -F;
  }
  // F = G 2^28 + R, R in [-2^27, 2^27): digits 0..3 from G, 4..7 from R,
  // each taken with round-half-up so that every remainder stays within
  // half a digit; 32-bit arithmetic
  const int G0 = (int)((F + (1ll << 27)) >> 28);
  const int parts[2] = {G0, (int)(F - (long long)G0 * (1ll << 28))};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    int x = parts[h];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int sh = 21 - 7 * j;
      const int d = j < 3 ? (x + (1 << (sh - 1))) >> sh : x;
      x -= d * (1 << sh);
      out[4 * h + j] = i2f_small(d);
    }
  }
}

}  // namespace oz
}  // namespace bta
