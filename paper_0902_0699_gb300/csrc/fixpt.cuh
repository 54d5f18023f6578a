// binary64 <-> 64-bit fixed point with a common exponent per tile (wht.cu), column
// (the register QFT of tile.cu) or row (rho_tc128.cu): sums are exact integer
// additions and no FP64 instruction is issued.  And a sum of FP64 terms in two
// words of fixed point, which does not depend on their order (adjoint.cu).
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define FX_HD __host__ __device__ __forceinline__
#else
#define FX_HD inline
#endif

namespace qc {

// One of many terms of a sum that is kept in two 64-bit integers:
// x = hi + lo 2^-FX_LOW to half a unit of lo.  |lo| <= 2^(FX_LOW - 1), so the
// low words of 2^27 terms add up without overflow, whatever their fractions
// (2^52 for 2^-FX_LOW would leave room for 2^12 equal ones).
constexpr int FX_LOW = 36;
FX_HD void fx_split(double x, long long& hi, long long& lo) {
  const double r = rint(x);
  hi = (long long)r;
  lo = (long long)rint((x - r) * (double)(1ll << FX_LOW));
}
FX_HD double fx_join(long long hi, long long lo) { return (double)hi + (double)lo * (1.0 / (double)(1ll << FX_LOW)); }

#ifdef __CUDACC__

// binary64 -> fixed point round(x 2^(1075 - G)) for a tile's G,
// rounding half away from zero (symmetric, so unbiased; exact
// values need no rounding at all).  x = m 2^(ex - 1075), so the value is
// m 2^(ex - G).  Numbers below 2^-1022 are dropped, or kept with SUBNORMAL.
template <bool SUBNORMAL = false>
__device__ __forceinline__ long long d2fix(double x, int G) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7FFu);
  if (!SUBNORMAL && ex == 0) return 0;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (ex ? 1ull << 52 : 0ull);
  if (SUBNORMAL) ex = max(ex, 1);
  const int sh = ex - G;
  unsigned long long v;
  if (sh >= 0) {
    v = m << sh;  // sh <= 9 - |B|: no overflow
  } else {
    const int r = -sh;
    v = r > 54 ? 0ull : ((m >> (r - 1)) + 1ull) >> 1;
  }
  return (b >> 63) ? -(long long)v : (long long)v;
}

// fixed point v 2^-F -> binary64, rounded half away from zero (results
// below 2^-1022 flush to zero, or are kept with SUBNORMAL)
template <bool SUBNORMAL = false>
__device__ __forceinline__ double fix2d(long long v, int F) {
  if (v == 0) return 0.0;
  const unsigned long long sgn = v < 0 ? (1ull << 63) : 0ull;
  const unsigned long long a = v < 0 ? (unsigned long long)(-v) : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  unsigned long long keep = (((a << lz) >> 10) + 1ull) >> 1;  // 53 bits, rounded
  int e = 63 - lz - F + 1023;
  if (keep >> 53) {
    keep >>= 1;
    ++e;
  }
  if (SUBNORMAL && e <= 0) {  // a 2^-F in units of 2^-1074: below 2^52 of them
    const int r = F - 1074;
    const unsigned long long m = r > 63 ? 0ull : r > 0 ? ((a >> (r - 1)) + 1ull) >> 1 : a << -r;
    return __longlong_as_double((long long)(sgn | m));
  }
  if (e <= 0) return __longlong_as_double((long long)sgn);
  if (e >= 2047) return __longlong_as_double((long long)(sgn | (0x7FFull << 52)));
  return __longlong_as_double((long long)(sgn | ((unsigned long long)e << 52) | (keep & 0xFFFFFFFFFFFFFull)));
}

#endif  // __CUDACC__

}  // namespace qc
