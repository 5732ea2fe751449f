// rcp64.cuh -- reciprocal of a pivot in FP64 without the FP64 pipe.
#pragma once

#include "common.cuh"

namespace jmg {

// 1 / d for normal d > 0 with a normal result, to within 0.501 ulp, on the integer
// pipe (an FP64 division holds the FP64 pipe for several hundred clocks).  With
// x = m / 2 in [1/2, 1) from the significand m and a 24-bit y0 ~ 1 / x from the
// FP32 reciprocal, e = 1 - x y0 is formed exactly enough in 64-bit fixed point
// (|e| < 2^-22) and 1 / x = y0 (1 + e + e^2) up to e^3 < 2^-66.
JMG_DEV double rcp_fixed(double d) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(d);
  const int ex = (int)(b >> 52);
  const unsigned long long m = (b & ((1ull << 52) - 1)) | (1ull << 52), X = m << 11;
  const unsigned xh = (unsigned)(X >> 32), xl = (unsigned)X;
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint2float_rn(xh) * 0x1p-32f));
  const unsigned Y0 = __float2uint_rz(y * 0x1p31f);
  const unsigned long long P = (unsigned long long)xh * Y0 + __umulhi(xl, Y0);
  const long long E = (long long)((1ull << 63) - P);  // e 2^63
  const int Es = (int)(E >> 20);
  const long long F = E + (((long long)Es * Es) >> 23);
  const unsigned long long R = ((unsigned long long)Y0 << 32) +
                               (unsigned long long)(2 * (long long)Y0 * (int)(F >> 32)) +
                               (((unsigned long long)Y0 * (unsigned)F) >> 31);
  unsigned long long o =
      ((unsigned long long)(2045 - ex) << 52) + (((R >> 10) + 1) >> 1) - (1ull << 52);
  if (m == (1ull << 52)) o = (unsigned long long)(2046 - ex) << 52;  // 1 / 2^k
  return __longlong_as_double((long long)o);
}
// 1 / pivot; *bad when d is not positive (or NaN)
JMG_DEV double pivot_rcp(double d, bool* bad) {
  const int ex = (__double2hiint(d) >> 20);  // sign and exponent
  if (ex >= 1 && ex <= 2044) return rcp_fixed(d);
  *bad = !(d > 0.0);
  return 1.0 / d;
}

}  // namespace jmg
