// |p|^beta and |p|^gamma of the constitutive law in 64-bit integer arithmetic.
//
// GB300 issues two FP64 operations per SM and clock but 64 integer multiply-adds, so
// the log and the two exponentials of the law, about 60 FP64 instructions through
// log()/exp(), are evaluated in fixed point on the otherwise idle integer pipe and cost
// no FP64 operation at all: the constitutive pass of 2.1M cells went from 370 to 94 us.
// Method: table-driven logarithm and exponential (P. T. P. Tang, ACM TOMS 15 (1989) and
// 16 (1990)) with 256-entry tables and short series, carried out in fixed point:
//   x = 2^e m;  r = m c_i - 1 with c_i ~ 1/m (table), |r| <= 2^-9, exact to 2^-71;
//   y = log2 x = e - log2 c_i + log2(1 + r), 57 fractional bits;
//   t = b y, 64 fractional bits kept;  x^b = 2^floor(t) 2^(j/256) 2^f, f < 2^-8.
// The relative error of x^b is at most 2^-53 (the final rounding) + 1.1 b 2^-57 (the 1.5
// units of y's last place, times b ln 2) + 2^-58: 1.4 x 2^-53 for the paper's exponents
// (exp(b log x) loses about |b log x| / 2 ulp).  Domain: x in [2^-30, 2^30), 0 < b < 32;
// the callers take pow() outside.
#pragma once

#include <stdint.h>

#include "pow_tables.cuh"

namespace rich {

constexpr int kFixPowExp = 30;       // |binary exponent| of the domain
constexpr double kFixPowMaxB = 32.0; // exponents below this

// An exponent b in (0, 32) as 2^58 b (host side, once per context).
inline unsigned long long fixpow_exponent(double b) {
  if (!(b > 0.0 && b < kFixPowMaxB)) return 0;  // 0: not representable, the callers take pow()
  return (unsigned long long)(b * 288230376151711744.0 + 0.5);
}

// 2^57 log2(x) of a positive double given by its bits, binary exponent in [-30, 29].
__device__ __forceinline__ long long fixpow_log2(unsigned long long bits) {
  const int e = (int)(bits >> 52) - 1023;
  const int i = (int)(bits >> 44) & 255;
  const unsigned long long M = (bits | 0x0010000000000000ull) << 11;  // m 2^63
  const unsigned C = __ldg(&kPowRcp[i]);
  const unsigned long long lo = (unsigned long long)(unsigned)M * C;
  const unsigned long long hi = (M >> 32) * C + (lo >> 32);  // m c 2^63
  const long long R = (long long)((hi - 0x8000000000000000ull) << 8 | (unsigned)lo >> 24);  // r 2^71
  const int r = (int)(R >> 32);  // r 2^39
  // log2(1 + r) = r (k1 - r (k2 - r (k3 - r (k4 - r (k5 - r k6))))), k_j = 1 / (j ln 2)
  const int k6 = 0x1ec709dc, k5 = 0x24eed8a2, k4 = 0x2e2a8eca;  // 2^31 k_j
  const int w = k5 - (__mulhi(r, k6) >> 7);
  const int v = k4 - (__mulhi(r, w) >> 7);
  const long long u = 0x3d8e13b87407fae9ll - (((long long)r * v) >> 7);                // 2^63 (k3 - ...)
  const long long s = 0x5c551d94ae0bf85ell - (__mul64hi(R, u) >> 7);                   // 2^63 (k2 - ...)
  const long long p = 0x5c551d94ae0bf85ell - (__mul64hi(R, s) >> 8);                   // 2^62 (k1 - ...)
  return ((long long)e << 57) + (long long)__ldg(&kPowLog[i]) + (__mul64hi(R, p) >> 12);
}

// 2^(b y) for y = 2^57 log2 x and b = 2^58 b, as a double (|b y| < 1000).
__device__ __forceinline__ double fixpow_exp2(long long y, unsigned long long b) {
  const long long hi = __mul64hi(y, (long long)b);  // the product has 115 fractional bits
  const unsigned long long lo = (unsigned long long)y * b;
  const int n = (int)(hi >> 51);
  const unsigned long long f = (unsigned long long)hi << 13 | lo >> 51;
  const unsigned long long E = __ldg(&kPowExp[f >> 56]);
  const unsigned long long phi = f << 8;  // 2^64 (256 x), x the remaining fraction
  const unsigned ph = (unsigned)(phi >> 32);
  // 2^x - 1 = x (l1 + x (l2 + x (l3 + x (l4 + x l5)))), l_j = (ln 2)^j / j!
  const unsigned a4 = 2581847u + __umulhi(ph, 1398u);
  const unsigned a3 = 3814213304u + __umulhi(ph, a4);                                          // 2^52
  const unsigned long long a2 = 0x003d7f7bff058b1dull + ((unsigned long long)ph * a3 >> 20);   // 2^64
  const unsigned long long a1 = 0xb17217f7d1cf79acull + __umul64hi(phi, a2);                   // 2^64
  const unsigned long long m = E + __umul64hi(E, __umul64hi(phi, a1) >> 8);                    // 2^63 [1, 2)
  const unsigned long long bits = ((unsigned long long)(unsigned)(n + 1022) << 52) + (m >> 11) + ((m >> 10) & 1);
  return __longlong_as_double((long long)bits);
}

// 1/q for a normal q well inside the exponent range.  With x within 2^-19 of 1/q and
// e = 1 - q x, 1/q = x / (1 - e) = x (1 + e + e^2 + ...): one step of the cubically convergent
// iteration x (1 + e + e^2) (M. Altman, Pacific J. Math. 10 (1960) 1107) from the machine's
// reciprocal of q's leading 20 bits.  What is cut off is below 2^-57, e is exact to
// 2^-53 |e|, and the last multiply-add rounds once: relative error at most 2^-53 (1 + 2^-3),
// below 1 ulp.  Three FP64 operations, on a pipe that a correctly rounded division would
// hold several times as long.
__device__ __forceinline__ double fast_rcp(double q) {
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(q));
  const double e = fma(-q, x, 1.0);
  return fma(x, fma(e, e, e), x);
}

}  // namespace rich
