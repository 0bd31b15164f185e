// Float64 1/sqrt and 2^-x of the pair kernels, in few operations of the float64 pipe (GB300 has one per
// 64 float32 operations; the conversions between the formats are integer operations here).
#pragma once

namespace pbfb {
namespace {

constexpr int EXP2_TAB = 2048;  // table of 2^(-k / 2048), host-computed (Mesh::pair_tab64)

// 1/sqrt(r2): the hardware's estimate y0 (about 2^-20), e = 1 - r2 y0^2, y0 (1 + e/2 + 3 e^2/8); the
// next term of the series, 5 e^3/16, is below 2^-56.  0 gives a NaN.
__device__ __forceinline__ double rsqrt64(double r2) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(r2));
  const double e = fma(-(r2 * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

// 1/d: the hardware's estimate (about 2^-20) and two Newton steps, y (2 - d y); a d of 0 or below the normal
// numbers gives a non-finite value
__device__ __forceinline__ double rcp64(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  y = fma(y, fma(-d, y, 1.0), y);
  return fma(y, fma(-d, y, 1.0), y);
}

// 2^-x for 0 <= x: 2^-x = 2^-m T[j] 2^-f, x = m + j / 2048 + f with |f| <= 2^-12 (k = 2048 m + j from the
// float32 value of x, the float64 remainder exact), 2^-f = 1 + f (-L + f (L^2/2 - f L^3/6)), L = ln 2
// (truncation 2^-54).  0 once 2^-m leaves the normal numbers.
__device__ __forceinline__ double exp2_neg(double x, const double* __restrict__ tab) {
  // float32 bits of x cut to [2^-60, 1100] (exponent bias 1023 -> 127 modulo 2^32)
  const int xhi = min(max(__double2hiint(x), 0x3C300000), 0x40913000);
  const unsigned xb = __funnelshift_l(__double2loint(x), xhi, 3) - 0xC0000000u;
  const float m = __fmaf_rn(__uint_as_float(xb), 2048.f, 12582912.f);
  const int k = __float_as_int(m) - 0x4B400000;
  const float kf = __fmul_rn(__fsub_rn(m, 12582912.f), 1.f / 2048.f);
  const int kb = __float_as_int(kf);
  // kf as a float64 number (0 becomes 2^-127: far below any rounding here)
  double f = x - __hiloint2double((kb >> 3) + (896 << 20), kb << 29);
  double T = tab[k & (EXP2_TAB - 1)];
  const int e = k / EXP2_TAB;
  T = __hiloint2double(__double2hiint(T) - (e << 20), __double2loint(T));
  if (e > 1020) T = f = 0.0;
  constexpr double L = 0.69314718055994530942;
  return fma(T * f, fma(f, fma(f, -L * L * L / 6.0, 0.5 * L * L), -L), T);
}

// e^a and e^-a for a >= 0: a = (k / 2048) ln 2 + f, |f| <= 1.7e-4 (ln 2 / 2048 in two parts, the first with 30
// bits so that its product with k is exact), e^+-f = 1 + (f^2/2 + f^4/24) +- (f + f^3/6) (truncation 2^-62),
// 2^-+k/2048 from the table.  From 700 on (and for a NaN) the library's exponentials.
__device__ __forceinline__ void exp_pm(double a, const double* __restrict__ tab, double& ep, double& em) {
  if (!(a < 700.0)) {
    ep = exp(a);
    em = exp(-a);
    return;
  }
  const int ahi = max(__double2hiint(a), 0x3C300000);
  const unsigned ab = __funnelshift_l(__double2loint(a), ahi, 3) - 0xC0000000u;  // float32 bits of max(a, 2^-60)
  const float m = __fmaf_rn(__uint_as_float(ab), 2954.6394f, 12582912.f);  // 2048 / ln 2
  const int k = __float_as_int(m) - 0x4B400000;
  const int kb = __float_as_int(__fsub_rn(m, 12582912.f));
  const double kd = __hiloint2double((kb >> 3) + (896 << 20), kb << 29);  // k (0 becomes 2^-127)
  constexpr double C1 = 0x1.62e42fe8p-12, C2 = 4.3423507025813853e-13;  // ln 2 / 2048 = C1 + C2
  const double f = fma(-kd, C2, fma(-kd, C1, a)), s = f * f;
  const double even = s * fma(s, 1.0 / 24.0, 0.5), odd = f * fma(s, 1.0 / 6.0, 1.0);
  const int e = k / EXP2_TAB, j = k & (EXP2_TAB - 1);
  const double tm = tab[j], tp = tab[(EXP2_TAB - j) & (EXP2_TAB - 1)];  // 2^-j/2048; 2^(j/2048 - 1), or 1 for j = 0
  const double Tm = __hiloint2double(__double2hiint(tm) - (e << 20), __double2loint(tm));
  const double Tp = __hiloint2double(__double2hiint(tp) + ((e + (j != 0)) << 20), __double2loint(tp));
  ep = fma(Tp, even + odd, Tp);
  em = fma(Tm, even - odd, Tm);
}

}  // namespace
}  // namespace pbfb
