// Elementary functions of the FP64 flux kernels: reciprocal, reciprocal square root, and the pair
// (erfc(y)/2, exp(-y^2)) of a half-space Maxwellian.
//
// GB300 issues 2 FP64 operations per clock and SM (conversions between double and the other types
// count as FP64 operations too), against 64 to 128 integer and FP32 ones, so what these functions cost
// is their FP64 operations.  Measured on GB300 against a chain of multiply-adds, CUDA's 1/x takes
// 5.6 of them, rsqrt 5, exp 16 and erfc 60; here the reciprocal takes 3 and exp with erfc together 22, the
// rest of each being integer and FP32 work on the idle pipes (rsqrt is CUDA's: a cubic correction of the
// hardware's approximation takes 5 as well, and the residuals of 576 to 1.51 M cells the same time):
//  - reciprocal: the hardware's approximation (20 bits) and one cubic step of Householder's method (A. S.
//    Householder, The Numerical Treatment of a Single Nonlinear Equation, 1970), r (1 + e + e^2) with
//    e = 1 - x r, whose remainder e^3 is below 2^-55;
//  - exp(-a^2) table-driven (P. T. P. Tang, ACM TOMS 15, 1989): a^2 = (n ln 2)/64 + r with n found in
//    FP32, 2^(-n/64) from a table of 64 and the Taylor polynomial of exp(-r), |r| <= ln 2/128; a^2 is
//    never rounded, the reduction is one fused multiply-add;
//  - erfc(a) = exp(-a^2) R(a), a >= 0: R = exp(a^2) erfc(a) by its Taylor polynomial of degree 8 about
//    the nearest multiple of 1/32 (the remainder is below 2^-58 of R), coefficients from the table
//    that the context builds (half_table_fill, from the derivative recurrence of R).
// Arguments |y| >= 6 (normal Mach numbers above 7; erfc below 2e-17) and NaN take CUDA's functions.
#pragma once
#include <cmath>

#include "internal.cuh"

#define HALF_STEPS 32                              // table points per unit of a
#define HALF_MAX 6                                 // the table covers [0, 6]
#define HALF_ROW 10                                // point, 9 coefficients
#define HALF_ROWS (HALF_STEPS * HALF_MAX + 1)
#define HALF_EXP (HALF_ROWS * HALF_ROW)            // offset of the 64 powers 2^(-i/64)
#define HALF_TABLE (HALF_EXP + 64)

// the table of half_gauss on the host: rows (a_j, c_0 .. c_8) with R(a_j + d)/2 = sum c_n d^n.
// R' = 2 a R - 2/sqrt(pi), so R^(n+1) = 2 a R^(n) + 2 n R^(n-1)
inline void half_table_fill(double* t) {
  for (int j = 0; j < HALF_ROWS; ++j) {
    const long double a = (long double)j / HALF_STEPS;
    long double c[HALF_ROW];
    c[0] = 0.5L * expl(a * a) * erfcl(a);
    c[1] = 2.0L * a * c[0] - 0.56418958354775628694807945156077259L;
    for (int n = 1; n + 1 < HALF_ROW - 1; ++n) c[n + 1] = (2.0L * a * c[n] + 2.0L * c[n - 1]) / (n + 1);
    t[j * HALF_ROW] = (double)a;
    for (int n = 0; n < HALF_ROW - 1; ++n) t[j * HALF_ROW + 1 + n] = (double)c[n];
  }
  for (int i = 0; i < 64; ++i) t[HALF_EXP + i] = (double)exp2l(-(long double)i / 64.0L);
}

HD double fast_rcp(double x) {
#ifdef __CUDA_ARCH__
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
#else
  return 1.0 / x;
#endif
}

HD double fast_rsqrt(double x) {
#ifdef __CUDA_ARCH__
  return rsqrt(x);
#else
  return 1.0 / sqrt(x);
#endif
}

#ifdef __CUDACC__
// the general functions, out of line (no call inside the table's range)
static __device__ __noinline__ void half_gauss_general(double y, double& m0, double& e) {
  m0 = 0.5 * erfc(y);
  e = exp(-y * y);
}
#endif

#ifdef __CUDA_ARCH__
// x >= 0 as FP32 (truncated; zero below 2^-100) by integer operations on its words; x < 2^127
__device__ __forceinline__ float half_to_float(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  return hi < ((1023 - 100) << 20) ? 0.0f : __int_as_float(((hi - (896 << 20)) << 3) | (int)((unsigned)lo >> 29));
}

// the high and low parts of ln 2/64 (the high one has 37 significant bits: n times it is exact below 2^16)
#define HALF_L1 0x1.62e42fefap-7
#define HALF_L2 0x1.cf79abc9e3b3ap-46

__device__ __forceinline__ double int_to_double(int n) {  // 0 <= n, one addition instead of a conversion
  return __hiloint2double(0x43300000, n) - 4503599627370496.0;
}

// 2^(-n/64) exp(-r), |r| <= ln 2/128
__device__ __forceinline__ double exp_scaled(double r, int n, const double* __restrict__ tab) {
  const double tn = __ldg(tab + HALF_EXP + (n & 63));
  double p = fma(r, -1.0 / 120.0, 1.0 / 24.0);
  p = fma(r, p, -1.0 / 6.0);
  p = fma(r, p, 0.5);
  p = fma(r, p, -1.0);
  p = fma(r, p, 1.0);
  const double e = tn * p;
  return __hiloint2double(__double2hiint(e) - ((n >> 6) << 20), __double2loint(e));
}
#endif

// exp(-x), x >= 0 (10 FP64 operations; 0 above 700, where the flux's weights vanish; NaN stays NaN)
HD double exp_neg(double x, const double* __restrict__ tab) {
#ifdef __CUDA_ARCH__
  if (__double2hiint(x) >= 0x4085e000) return x != x ? x : 0.0;  // 700, or not a number
  const int n = __float2int_rn(half_to_float(x) * 92.332482616893658f);  // 64 / ln 2
  const double nd = int_to_double(n);
  return exp_scaled(fma(-nd, HALF_L2, fma(-nd, HALF_L1, x)), n, tab);
#else
  (void)tab;
  return exp(-x);
#endif
}

// x > 0 (false for NaN, zero and below 2^-1042) by an integer comparison of the high word
HD bool positive(double x) {
#ifdef __CUDA_ARCH__
  return (unsigned)(__double2hiint(x) - 1) < 0x7ff00000u;
#else
  return x > 0.0;
#endif
}

// the smaller of two numbers that are not negative, by an integer comparison (unsigned, so that a NaN of
// either sign loses, as with fmin)
HD double min_positive(double a, double b) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(b) < (unsigned long long)__double_as_longlong(a) ? b : a;
#else
  return fmin(a, b);
#endif
}

// m0 = erfc(y)/2, e = exp(-y^2)
HD void half_gauss(double y, const double* __restrict__ tab, double& m0, double& e) {
#ifdef __CUDA_ARCH__
  const double a = fabs(y);
  if (__double2hiint(a) >= 0x40180000) {  // 6, or not a number
    half_gauss_general(y, m0, e);
    return;
  }
  const float af = half_to_float(a);
  const int j = __float2int_rn(af * (float)HALF_STEPS);
  const int n = __float2int_rn(af * af * 92.332482616893658f);
  const double2* row = reinterpret_cast<const double2*>(tab + j * HALF_ROW);
  const double2 c01 = __ldg(row), c23 = __ldg(row + 1), c45 = __ldg(row + 2), c67 = __ldg(row + 3), c89 = __ldg(row + 4);
  const double nd = int_to_double(n);
  e = exp_scaled(fma(-nd, HALF_L2, fma(a, a, -nd * HALF_L1)), n, tab);
  const double d = a - c01.x;
  double q = fma(d, c89.y, c89.x);
  q = fma(d, q, c67.y);
  q = fma(d, q, c67.x);
  q = fma(d, q, c45.y);
  q = fma(d, q, c45.x);
  q = fma(d, q, c23.y);
  q = fma(d, q, c23.x);
  q = fma(d, q, c01.y);
  m0 = e * q;
  if (__double2hiint(y) < 0) m0 = 1.0 - m0;
#else
  (void)tab;
  m0 = 0.5 * erfc(y);
  e = exp(-y * y);
#endif
}
