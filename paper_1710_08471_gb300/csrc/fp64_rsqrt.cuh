// 1/sqrt(d) and sqrt(d) for the Cholesky pivots, in few FP64 operations.
//
// The pivots of a right-looking Cholesky are a serial chain (each waits for
// the previous column), and on GB300 every dependent FP64 operation costs 64
// clocks (a conversion between FP32 and FP64 as much), while integer and FP32
// operations take a few. The library's correctly rounded sqrt and division
// take many FP64 operations each. Here instead:
//   d = f 2^(2k) with f in [1, 4) (exponent split by integer operations),
//   y0 = single-precision 1/sqrt(f) of f's leading 24 bits (the operand and
//        the result moved between the formats by bit operations, not by
//        conversion instructions; about 22 correct bits),
//   one third-order step for the root of 1/y^2 - f:
//     e = 1 - f y0^2,  y = y0 (1 + e/2 + 3 e^2/8),
//   whose error term 5 e^3 / 16 is below 2^-60 (four dependent FP64
//   operations against six for two Newton-Raphson steps), then
//   1/sqrt(d) = y 2^(-k) (exact exponent shift) and sqrt(d) = d * (1/sqrt(d)).
// Both results are within a few ulps, which the factorization's rounding
// analysis absorbs. Zero, subnormal, negative and non-finite pivots take the
// library functions (a breakdown is reported from the pivot value anyway).
// Host-compilable, so the error bound is checked on the CPU.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define RS_HD __host__ __device__ __forceinline__
#else
#define RS_HD inline
#endif

namespace cqr2 {

RS_HD unsigned long long rs_bits(double x) {
#if defined(__CUDA_ARCH__)
  return (unsigned long long)__double_as_longlong(x);
#else
  unsigned long long b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}

RS_HD double rs_from_bits(unsigned long long b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, sizeof x);
  return x;
#endif
}

RS_HD unsigned rs_f32_bits(float x) {
#if defined(__CUDA_ARCH__)
  return (unsigned)__float_as_uint(x);
#else
  unsigned b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}

RS_HD float rs_f32_from_bits(unsigned b) {
#if defined(__CUDA_ARCH__)
  return __uint_as_float(b);
#else
  float x;
  memcpy(&x, &b, sizeof x);
  return x;
#endif
}

// Single-precision seed of 1/sqrt(f), f in [1, 4).
RS_HD float rs_seed(float f) {
#if defined(__CUDA_ARCH__)
  return rsqrtf(f);
#else
  return 1.0f / sqrtf(f);
#endif
}

// One third-order step from a seed y0 ~ 1/sqrt(f), f in [1, 4):
// y = y0 (1 + e/2 + 3 e^2/8) with e = 1 - f y0^2.
RS_HD double rs_refine3(double f, double y0) {
  const double t = f * y0;
  const double e = fma(-t, y0, 1.0);
  const double p = fma(e, 0.375, 0.5);
  const double ye = y0 * e;
  return fma(ye, p, y0);
}

// The FP64 value of a positive normal float, by bit operations.
RS_HD double rs_f32_to_f64(float x) {
  const unsigned b = rs_f32_bits(x);
  return rs_from_bits(((unsigned long long)((b >> 23) - 127 + 1023) << 52) | ((unsigned long long)(b & 0x7FFFFF) << 29));
}

// r = 1/sqrt(d) for a positive normal d; returns false (and fills r and l
// from the library functions) otherwise. l is left to the caller on success
// (l = d * r, which a kernel can fold into its column scaling).
RS_HD bool chol_rsqrt_r(double d, double* r, double* l) {
  const unsigned long long b = rs_bits(d);
  const int ex = (int)((b >> 52) & 0x7FF);
  if ((b >> 63) != 0 || ex == 0 || ex == 0x7FF) {
    *l = sqrt(d);
    *r = 1.0 / *l;
    return false;
  }
  const int e = ex - 1023;                 // d = 1.m 2^e
  const int k = (e >= 0 ? e : e - 1) / 2;  // floor(e / 2)
  const int fe = e - 2 * k;                // 0 or 1: f = 1.m 2^fe in [1, 4)
  const unsigned long long m = b & ((1ull << 52) - 1);
  const double f = rs_from_bits(m | ((unsigned long long)(1023 + fe) << 52));
  const float ff = rs_f32_from_bits(((unsigned)(127 + fe) << 23) | (unsigned)(m >> 29));  // f truncated
  const double y = rs_refine3(f, rs_f32_to_f64(rs_seed(ff)));
  // 1/sqrt(d) = y 2^-k: y is in (1/2, 1], so the shifted exponent stays normal
  *r = rs_from_bits(rs_bits(y) - ((unsigned long long)(long long)k << 52));
  return true;
}

// r = 1/sqrt(d) and l = sqrt(d) for a positive normal d; returns false (and
// fills both from the library functions) otherwise.
RS_HD bool chol_rsqrt(double d, double* r, double* l) {
  if (!chol_rsqrt_r(d, r, l)) return false;
  *l = d * *r;
  return true;
}

// r = 1/sqrt(d) and l = sqrt(d) within 0.51 ulp for a positive normal d: one
// more step for each, from the residual d - l^2 (exact but for its rounding),
// for where they are not on a chain.
RS_HD void chol_rsqrt_tight(double d, double* r, double* l) {
  if (!chol_rsqrt(d, r, l)) return;
  const double r0 = *r, l0 = *l;
  *l = fma(0.5 * r0, fma(-l0, l0, d), l0);
  const double lo = fma(d, r0, -l0);
  *r = fma(0.5 * r0, fma(-lo, r0, fma(-l0, r0, 1.0)), r0);
}

// a / d, correctly rounded, from r = 1 / d (correctly rounded): the product and
// one correction by its exact remainder (P. Markstein, IBM J. Res. Dev. 34(1),
// 1990), for where many quotients share a divisor. For intermediates in the
// normal range.
RS_HD double rs_quotient(double a, double d, double r) {
  const double q = a * r;
  return fma(fma(-q, d, a), r, q);
}

// Single-precision seed of 1/f, f in [1, 2).
RS_HD float rs_rcp_seed(float f) {
#if defined(__CUDA_ARCH__)
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  return r;
#else
  return 1.0f / f;
#endif
}

// 1/d for a positive d with an exponent in [2^-999, 2^996], in integers: on
// GB300 an FP64 operation costs 64 clocks of latency and of its partition's
// pipe, an integer one 4 or 5, and the chain of pivots waits for this. With
// d = F 2^(x-52), F a 53-bit integer, and the seed y0 = Y0 2^-24 of 1/f,
// f = F 2^-52 (about 22 correct bits):
//   e = 1 - f y0 = -(F Y0 mod 2^64) 2^-76   (exact: F Y0 = 2^76 (1 - e)),
//   y = y0 (1 + e + e^2)                     (the next term is below 2^-64),
// formed in units of 2^-60 and rounded to 53 bits: within 0.52 ulp.
RS_HD double pivot_rcp(double d) {
  const unsigned long long b = rs_bits(d);
  const unsigned long long F = (b & ((1ull << 52) - 1)) | (1ull << 52);
  const float y0 = rs_rcp_seed(rs_f32_from_bits((127u << 23) | (unsigned)((b >> 29) & 0x7FFFFF)));
  const unsigned Y0 = rs_f32_bits(y0) - ((125u << 23));  // y0 2^24 for y0 in [1/2, 1]
  const long long E = -(long long)(F * Y0);  // units of 2^-76, |E| < 2^55
  const int Eh = (int)(E >> 32);
  const long long T = E + (((long long)Eh * Eh) >> 12);
  const long long Y = ((long long)Y0 << 36) + (((T >> 16) * (long long)Y0) >> 24);
  // Y in (2^59, 2^60]: the value 1/f in (1/2, 1], then the exponent of d
  const unsigned long long m = ((unsigned long long)Y + 64) >> 7;
  return rs_from_bits(m + ((1021ull - (((b >> 52) & 0x7FF) - 1023ull)) << 52));
}
RS_HD bool pivot_rcp_ok(double d) {  // positive, finite, exponent in pivot_rcp's range
  const unsigned e = (unsigned)(rs_bits(d) >> 52);  // sign included
  return e >= 24 && e <= 2019;
}

}  // namespace cqr2
