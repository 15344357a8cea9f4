// Integer arithmetic of the split-precision path, host-compilable so that it
// can be checked on the CPU against exact rational arithmetic:
// - slicing: an FP64 entry x with shared exponent e (|x| < 2^e) becomes the
//   fixed-point integer v = round(x 2^(7 + 8 (S - 1) - e)) and then S
//   balanced base-256 digits, v = sum_s d_s 256^(S - 1 - s);
// - recombination: the fixed-point accumulators back to FP64, with integer
//   operations only (GB300's FP64 pipe is far too slow even for conversions).
#pragma once

#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define OZ_HD __host__ __device__ __forceinline__
#else
#define OZ_HD inline
#endif

namespace cqr2 {

constexpr int OZ_EXP_NONFINITE = 1 << 20;  // exponent sentinel: a non-finite entry was seen

OZ_HD long long oz_double_bits(double x) {
#if defined(__CUDA_ARCH__)
  return __double_as_longlong(x);
#else
  long long b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}

// v = x 2^(7 + 8 (S - 1) - e), rounded half away from zero, for |x| < 2^e:
// |v| < 2^(7 + 8 (S - 1)). Zero for a non-finite x or exponent.
OZ_HD long long oz_to_fixed(double x, int e, int S) {
  const unsigned long long b = (unsigned long long)oz_double_bits(x);
  int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long mant = b & ((1ull << 52) - 1);
  if (ex == 0) {
    if (mant == 0) return 0;
    ex = 1;
  } else {
    mant |= 1ull << 52;
  }
  if (e >= OZ_EXP_NONFINITE || ex == 0x7FF) return 0;
  const int sh = ex - 1075 + 7 + 8 * (S - 1) - e;  // < 8S - 53 because |x| < 2^e
  long long v;
  if (sh >= 0) {
    v = (long long)(mant << sh);
  } else if (sh > -63) {
    v = (long long)((mant + (1ull << (-sh - 1))) >> (-sh));
  } else {
    v = 0;
  }
  return (b >> 63) ? -v : v;
}

// Balanced base-256 digits of v, most significant first: d[1..S-1] in
// [-128, 127] and v = sum_s d[s] 256^(S - 1 - s). With B = 128 in each of the
// S - 1 low bytes, the low digits are the bytes of v + B minus 128 and the
// top digit is v + B shifted down arithmetically -- the same digits as
// peeling the signed low byte off one at a time (d = sext(v mod 256), v =
// (v - d) / 256), without that serial chain.
template <int S>
OZ_HD void oz_balanced_digits(long long v, int (&d)[S]) {
  constexpr unsigned long long B = ((1ull << (8 * (S - 1))) - 1) / 255 * 128;
  const unsigned long long u = (unsigned long long)v + B;
  const unsigned lo = (unsigned)u, hi = (unsigned)(u >> 32);
#if defined(__CUDA_ARCH__)
#pragma unroll
#endif
  for (int i = 0; i < S - 1; ++i) {
    const unsigned byte = ((i < 4 ? lo : hi) >> (8 * (i & 3))) & 0xFFu;
    d[S - 1 - i] = (int)byte - 128;
  }
  d[0] = (int)((long long)u >> (8 * (S - 1)));
}

OZ_HD int oz_clz64(unsigned long long x) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

OZ_HD double oz_bits_to_double(unsigned long long b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, sizeof d);
  return d;
#endif
}

// Exact value m 2^e (m < 2^53) rounded into the subnormal range (or zero),
// for the rare results below the normal range. Round to nearest, ties to even.
OZ_HD double oz_scale_small(unsigned long long mant53, unsigned long long sticky_in, int e) {
  // result bits = round(mant53 2^(e + 1074)); e + 1074 < 0 here
  const int sh = -(e + 1074);
  if (sh >= 64) return 0.0;
  const unsigned long long q = mant53 >> sh;
  const unsigned long long r = mant53 & ((1ull << sh) - 1ull);
  const unsigned long long halfv = 1ull << (sh - 1);
  const bool up = r > halfv || (r == halfv && (sticky_in || (q & 1ull)));
  return oz_bits_to_double(q + (up ? 1ull : 0ull));
}

// (hi 2^32 + lo) 2^E rounded to the nearest double, ties to even, for
// |hi|, |lo| < 2^62 (the accumulators of 2^20 rows stay far below that).
OZ_HD double oz_fixed_to_double(long long hi, long long lo, int E) {
  // T = H 2^32 + L with 0 <= L < 2^32
  const long long H = hi + (lo >> 32);
  const unsigned L = (unsigned)(unsigned long long)lo;
  const bool neg = H < 0;
  // |T| = W 2^32 + w0
  const unsigned w0 = neg ? 0u - L : L;
  const unsigned long long W = neg ? ~(unsigned long long)H + (L == 0u ? 1ull : 0ull) : (unsigned long long)H;
  unsigned long long hw = W, lw = (unsigned long long)w0 << 32;
  int top = 95;  // bit of |T| that bit 63 of hw holds
  if (hw == 0) {
    hw = lw;
    lw = 0;
    top = 31;
  }
  if (hw == 0) return 0.0;
  const int lz = oz_clz64(hw);
  const unsigned long long N = (hw << lz) | (lw >> 1 >> (63 - lz));  // top 64 bits, bit 63 set
  const unsigned long long rest = lw << lz;                           // bits below N
  const int msb = top - lz;                                            // |T| in [2^msb, 2^(msb+1))
  unsigned long long mant = N >> 11;                                   // 53 bits, bit 52 set
  const unsigned long long halfbit = (N >> 10) & 1ull;
  const unsigned long long sticky = ((N & 0x3FFull) | rest) != 0 ? 1ull : 0ull;
  const int biased = msb + E + 1023;
  if (biased < 1) {
    const double mag = oz_scale_small(mant, halfbit | sticky, msb + E - 52);
    return neg ? -mag : mag;
  }
  mant += halfbit & (sticky | (mant & 1ull));
  // the implicit bit adds one to the exponent field; a rounding carry to
  // 2^53 moves it one further, as it must
  unsigned long long bits = ((unsigned long long)(biased - 1) << 52) + mant;
  if (biased > 2046) bits = 0x7FF0000000000000ull;  // overflow to infinity
  return oz_bits_to_double(bits | (neg ? 1ull << 63 : 0ull));
}

// The accumulators as kept by the kernel: T = X 2^24 + Y with X holding
// groups 0-3 and Y groups 4-6. Exact conversion through (hi, lo).
OZ_HD double oz_xy_to_double(long long X, long long Y, int E) {
  const long long hi = X >> 8;  // T = hi 2^32 + ((X mod 2^8) 2^24 + Y)
  const long long lo = (long long)((unsigned long long)(X & 0xFF) << 24) + Y;
  return oz_fixed_to_double(hi, lo, E);
}

#if defined(__CUDA_ARCH__)
// The exact routine as an out-of-line call for the fast routine's rare
// subnormal case: inlined at every output it would crowd the instruction
// cache of the epilogue loop with code that almost never runs.
static __device__ __noinline__ double oz_xy_to_double_cold(long long X, long long Y, int E) {
  return oz_xy_to_double(X, Y, E);
}
#define OZ_XY_COLD oz_xy_to_double_cold
#else
#define OZ_XY_COLD oz_xy_to_double
#endif

// Faster conversion of T = X 2^24 + Y (|X| < 2^61, |Y| < 2^55) to within one ulp
// of T 2^E: T 2^-(24-s) = X 2^s + Y 2^-(24-s) fits 62 bits when s = min(24, 62 -
// (bits of |X|)), and what falls off Y is then below 2^-61 of |T|. The hardware
// converts that integer with one correct rounding (one FP64 operation), and the
// exponent is added to its bits. Each output has its own shift: with one for a
// group of outputs the bits that fall off would be below 2^-61 of the group's
// largest only, and it was no faster (group shift of a thread's four or eight
// outputs with 64-bit shifts, and this: 2^23 x 128 29.13, 29.15 ms; 2^21 x 512
// 57.7, 57.1; 1000037 x 200 with six slices 7.63, 7.70).
OZ_HD unsigned oz_high_bits(long long X) {
  const int hi = (int)(X >> 32);
  return (unsigned)(hi ^ (hi >> 31));
}
// h: oz_high_bits(X), or their OR over outputs that share a shift.
OZ_HD int oz_group_shift(unsigned h) {
#if defined(__CUDA_ARCH__)
  const int lz = __clz((int)h);
#else
  const int lz = h ? __builtin_clz(h) : 32;
#endif
  return lz - 2 < 24 ? lz - 2 : 24;
}
OZ_HD unsigned oz_funnel_l(unsigned lo, unsigned hi, int s) {  // high word of (hi:lo) << s, s < 32
#if defined(__CUDA_ARCH__)
  return __funnelshift_l(lo, hi, s);
#else
  return (unsigned)(((((unsigned long long)hi << 32) | lo) << s) >> 32);
#endif
}
// floor(X 2^s + Y 2^-(24-s)): T = hi 2^24 + lo with lo's 24 bits in one word, so
// that two funnel shifts form it (64-bit shifts by a variable count take several
// instructions each).
OZ_HD long long oz_shifted_int(long long X, long long Y, int s) {
  const unsigned long long hi = (unsigned long long)(X + (Y >> 24));
  const unsigned h1 = (unsigned)(hi >> 32), h0 = (unsigned)hi, lo = (unsigned)Y << 8;
  return (long long)(((unsigned long long)oz_funnel_l(h0, h1, s) << 32) | oz_funnel_l(lo, h0, s));
}
// Z 2^e without the rare cases, so that a kernel can run several side by side
// without branches; ok is false for zero and for a result outside the normal range.
OZ_HD double oz_int_to_double(long long Z, int e, bool* ok) {
#if defined(__CUDA_ARCH__)
  const double d = __ll2double_rn(Z);
#else
  const double d = (double)Z;
#endif
  const unsigned long long b = (unsigned long long)oz_double_bits(d);
  const int ex = (int)((b >> 52) & 0x7FF);
  *ok = ex != 0 && (unsigned)(ex + e - 1) < 2046u;
  return oz_bits_to_double(b + ((unsigned long long)(long long)e << 52));
}
// With a given shift, Y rounded to it; the rare cases exactly.
OZ_HD double oz_xy_to_double_group(long long X, long long Y, int s, int E) {
  const long long Z = oz_shifted_int(X, Y + (0x800000u >> s), s);
  bool ok;
  const double v = oz_int_to_double(Z, E + 24 - s, &ok);
  if (ok) return v;
  return Z == 0 ? 0.0 : OZ_XY_COLD(X, Y, E);
}
// With the output's own shift: without its rare cases, and complete.
OZ_HD double oz_xy_to_double_fast_normal(long long X, long long Y, int E, bool* ok) {
  const int s = oz_group_shift(oz_high_bits(X));
  return oz_int_to_double(oz_shifted_int(X, Y, s), E + 24 - s, ok);
}
OZ_HD double oz_xy_to_double_fast(long long X, long long Y, int E) {
  bool ok;
  const double v = oz_xy_to_double_fast_normal(X, Y, E, &ok);
  return ok ? v : oz_xy_to_double_group(X, Y, oz_group_shift(oz_high_bits(X)), E);
}

}  // namespace cqr2
