// fp_bits.h -- IEEE-754 operations on doubles computed with integer (and float)
// arithmetic.  On GB300 a double operation, a comparison and a conversion each
// hold the FP64 pipe for about 64 cycles per warp instruction per sub-partition,
// while the integer pipes are otherwise idle in the FP64-bound kernels; these
// functions give the same result as the hardware instruction (bit for bit, save
// for which NaN a NaN becomes).  Plain C as well as CUDA, so that host unit
// tests check them against the host's own IEEE arithmetic.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FPB_FN __host__ __device__ __forceinline__
#else
#define FPB_FN static inline
#endif

// On the device by the two halves: a test of the pattern of a reinterpreted
// double (is it zero, an infinity) the compiler turns back into an FP64 compare.
FPB_FN uint64_t fpb_bits_of_double(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)(uint32_t)__double2hiint(x) << 32 | (uint32_t)__double2loint(x);
#else
  uint64_t b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}

FPB_FN float fpb_float_of_bits(uint32_t b) {
  float f;
  memcpy(&f, &b, sizeof f);
  return f;
}

// x rounded to the nearest float, ties to even (cvt.rn.f32.f64): overflow
// gives an infinity, results below the smallest normal float are the
// correctly rounded subnormals (no flush to zero), a NaN gives a quiet NaN
// with the sign and the leading payload bits of x
FPB_FN float fpb_double_to_float_rn(double x) {
  const uint64_t b = fpb_bits_of_double(x);
  const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
  const int e = (int)((b >> 52) & 0x7ff);
  const uint64_t m = b & 0x000fffffffffffffull;
  if (e == 0x7ff)  // infinity, or NaN made quiet
    return fpb_float_of_bits(sign | 0x7f800000u | (m ? 0x00400000u | (uint32_t)(m >> 29) : 0u));
  const int fe = e - 1023 + 127;  // biased float exponent of a normal result
  if (fe >= 0xff) return fpb_float_of_bits(sign | 0x7f800000u);
  if (fe > 0) {
    // 52 -> 23 fraction bits; a carry out of the fraction steps the
    // exponent, up to infinity, which is the right result
    uint32_t r = (uint32_t)(m >> 29);
    const uint32_t rem = (uint32_t)(m & 0x1fffffffu);
    if (rem > 0x10000000u || (rem == 0x10000000u && (r & 1u))) r += 1u;
    return fpb_float_of_bits(sign | (((uint32_t)fe << 23) + r));
  }
  if (e == 0) return fpb_float_of_bits(sign);  // zero or a double subnormal
  // a float subnormal: k = round(M 2^-s) units of 2^-149, M the 53-bit
  // significand; s >= 30, and beyond 54 the result is zero
  const int s = 926 - e;
  if (s > 54) return fpb_float_of_bits(sign);
  const uint64_t M = m | 0x0010000000000000ull;
  uint64_t k = M >> s;
  const uint64_t rem = M & ((1ull << s) - 1ull), half = 1ull << (s - 1);
  if (rem > half || (rem == half && (k & 1ull))) k += 1ull;
  return fpb_float_of_bits(sign | (uint32_t)k);
}

FPB_FN double fpb_double_of_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)(b >> 32), (int)b);
#endif
  double x;
  memcpy(&x, &b, sizeof x);
  return x;
}

// the double difference of two floats, (double)a - (double)b, from the float
// difference d and its error e (Knuth's two-sum: d + e is exact): e is counted
// in units of the double's last place and added to d's bit pattern.  *ok: the
// result is right; not so for infinities, NaNs and subnormals, or, with e not
// zero, where d is a power of two (the sum may lie in the binade below) or tiny.
FPB_FN double fpb_diff(float a, float b, int* ok) {
  const float d = a - b, t = d - a, e = (a - (d - t)) - (b + t);
  uint32_t bits;
  memcpy(&bits, &d, sizeof bits);
  const uint32_t m = bits & 0x7fffffffu;
  *ok = e == 0.0f ? m - 1u >= 0x007fffffu
                  : m - 0x1a800000u < 0x7f800000u - 0x1a800000u && (m & 0x007fffffu) != 0;
  // |e| <= 2^-24 |d|, so |q| <= 2^28
  const float u = e * fpb_float_of_bits((306u << 23) - (bits & 0x7f800000u));
#ifdef __CUDA_ARCH__
  const int q = e == 0.0f ? 0 : __float2int_rn(u);
#else
  const int q = e != 0.0f && *ok ? (int)rintf(u) : 0;
#endif
  const int s = -(int)(bits >> 31);
  const uint32_t hi = (bits & 0x80000000u) | (m ? (m >> 3) + (896u << 20) : 0u);
  return fpb_double_of_bits(((uint64_t)hi << 32 | (uint64_t)(bits << 29)) +
                            (uint64_t)(int64_t)((q ^ s) - s));
}

// x c for c a power of two (fpb_is_pow2) as a step of the exponent, where operand
// and result are normal numbers or x is zero (fpb_pow2_steps)
FPB_FN int fpb_is_pow2(double c) {  // a normal positive power of two
  const uint64_t b = fpb_bits_of_double(c);
  return (b & 0x800fffffffffffffull) == 0 && b != 0 && b != 0x7ff0000000000000ull;
}
FPB_FN int fpb_pow2_steps(double x, double c) {
  const uint64_t b = fpb_bits_of_double(x);
  const int e = (int)(b >> 52) & 0x7ff, r = e + (int)(fpb_bits_of_double(c) >> 52) - 1023;
  return (b << 1) == 0 || (e > 0 && e < 0x7ff && r > 0 && r < 0x7ff);
}
FPB_FN double fpb_step_exponent(double x, double c) {
  const uint64_t b = fpb_bits_of_double(x);
  return (b << 1) == 0 ? x
                       : fpb_double_of_bits(b + (fpb_bits_of_double(c) - 0x3ff0000000000000ull));
}

// comparisons of doubles on integer arithmetic.  The IEEE order of doubles
// that are not NaN is the order of the keys b ^ ((b >> 63) & 0x7fff...) of
// their bit patterns b, read as signed integers, save that -0 and +0 compare
// equal.  Each function gives exactly the IEEE answer for the inputs its
// name allows ("num": neither is NaN; "ieee": any input, false with a NaN).
FPB_FN int64_t fpb_order_key(double x) {
  const int64_t b = (int64_t)fpb_bits_of_double(x);
  return b ^ ((b >> 63) & INT64_MAX);
}
FPB_FN int fpb_is_nan(double x) {
  return (int64_t)(fpb_bits_of_double(x) & 0x7fffffffffffffffull) > 0x7ff0000000000000ll;
}
// a < b
FPB_FN int fpb_lt_num(double a, double b) {
  const uint64_t both = fpb_bits_of_double(a) | fpb_bits_of_double(b);
  return fpb_order_key(a) < fpb_order_key(b) && (both << 1) != 0;
}
FPB_FN int fpb_lt_ieee(double a, double b) {
  return !fpb_is_nan(a) && !fpb_is_nan(b) && fpb_lt_num(a, b);
}
// a <= b
FPB_FN int fpb_le_ieee(double a, double b) {
  return !fpb_is_nan(a) && !fpb_is_nan(b) && !fpb_lt_num(b, a);
}
// x >= 0 and x > 0
FPB_FN int fpb_ge0_num(double x) {
  const int64_t b = (int64_t)fpb_bits_of_double(x);
  return b >= 0 || b == INT64_MIN;
}
FPB_FN int fpb_gt0_num(double x) { return (int64_t)fpb_bits_of_double(x) > 0; }
