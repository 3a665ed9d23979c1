// fp_newton.h -- reciprocal and square root of doubles on the integer pipes:
// a 22-bit seed from the float special-function unit, one Newton-Raphson
// step in 32-bit fixed point, and a second one whose residual is exact in
// 64 bits, rounded once to the nearest double.  About 35 and 45 integer
// instructions, next to 3 and 6 FP64 ones that hold the FP64 pipe 64 cycles
// each.  Errors below 0.54 (reciprocal) and 0.52 (square root) units in the last
// place for seeds within 2^-22; the largest met in 4 million are 0.517 and 0.509.
// For finite normal arguments (sqrt: positive); anything else gives an
// unspecified value.
// Plain C as well as CUDA: on the host the seeds are passed in, so that a
// test can put every error the hardware may make into them.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FPN_FN __host__ __device__ __forceinline__
#else
#define FPN_FN static inline
#endif

FPN_FN uint32_t fpn_mulhi(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}
FPN_FN uint64_t fpn_bits(double x) {
  uint64_t b;
  memcpy(&b, &x, sizeof b);
  return b;
}
FPN_FN float fpn_float(uint32_t b) {
  float f;
  memcpy(&f, &b, sizeof f);
  return f;
}
// a seed in [1/2, 1) as a multiple of 2^-32 (held to that range, which a
// seed's own error can leave)
FPN_FN uint32_t fpn_seed(float s) {
  const float lo = 0.5f, hi = 0x1.fffffep-1f;
  s = s < lo ? lo : s;
  s = s > hi ? hi : s;
  uint32_t b;
  memcpy(&b, &s, sizeof b);
  return (b << 8) | 0x80000000u;
}

// the significand of x in [1, 2), cut to a float, for the seed of 1/x
FPN_FN float fpn_recip_arg(double x) {
  const uint64_t b = fpn_bits(x);
  return fpn_float(((uint32_t)(b >> 29) & 0x007fffffu) | 0x3f800000u);
}
// 1/x from a float seed of 1 / fpn_recip_arg(x)
FPN_FN double fpn_recip_seeded(double x, float seed) {
  const uint64_t b = fpn_bits(x);
  const uint32_t bh = (uint32_t)(b >> 32);
  const uint64_t M = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;  // x 2^52
  const uint32_t X = (uint32_t)(M >> 21);                                  // x 2^31
  const uint32_t R0 = fpn_seed(seed);                                      // r 2^32
  // r (1 + d), d = 1 - x r to 2^-31
  const int32_t d = (int32_t)(0x80000000u - fpn_mulhi(R0, X));
  const uint32_t R = R0 + (uint32_t)(((int64_t)(int32_t)(R0 >> 1) * d) >> 30);
  // 1 - x r = -P 2^-84, |P| < 2^56: exact in the low 64 bits
  const int64_t P = (int64_t)(M * R);
  const int32_t Ph = (int32_t)(P >> 25);
  const int64_t c = ((int64_t)Ph * (int32_t)(R >> 1)) >> 28;  // r (x r - 1) 2^62
  const uint64_t Q = ((uint64_t)R << 30) - (uint64_t)c;       // 2^62 / x
  const uint64_t q = (Q + 256) >> 9;
  // q in [2^52, 2^53] carries the exponent's last one
  const uint32_t eh = 0x7fc00000u - (bh & 0x7ff00000u);  // (2044 - e) << 20
  uint64_t r = q + ((uint64_t)eh << 32);
  r |= (uint64_t)(bh & 0x80000000u) << 32;
  double y;
  memcpy(&y, &r, sizeof y);
  return y;
}

// z scaled by an even power of two into [1, 4), cut to a float, for the seed
// of 1/sqrt
FPN_FN float fpn_sqrt_arg(double z) {
  const uint64_t b = fpn_bits(z);
  const uint32_t odd = ~(uint32_t)(b >> 52) & 1u;  // an odd power of two in z
  return fpn_float((((uint32_t)(b >> 29) & 0x007fffffu) | 0x3f800000u) + (odd << 23));
}
// sqrt(z) from a float seed of 1 / sqrt(fpn_sqrt_arg(z))
FPN_FN double fpn_sqrt_seeded(double z, float seed) {
  const uint64_t b = fpn_bits(z);
  const uint32_t e = (uint32_t)(b >> 52);
  const uint32_t odd = ~e & 1u;
  const uint64_t M = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  const uint64_t Z = M << (10 + odd);        // m 2^62, m in [1, 4)
  const uint32_t Zh = (uint32_t)(Z >> 32);   // m 2^30
  const uint32_t Y0 = fpn_seed(seed);        // y 2^32
  // y (1 + d / 2), d = 1 - m y^2 to 2^-30
  const int32_t d = (int32_t)(0x40000000u - fpn_mulhi(fpn_mulhi(Y0, Y0), Zh));
  const uint32_t Y = Y0 + (uint32_t)(((int64_t)(int32_t)(Y0 >> 1) * d) >> 30);
  const uint64_t s62 = (uint64_t)Zh * Y;     // m y = sqrt(m), 2^62
  // 2^31, held below 2 (m close to 4 and y too large)
  const uint32_t S = (int64_t)s62 < 0 ? 0xffffffffu : (uint32_t)(s62 >> 31);
  // s + (m - s^2) y / 2, the residual exact
  const int64_t res = (int64_t)(Z - (uint64_t)S * S);
  const int64_t c = ((int64_t)(int32_t)(res >> 4) * (int32_t)(Y >> 1)) >> 28;
  const uint64_t Q = ((uint64_t)S << 31) + (uint64_t)c;  // sqrt(m) 2^62
  const uint64_t q = (Q + 512) >> 10;
  const uint64_t r = q + ((uint64_t)(((e + 1023) >> 1) - 1) << 52);
  double y;
  memcpy(&y, &r, sizeof y);
  return y;
}
