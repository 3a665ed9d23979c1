// fixed_dot.h -- weighted sums of doubles in 64-bit fixed point, on the
// integer pipes.
//
// An FP64 instruction holds a GB300 SM sub-partition for 64 cycles; a
// 32 x 32 + 64-bit integer multiply-add takes 2 and a 64-bit add takes 2
// (measured).  So a stencil sum sum_m z_m x_m is formed as
//   x_m  -> X_m, an integer multiple of 2^-58 of the largest power of two in
//           the stencil (59 bits and a sign), the nearest,
//   z_m  -> C_m, an integer multiple of 2^-T, T = 60 where |z| < 1,
//   the sum of products exactly, in two limbs of 30 low bits and the rest,
//   the sum cut to 2^-60 of the stencil's scale (to odd, fxd_round), and
//   rounded once to a double.
// A value within a factor of 64 of the stencil's largest is converted without
// loss, so the sum carries the rounding of its weights (2^-61) and the one to
// double: 4.5e-17 rms of the result, where an FP64 FMA chain leaves 1.5e-16
// (R = 3).  Smaller values are rounded to 2^-59 of the largest power: with the
// stencil's outermost cell 10^3 to 10^10 times the others, so that a small
// weight's product is all there is, 1.4e-16 next to the chain's 1.4e-16 (R = 2)
// and 1.9e-16 (R = 3); the parity sums of the FP64 kernels before had 1.2e-16
// there.  Every step is odd (the sum of the negated values is the negated sum,
// bit for bit) and does not depend on the order of the terms, so mirror images
// stay mirror images.
// Plain C as well as CUDA, so that a host unit test can check it.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FXD_FN __host__ __device__ __forceinline__
#else
#define FXD_FN static inline
#endif

#define FXD_SPLIT 30     // bits of the low limbs
#define FXD_EMIN 64      // smallest reference exponent (all-zero stencils)
#define FXD_ROUND 58     // bits of a sum of products that fxd_round takes off

// the words of a double
FXD_FN uint32_t fxd_hi(double x) {
  uint64_t b;
  memcpy(&b, &x, sizeof b);
  return (uint32_t)(b >> 32);
}
FXD_FN uint32_t fxd_lo(double x) {
  uint64_t b;
  memcpy(&b, &x, sizeof b);
  return (uint32_t)b;
}

// v >> s for 0 <= s, zero from 64 on
FXD_FN uint64_t fxd_shr(uint64_t v, int s) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));  // PTX clamps the amount
  return r;
#else
  return s > 63 ? 0 : v >> s;
#endif
}
FXD_FN int fxd_clz(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

// x as the nearest multiple of 2^(E - 1081), E >= the biased exponent of x: 53
// significant bits moved up by 6 and down by E - e, and the first bit cut off
// added (halves away from zero).  Zeros and subnormals (e = 0 < FXD_EMIN <= E)
// give zero.
FXD_FN int64_t fxd_from_double(double x, int E) {
  const uint32_t h = fxd_hi(x), l = fxd_lo(x);
  const int e = (int)((h >> 20) & 0x7ffu);
  const uint32_t mh = ((h << 7 | l >> 25) & 0x07ffffffu) | 0x08000000u;
  const uint64_t M = (uint64_t)mh << 32 | (uint32_t)(l << 7);  // moved up by one more
  const uint64_t m = fxd_shr(M, E + 1 - e);
  const uint32_t next = (uint32_t)fxd_shr(M, E - e);  // its last bit
  const int64_t s = (int32_t)h >> 31;
  // m + bit, or ~m + 1 - bit = -(m + bit)
  return (int64_t)((m ^ (uint64_t)s) + ((next ^ (uint32_t)s) & 1u));
}

// the limbs of a stencil sum |s| < 2^61: s = hi 2^30 + lo, 0 <= lo < 2^30
FXD_FN int32_t fxd_limb_hi(int64_t s) { return (int32_t)(s >> FXD_SPLIT); }
FXD_FN int32_t fxd_limb_lo(int64_t s) { return (int32_t)s & ((1 << FXD_SPLIT) - 1); }

// the limbs of a weight |c| 2^T < 2^60: C = hi 2^30 + lo, |lo| <= 2^29
FXD_FN void fxd_weight(double c, int T, int32_t* hi, int32_t* lo) {
  // c 2^T to the nearest integer; a product by a power of two is exact (a half
  // added would be rounded itself from 2^52 on)
  const int64_t C = (int64_t)rint(c * (double)(1ll << T));
  const int64_t h = (C + (1ll << (FXD_SPLIT - 1))) >> FXD_SPLIT;
  *hi = (int32_t)h;
  *lo = (int32_t)(C - h * (1ll << FXD_SPLIT));
}

// the running sum of products: hh 2^60 + mid 2^30 + ll (fxd_fits: no sum of a
// set of weights can overflow)
typedef struct {
  int64_t hh, mid, ll;
} fxd_acc;
FXD_FN void fxd_mac(fxd_acc* a, int32_t ch, int32_t cl, int32_t sh, int32_t sl) {
  a->hh += (int64_t)ch * sh;
  a->mid += (int64_t)ch * sl;
  a->mid += (int64_t)cl * sh;
  a->ll += (int64_t)cl * sl;
}
// what one weight's limbs add to the bounds of its sum's middle and low limbs;
// cnt: cells in its stencil sum, each below 2^59
typedef struct {
  double mid, up, down;
} fxd_load;
FXD_FN void fxd_count(fxd_load* b, int32_t ch, int32_t cl, int cnt) {
  b->mid += fabs((double)ch) * 0x1p30 + fabs((double)cl) * cnt * 0x1p29;
  if (cl > 0) b->up += cl * 0x1p30;
  else b->down -= cl * 0x1p30;
}
FXD_FN int fxd_fits(const fxd_load* b) {
  return b->mid < 0x1p63 - 0x1p40 && b->up < 0x1p63 && b->down < 0x1p63;
}
// the sum over 2^58, exact or the odd one of its two neighbours (the last bit
// set where anything is cut off).  Odd as a function: the sum alone decides, not
// how it is spread over the limbs, and a sum and its negative have the same
// neighbours.  (To the nearest would need the sign of the whole sum for ties.)
FXD_FN int64_t fxd_round(fxd_acc a) {
  const int64_t m = a.mid + (a.ll >> FXD_SPLIT);
  const int shift = FXD_ROUND - FXD_SPLIT;
  const uint32_t cut = ((uint32_t)m & ((1u << shift) - 1u)) |
                       ((uint32_t)a.ll & ((1u << FXD_SPLIT) - 1u));
  return (int64_t)((uint64_t)a.hh << (2 * FXD_SPLIT - FXD_ROUND)) + ((m >> shift) | (cut != 0u));
}

// the double nearest r 2^(E + off - 1086): off = 3 + 60 - T takes the sums of
// fxd_round with weights of T bits and values of reference exponent E.  Beyond
// the largest double: a NaN (or an infinity).  `special`: bits OR-ed into the
// high word (0x7ff80000: a NaN, for a stencil that holds a NaN or an infinity;
// else 0).
FXD_FN double fxd_to_double(int64_t r, int E, int off, uint32_t special) {
  const uint64_t s = (uint64_t)(r >> 63);
  const uint64_t m = ((uint64_t)r ^ s) - s;
  uint32_t h = (uint32_t)(m >> 32), l = (uint32_t)m;
  int e = E + off - 1;  // the leading one of the significand adds one
  if (h == 0) {
    h = l;
    l = 0;
    e -= 32;
  }
  const int z = fxd_clz(h);  // 32 for r = 0
  const uint64_t n = ((uint64_t)h << 32 | l) << z;
  const uint64_t q = (n >> 11) + ((n >> 10) & 1u);  // halves away from zero
  uint64_t b = q + ((uint64_t)(uint32_t)(e - z) << 52);
  // an exponent past the range stays there, and out of the sign
  uint32_t bh = (uint32_t)(b >> 32);
  bh = bh < 0x7ff80000u ? bh : 0x7ff80000u;
  b = (uint64_t)bh << 32 | (uint32_t)b;
  if (h == 0) b = 0;
  b |= (s & 0x8000000000000000ull) | ((uint64_t)special << 32);
  double x;
  memcpy(&x, &b, sizeof b);
  return x;
}
