// Quotients of doubles with most of the work off the FP64 unit: quick_div and quick_recip,
// and exact_div and exact_recip where the bits of a / b are wanted.  Plain C++ as well, so that
// the arithmetic can be checked on the host.
//
// GB300 issues one FP64 warp instruction per 68-76 cycles, and a / b costs nine of them
// (refinements of a hardware seed).  Here the seed is carried to 41 bits on the FP32
// and integer units, which leaves a product, its remainder and one correction (Markstein
// 1990): the result is (a / b)(1 + d), |d| < 2^-82, rounded once.  Measured in the kernel
// that adds a / b to a field of 250^3 cells: 350 -> 165 us (74 by its bytes); batched rates
// with optical-depth weights (128^3, 2e3 sources): 4.31 -> 2.83 ms.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "scaled_sum.cuh"

namespace asora {

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float qd_float(uint32_t b) { return __uint_as_float(b); }
__device__ __forceinline__ uint32_t qd_bits(float x) { return __float_as_uint(x); }
__device__ __forceinline__ uint32_t qd_round(float x) { return __float2uint_rn(x); }
__device__ __forceinline__ float qd_seed(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
#else
inline float qd_float(uint32_t b) { float x; memcpy(&x, &b, 4); return x; }
inline uint32_t qd_bits(float x) { uint32_t b; memcpy(&b, &x, 4); return b; }
inline uint32_t qd_round(float x) { return (uint32_t)llrintf(x); }
#ifndef ASORA_QD_SEED  // (a test replaces it by results one unit off, the bound of rcp.approx)
#define ASORA_QD_SEED(x) (1.0f / (x))
#endif
inline float qd_seed(float x) { return ASORA_QD_SEED(x); }
#endif

// 1/b from below or above by less than 2^-41, for 2^-400 <= b < 2^400.  b = f 2^k, f in
// [1, 2); h: f's first 24 bits, l: the next 23, as a number in [0, 1).  s, a float below
// 1/f (rcp.approx is within 2^-23, h adds 2^-23, the fused step 2^-24) and not below 1/2;
// 1/f = s + s (1 - f s) (1 + ..), where 1 - f s < 2^-20.8 is formed in two fused steps.  The
// correction is added to the double s as an integer count of units of 2^-53: s is in
// [1/2, 1), so the sum never leaves its binade except to become 1.
ASORA_HD double recip41(uint32_t hi, uint32_t lo) {
  const float h = qd_float(0x3f800000u | ((hi << 3) & 0x7ffff8u) | (lo >> 29));
  const float l = qd_float(0x3f800000u | ((lo << 3) >> 9)) - 1.0f;
  const float s0 = qd_seed(h);
  const float s = fmaxf(fmaf(s0, -0x1.8p-22f, s0), 0.5f);
  const float e = fmaf(l * -0x1p-23f, s, fmaf(-h, s, 1.0f));
  const uint32_t v = qd_round((s * e) * 0x1p53f);
  const uint32_t sb = qd_bits(s);
  const uint64_t r = (((uint64_t)((sb >> 3) + 0x38000000u) << 32) | (uint32_t)(sb << 29)) + v;
  return bits_dbl((uint32_t)(r >> 32) + 0x3ff00000u - (hi & 0x7ff00000u), (uint32_t)r);
}

// 2^-400 <= x < 2^400 by the high word (no NaN, negative number or subnormal)
ASORA_HD bool qd_middle(uint32_t hi) { return hi - 0x26f00000u < 0x32000000u; }

#ifdef __CUDACC__
static __host__ __device__ __noinline__ double plain_div(double a, double b) { return a / b; }
#else
inline double plain_div(double a, double b) { return a / b; }
#endif

ASORA_HD double quick_div(double a, double b) {
  const uint64_t ab = dbl_bits(a), bb = dbl_bits(b);
  if (!(qd_middle((uint32_t)(bb >> 32)) && (qd_middle((uint32_t)(ab >> 32)) || ab == 0)))
    return plain_div(a, b);
  const double r = recip41((uint32_t)(bb >> 32), (uint32_t)bb);
  const double q = a * r;
  return fma(fma(-b, q, a), r, q);
}

ASORA_HD double quick_recip(double b) {
  const uint64_t bb = dbl_bits(b);
  if (!qd_middle((uint32_t)(bb >> 32))) return plain_div(1.0, b);
  const double r = recip41((uint32_t)(bb >> 32), (uint32_t)bb);
  return fma(fma(-b, r, 1.0), r, r);
}

// The quotients rounded correctly, as a / b gives them.  With q the first approximation, t its
// remainder and r the reciprocal, q + t r is within 2^-29 ulp of the quotient, so its rounding
// can only be wrong next to a tie: where x = |t r| in units of ulp(q) is close to halfway between
// whole numbers.  x < 2^12 is formed from 32 bits of t and r each, beside the last FP64 step:
// frac is its fraction, too low by less than 2^16 of 2^32.  q within 2^12 ulps of a power of
// two counts as close to a tie as well: the rounded quotient may have another ulp.
// Batched rates with optical-depth weights (128^3, 2e3 sources; with rates everywhere; 58^3,
// two sources), quick_div / these / the exact remainder of the rounded quotient instead of x:
// 2.51 / 2.52 / 2.59 ms, 7.38 / 7.43 / 8.74 ms, 144 / 148 / 164 us.
ASORA_HD uint32_t qd_top32(uint64_t x) { return 0x80000000u | (uint32_t)(x >> 21); }

ASORA_HD bool qd_near_tie(double q, double t, double r) {
  const uint64_t qb = dbl_bits(q), tb = dbl_bits(t), rb = dbl_bits(r);
  const uint32_t p = (uint32_t)(((uint64_t)qd_top32(tb) * qd_top32(rb)) >> 32);
  const int k = ((int)(tb >> 52) & 0x7ff) + (int)(rb >> 52) - (int)(qb >> 52) - 1023 + 52;
  const uint32_t frac = (uint32_t)shr64((uint64_t)p << 16, 14 - k);  // x = p 2^(k - 30)
  const bool edge = ((qb + 4096) & 0xfffffffffffffull) < 8192;
  return edge || frac - 0x7ffe0000u < 0x40000u;
}

ASORA_HD double exact_div(double a, double b) {
  const uint64_t ab = dbl_bits(a), bb = dbl_bits(b);
  if (!(qd_middle((uint32_t)(bb >> 32)) && qd_middle((uint32_t)(ab >> 32)))) return plain_div(a, b);
  const double r = recip41((uint32_t)(bb >> 32), (uint32_t)bb);
  const double q = a * r;
  const double t = fma(-b, q, a);
  return qd_near_tie(q, t, r) ? plain_div(a, b) : fma(t, r, q);
}

ASORA_HD double exact_recip(double b) {
  const uint64_t bb = dbl_bits(b);
  if (!qd_middle((uint32_t)(bb >> 32))) return plain_div(1.0, b);
  const double r = recip41((uint32_t)(bb >> 32), (uint32_t)bb);
  const double t = fma(-b, r, 1.0);
  return qd_near_tie(r, t, r) ? plain_div(1.0, b) : fma(t, r, r);
}

}  // namespace asora
