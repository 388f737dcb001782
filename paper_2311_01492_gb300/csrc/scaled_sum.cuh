// Sums of non-negative doubles on the integer units (rates.cu).  Plain C++ as well, so
// that the arithmetic can be checked on the host.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define ASORA_HD __host__ __device__ __forceinline__
#else
#define ASORA_HD inline
#endif

namespace asora {

// A sum of doubles (hi:lo) 2^(e/2^20 - 1023 - 61): the leading bit is bit 61 (or 62
// after a carry), e the biased exponent in place (bits 20..30).
struct PairSum {
  uint32_t lo, hi, e;
};

ASORA_HD uint64_t dbl_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
#endif
}

ASORA_HD double bits_dbl(uint32_t hi, uint32_t lo) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((int)hi, (int)lo);
#else
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

ASORA_HD uint64_t shr64(uint64_t x, uint32_t d) {  // 0 for d >= 64
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));
  return r;
#else
  return d < 64 ? x >> d : 0;
#endif
}

// Mantissa of x with its leading bit at bit 61 (nine guard bits below the last).  Zero
// is taken as 2^-1022: far below the last bit of anything it is added to.
ASORA_HD uint64_t mantissa61(uint32_t hi, uint32_t lo) {
  return (((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo) << 9;
}

// x + y for finite x, y >= +0, cut at the guard bits.
ASORA_HD PairSum pair_sum(double x, double y) {
  const uint64_t xb = dbl_bits(x), yb = dbl_bits(y);
  const uint32_t xh = (uint32_t)(xb >> 32), xl = (uint32_t)xb;
  const uint32_t yh = (uint32_t)(yb >> 32), yl = (uint32_t)yb;
  const bool sw = yh > xh;
  const uint32_t H = sw ? yh : xh, L = sw ? xh : yh, hl = sw ? yl : xl, ll = sw ? xl : yl;
  const uint32_t e = H & 0x7ff00000u;
  const uint32_t d = (e - (L & 0x7ff00000u)) >> 20;
  const uint64_t s = mantissa61(H, hl) + shr64(mantissa61(L, ll), d);
  return {(uint32_t)s, (uint32_t)(s >> 32), e};
}

// x + y rounded to the nearest double (ties to even), x a double >= +0.
ASORA_HD double round_sum(double x, const PairSum& y) {
  const uint64_t xb = dbl_bits(x);
  const uint32_t xh = (uint32_t)(xb >> 32), xl = (uint32_t)xb;
  const uint32_t xe = xh & 0x7ff00000u;
  const uint64_t A = mantissa61(xh, xl);
  const uint64_t B = ((uint64_t)y.hi << 32) | y.lo;
  const bool sw = y.e > xe;
  const uint32_t e = sw ? y.e : xe, f = sw ? xe : y.e;
  const uint64_t X = sw ? B : A, Y = sw ? A : B;
  const uint64_t v = X + shr64(Y, (e - f) >> 20);
  const uint32_t vh = (uint32_t)(v >> 32), vl = (uint32_t)v;
  const uint32_t top = vh >> 30;  // leading bit 61, 62 or 63
  const uint32_t inc = top < 2u ? top : 2u;
  const uint32_t sh = 9 + inc;
  const uint32_t g = vl << (32 - sh);             // the bits cut off, left-aligned
  const uint32_t exp = e + (inc << 20) - 0x100000u;  // (the hidden bit adds one)
#ifdef __CUDA_ARCH__
  const uint32_t ql = __funnelshift_r(vl, vh, sh), qh = vh >> sh;
  const uint32_t half = (ql & 1) + 0x7fffffffu;
  uint32_t rl, rh;
  asm("{\n\t.reg .u32 c;\n\t"
      "add.cc.u32 c, %2, %3;\n\t"
      "addc.cc.u32 %0, %4, 0;\n\t"
      "addc.u32 %1, %5, %6;\n\t}"
      : "=r"(rl), "=r"(rh)
      : "r"(g), "r"(half), "r"(ql), "r"(qh), "r"(exp));
  return bits_dbl(rh, rl);
#else
  uint64_t q = v >> sh;
  q += ((uint64_t)g + 0x7fffffffu + (uint32_t)(q & 1)) >> 32;
  return bits_dbl((uint32_t)(q >> 32) + exp, (uint32_t)q);
#endif
}

}  // namespace asora
