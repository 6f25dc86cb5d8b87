// 64-bit integer arithmetic that takes work off the FP64 pipe.
//
// A GB300 SM starts one FP64 warp instruction every 16 clocks (measured: 1.98
// DFMA per clock per SM) while its other pipes accept 64 instructions in the
// same time. A product of two 64-bit mantissas kept to its upper half is 3
// IMAD.WIDE and 2 additions, about 2 clocks per warp; a shift or an addition
// of 64-bit words about 1. So quantities that only need to be accurate, not
// to be IEEE doubles (the WENO5 weights), are carried here as integers with
// more bits than a double's 53, and converted once.
//
// Everything also compiles for the host, for the CPU tests.
#pragma once

#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define JANC_HD __host__ __device__ __forceinline__
#else
#include <math.h>
#define JANC_HD inline
#endif

namespace janc {
namespace soft {

typedef unsigned long long u64;
typedef unsigned int u32;

JANC_HD u32 lo32(u64 x) { return (u32)x; }
JANC_HD u32 hi32(u64 x) { return (u32)(x >> 32); }
JANC_HD u64 bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
JANC_HD double double_of(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

// Shifts by n >= 0 that give 0 for n > 63 (as PTX's do).
JANC_HD u64 shr(u64 x, int n) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? 0 : x >> n;
#endif
}
JANC_HD u64 shl(u64 x, int n) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return n > 63 ? 0 : x << n;
#endif
}

// a b / 2^64, at most 2 below the exact quotient (the product of the low
// words is left out). 3 wide products.
JANC_HD u64 mulhi(u64 a, u64 b) {
  return (u64)hi32(a) * hi32(b) + (((u64)hi32(a) * lo32(b)) >> 32) + (((u64)lo32(a) * hi32(b)) >> 32);
}
// a^2 / 2^64, at most 3 below the exact quotient. 2 wide products.
JANC_HD u64 sqhi(u64 a) {
  const u64 t = ((u64)hi32(a) * lo32(a)) >> 32;
  return (u64)hi32(a) * hi32(a) + t + t;
}

// The float below x (rounded towards zero), as bits. The conversion runs at
// 62 per clock per SM, a count of leading zeros at 16, and the exponent field
// is 158 minus the leading zeros.
JANC_HD u32 float_bits_below(u32 x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(__uint2float_rz(x));
#else
  if (!x) return 0;
  const int z = __builtin_clz(x);
  return ((u32)(158 - z) << 23) | (((x << z) >> 8) & 0x7fffffu);
#endif
}
// Leading zeros of x; 158 for x = 0.
JANC_HD int leading_zeros(u32 x) { return 158 - (int)(float_bits_below(x) >> 23); }

// n 2^e with n in [2^63, 2^64).
struct Num {
  u64 n;
  int e;
};
// x 2^e for x >= 2^32.
JANC_HD Num normal(u64 x, int e) {
  const int z = leading_zeros(hi32(x));
  return Num{shl(x, z), e - z};
}

// x 2^(e - 64) as a double, truncated to 53 bits, for x >= 2^32. No range
// check on the result's exponent.
JANC_HD double to_double(u64 x, int e) {
  const int z = leading_zeros(hi32(x));
  return double_of((shl(x, z) >> 11) + ((u64)(u32)((1021 + e - z) << 20) << 32));
}

// The reciprocal of x >= 2^56 (its upper word fills a float): z = leading zeros of x, result y = 2^127 / (x 2^z)
// within 8 units, in (2^63, 2^64). A float approximation biased down by 2^-21
// (so that it stays below 2 and the remainder is positive), then
// y = y0 (1 + e + e^2) on integers.
JANC_HD u64 recip(u64 x, int* zeros) {
  const u32 fb = float_bits_below(hi32(x));
  const int z = 158 - (int)(fb >> 23);
  const u64 d = shl(x, z);
  const u32 sb = (fb & 0x7f800000u) + (0x800000u - 8u);  // (1 - 2^-21) 2^(32 - z) as a float
  // 2 + y0 in [3, 4): the mantissa field is y0 as Q1.22
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(fb)));
  const u32 y0 = __float_as_uint(__fmaf_rn(r, __uint_as_float(sb), 2.0f)) << 9;
#else
  float fd, sc;
  memcpy(&fd, &fb, 4);
  memcpy(&sc, &sb, 4);
  // the scale's exponent is that of 2^(32 - z), fd's that of 2^(31 - z)
  const float yf = fmaf(1.0f / fd, sc, 2.0f);
  u32 y0;
  memcpy(&y0, &yf, 4);
  y0 <<= 9;
#endif
  const u64 t = (u64)hi32(d) * y0 + (((u64)lo32(d) * y0) >> 32);  // d y0 in units of 2^-63
  u64 e = 0ull - (t << 1);                                        // 1 - d y0 in units of 2^-64, below 2^44
  const u32 es = (u32)(e >> 12);
  e += ((u64)es * es) >> 40;
  *zeros = z;
  return (u64)y0 * hi32(e) + ((u64)y0 << 32) + (((u64)y0 * lo32(e)) >> 32);
}

}  // namespace soft
}  // namespace janc
