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

// a b / 2^64 exactly.
JANC_HD u64 mulhi_exact(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (u64)(((unsigned __int128)a * b) >> 64);
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

// x / 2^n for n >= 0, rounded down.
JANC_HD long long sar(long long x, int n) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(n));
  return r;
#else
  return x >> (n > 63 ? 63 : n);
#endif
}

// a b / 2^64, at most 2 below the exact quotient (the product of the low
// words is left out). 3 wide products.
JANC_HD u64 mulhi(u64 a, u64 b) {
  return (u64)hi32(a) * hi32(b) + (((u64)hi32(a) * lo32(b)) >> 32) + (((u64)lo32(a) * hi32(b)) >> 32);
}
// a^2 / 2^64, at most 1 below the exact quotient. 2 wide products.
JANC_HD u64 sqhi(u64 a) {
  return (u64)hi32(a) * hi32(a) + (((u64)hi32(a) * lo32(a)) >> 31);
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

// 2^127 / d within 8 units for d in [2^63, 2^64), in (2^63, 2^64); fb is the
// float below hi32(d) 2^k, sb (1 - 2^-21) 2^(32 + k), both as bits. A float
// approximation biased down by 2^-21 (so that it stays below 2 and the
// remainder is positive), then y = y0 (1 + e + e^2) on integers.
JANC_HD u64 recip_from(u64 d, u32 fb, u32 sb) {
  // 2 + y0 in [3, 4): the mantissa field is y0 as Q1.22
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(fb)));
  const u32 y0 = __float_as_uint(__fmaf_rn(r, __uint_as_float(sb), 2.0f)) << 9;
#else
  float fd, sc;
  memcpy(&fd, &fb, 4);
  memcpy(&sc, &sb, 4);
  const float yf = fmaf(1.0f / fd, sc, 2.0f);
  u32 y0;
  memcpy(&y0, &yf, 4);
  y0 <<= 9;
#endif
  const u64 t = (u64)hi32(d) * y0 + (((u64)lo32(d) * y0) >> 32);  // d y0 in units of 2^-63
  u64 e = 0ull - (t << 1);                                        // 1 - d y0 in units of 2^-64, below 2^44
  const u32 es = (u32)(e >> 12);
  e += ((u64)es * es) >> 40;
  return (u64)y0 * hi32(e) + ((u64)y0 << 32) + (((u64)y0 * lo32(e)) >> 32);
}
// The reciprocal of x >= 2^56 (its upper word fills a float): z = leading zeros
// of x, result 2^127 / (x 2^z).
JANC_HD u64 recip(u64 x, int* zeros) {
  const u32 fb = float_bits_below(hi32(x));
  const int z = 158 - (int)(fb >> 23);
  *zeros = z;
  return recip_from(shl(x, z), fb, (fb & 0x7f800000u) + (0x800000u - 8u));
}
// The same for a normalised m.
JANC_HD u64 recip_normal(u64 m) {
  return recip_from(m, 0x4f000000u | (hi32(m) >> 8 & 0x7fffffu), 0x4f800000u - 8u);
}

// Tables, each entry rounded from 300-bit values: 2^(j/64) in units of 2^-63;
// c_j = 64 / (64 + j) rounded up, in units of 2^-31; -log2(c_j) in units of 2^-64.
#ifndef __CUDACC__
#define JANC_TABLE static const
#else
#define JANC_TABLE static __device__ const
#endif
JANC_TABLE u64 kExp2[64] = {
    0x8000000000000000ull, 0x8164d1f3bc030773ull, 0x82cd8698ac2ba1d7ull, 0x843a28c3acde4046ull,
    0x85aac367cc487b15ull, 0x871f61969e8d1010ull, 0x88980e8092da8527ull, 0x8a14d575496efd9aull,
    0x8b95c1e3ea8bd6e7ull, 0x8d1adf5b7e5ba9e6ull, 0x8ea4398b45cd53c0ull, 0x9031dc431466b1dcull,
    0x91c3d373ab11c336ull, 0x935a2b2f13e6e92cull, 0x94f4efa8fef70961ull, 0x96942d3720185a00ull,
    0x9837f0518db8a96full, 0x99e0459320b7fa65ull, 0x9b8d39b9d54e5539ull, 0x9d3ed9a72cffb751ull,
    0x9ef5326091a111aeull, 0xa0b0510fb9714fc2ull, 0xa27043030c496819ull, 0xa43515ae09e6809eull,
    0xa5fed6a9b15138eaull, 0xa7cd93b4e965356aull, 0xa9a15ab4ea7c0ef8ull, 0xab7a39b5a93ed337ull,
    0xad583eea42a14ac6ull, 0xaf3b78ad690a4375ull, 0xb123f581d2ac2590ull, 0xb311c412a9112489ull,
    0xb504f333f9de6484ull, 0xb6fd91e328d17791ull, 0xb8fbaf4762fb9ee9ull, 0xbaff5ab2133e45fbull,
    0xbd08a39f580c36bfull, 0xbf1799b67a731083ull, 0xc12c4cca66709456ull, 0xc346ccda24976407ull,
    0xc5672a115506daddull, 0xc78d74c8abb9b15dull, 0xc9b9bd866e2f27a3ull, 0xcbec14fef2727c5dull,
    0xce248c151f8480e4ull, 0xd06333daef2b2595ull, 0xd2a81d91f12ae45aull, 0xd4f35aabcfedfa1full,
    0xd744fccad69d6af4ull, 0xd99d15c278afd7b6ull, 0xdbfbb797daf23755ull, 0xde60f4825e0e9124ull,
    0xe0ccdeec2a94e111ull, 0xe33f8972be8a5a51ull, 0xe5b906e77c8348a8ull, 0xe8396a503c4bdc68ull,
    0xeac0c6e7dd24392full, 0xed4f301ed9942b84ull, 0xefe4b99bdcdaf5cbull, 0xf281773c59ffb13aull,
    0xf5257d152486cc2cull, 0xf7d0df730ad13bb9ull, 0xfa83b2db722a033aull, 0xfd3e0c0cf486c175ull};
JANC_TABLE u32 kLogC[64] = {
    0x80000000u, 0x7e07e07fu, 0x7c1f07c2u, 0x7a44c6b0u, 0x78787879u, 0x76b981dbu, 0x75075076u, 0x73615a25u,
    0x71c71c72u, 0x70381c0fu, 0x6eb3e454u, 0x6d3a06d4u, 0x6bca1af3u, 0x6a63bd82u, 0x6906906au, 0x67b23a55u,
    0x66666667u, 0x6522c3f4u, 0x63e7063fu, 0x62b2e43eu, 0x61861862u, 0x60606061u, 0x5f417d06u, 0x5e293206u,
    0x5d1745d2u, 0x5c0b8171u, 0x5b05b05cu, 0x5a05a05bu, 0x590b2165u, 0x58160582u, 0x572620afu, 0x563b48c3u,
    0x55555556u, 0x54741facu, 0x5397829du, 0x52bf5a82u, 0x51eb851fu, 0x511be196u, 0x50505051u, 0x4f88b2f4u,
    0x4ec4ec4fu, 0x4e04e04fu, 0x4d4873edu, 0x4c8f8d29u, 0x4bda12f7u, 0x4b27ed37u, 0x4a7904a8u, 0x49cd42e3u,
    0x4924924au, 0x487ede05u, 0x47dc11f8u, 0x473c1ab7u, 0x469ee585u, 0x46046047u, 0x456c797eu, 0x44d72045u,
    0x44444445u, 0x43b3d5b0u, 0x4325c53fu, 0x429a042au, 0x42108422u, 0x4189374cu, 0x41041042u, 0x40810205u};
JANC_TABLE u64 kLog2[64] = {
    0x0000000000000000ull, 0x05b9e59e99964173ull, 0x0b5d69ba995434ceull, 0x10eb389ee9f55f8bull,
    0x1663f6f929941161ull, 0x1bc842405ce14082ull, 0x2118b116a4204bc0ull, 0x2655d3c1ec135c85ull,
    0x2b8034733f02d416ull, 0x3098579d2a93ff78ull, 0x359ebc582adb1da9ull, 0x3a93dc972188f80aull,
    0x3f782d7065510f2bull, 0x444c1f6a20193709ull, 0x49101ea8caf44d09ull, 0x4dc49337ea43f940ull,
    0x5269e12d0a6f7a7full, 0x570068e59730de3aull, 0x5b888734614a0f49ull, 0x6002958b2c5cb0a8ull,
    0x646eea22aeb28eedull, 0x68cdd82799cd5e7full, 0x6d1fafdcb3dff3c6ull, 0x7164beb43202f500ull,
    0x759d4f7ea1a98a7full, 0x79c9aa8452ca9a48ull, 0x7dea159f3472f5daull, 0x81fed458b999108cull,
    0x8608280344ac99c4ull, 0x8a064fd271c1067dull, 0x8df988f1b4c23b16ull, 0x91e20e9d07e0c866ull,
    0x95c01a37192d9afdull, 0x9993e353a9111393ull, 0x9d5d9fd3d4f69644ull, 0xa11d83f19b6c8867ull,
    0xa4d3c25d25b2706aull, 0xa8808c36325e5cdaull, 0xac2411319d00db4bull, 0xafbe7f9ef4795316ull,
    0xb3500471274705acull, 0xb6d8cb4f0c0271f9ull, 0xba58feb0e7d0e080ull, 0xbdd0c7c81422bee6ull,
    0xc1404eab9b5a569aull, 0xc4a7ba536489ee67ull, 0xc80730add617b678ull, 0xcb5ed6907ba7fc7eull,
    0xceaecfe62c883842ull, 0xd1f73f9a0d0d128dull, 0xd53847a6f3fefdceull, 0xd8720933828f7ac6ull,
    0xdba4a47798c356eeull, 0xded038e104abe479ull, 0xe1f4e516262ddfa8ull, 0xe512c6e46e4e8b6full,
    0xe829fb65389c6e3bull, 0xeb3a9eff6d51c678ull, 0xee44cd59ba6b8cc4ull, 0xf148a16e5d2096e8ull,
    0xf4463595aa56d9a5ull, 0xf73da38c5a209c64ull, 0xfa2f0458e10b5ffdull, 0xfd1a70863274f451ull};
#undef JANC_TABLE

#ifdef __CUDA_ARCH__
#define JANC_LDG(p) __ldg(p)
#else
#define JANC_LDG(p) (*(p))
#endif

// 2^f for f in units of 2^-64, in units of 2^-63, within 2^-57 of itself:
// f = j/64 + r/64, e^z - 1 = z + z^2 (1/2 + z/6 + z^2 (1/24 + z/120 + z^2/720))
// with z = r ln2 / 64 < 0.0109 (P. T. P. Tang, ACM TOMS 15(2), 1989, with a
// 64-entry table), the inner bracket in 32 bits. About 45 integer instructions.
JANC_HD u64 exp2_frac(u64 f) {
  const u64 t = JANC_LDG(&kExp2[f >> 58]);
  const u64 z = mulhi(f << 6, 0xb17217f7d1cf79acull);                     // units of 2^-70
  const u32 zh = hi32(z);                                        // 2^-38
  const u32 zz = (u32)(((u64)zh * zh) >> 32);                    // z^2, 2^-44
  const u32 g = 2863311531u + (u32)(((u64)zh * 8947849u) >> 32) + (u32)(((u64)zz * 23302u) >> 32);  // 2^-36
  const u64 h = (1ull << 63) + mulhi(z, 0x00aaaaaaaaaaaaabull) + (((u64)zz * g) >> 16);
  const u64 p = z + (mulhi(sqhi(z), h) >> 6);                    // e^z - 1, 2^-70
  return t + (mulhi(t, p) >> 6);
}

// log2(m / 2^63) of m in [2^63, 2^64), in units of 2^-64, within 2^-58:
// m c_j = 1 + r with r in [0, 1/64 + 2^-30), log(1 + r) = r - r^2 (1/2 - r/3 +
// r^2 (1/4 - r/5 + ..)), the inner bracket in 32 bits.
JANC_HD u64 log2_frac(u64 m) {
  const u32 j = hi32(m) >> 25 & 63u;
  const u32 c = JANC_LDG(&kLogC[j]);
  const u64 r = ((u64)hi32(m) * c + (((u64)lo32(m) * c) >> 32) - (1ull << 62)) << 7;  // units of 2^-69
  const u32 rh = hi32(r);                                        // 2^-37
  const u64 rr = sqhi(r);                                        // r^2, 2^-74
  const u32 r2 = hi32(rr);                                       // 2^-42
  // 1/4 - r/5 + r^2/6 - r^3/7 + r^4/8 - r^5/9 in units of 2^-33
  u32 k = 1073741824u - (u32)(((u64)rh * 29826162u) >> 32);      // 1/8 - r/9
  k = 1227133513u - (u32)(((u64)rh * k) >> 37);                  // 1/7 - r ()
  k = 1431655765u - (u32)(((u64)rh * k) >> 37);
  k = 1717986918u - (u32)(((u64)rh * k) >> 37);
  k = 2147483648u - (u32)(((u64)rh * k) >> 37);
  // r^2 (1/2 - r/3 + r^2 k): the bracket in units of 2^-64
  const u64 h = (1ull << 63) - mulhi(r, 0x02aaaaaaaaaaaaabull) + ((((u64)r2 * k) + (((u64)lo32(rr) * k) >> 32)) >> 11);
  const u64 l = r - (mulhi(rr, h) >> 5);                         // log(1 + r), 2^-69
  return JANC_LDG(&kLog2[j]) + (mulhi(l, 0xb8aa3b295c17f0bcull) >> 4);     // log2 e in units of 2^-63
}

// a b / 2^64 for signed b, at most 3 below the exact quotient.
JANC_HD long long mulhi_signed(u64 a, long long b) {
  return (long long)(mulhi(a, (u64)b) - (b < 0 ? a : 0ull));
}

// |x| = m 2^(e - 1086) with m in [2^63, 2^64), for a normal double.
struct Parts {
  u64 m;
  int e;
  bool neg;
  JANC_HD explicit Parts(double x) {
    const u64 b = bits_of(x);
    e = (int)(hi32(b) >> 20) & 0x7ff;
    m = (b << 11) | (1ull << 63);
    neg = (int)hi32(b) < 0;
  }
};
// m 2^(e - 63), m in [2^63, 2^64), rounded to the nearest double (ties up).
JANC_HD double round_double(u64 m, int e) {
  return double_of((m >> 11) + ((m >> 10) & 1) + ((u64)(u32)((1022 + e) << 20) << 32));
}

// x cut to a float, 0 below a float's normal range; no check above it. And a
// float as a double (2^-127 for 0). (The conversion instructions occupy the FP64 pipe.)
JANC_HD float cut_float(double x) {
  const u64 b = bits_of(x);
  const u32 a = hi32(b) & 0x7fffffffu, n = a - 0x38000000u;
  u32 f = (n << 3 | lo32(b) >> 29) | (hi32(b) & 0x80000000u);
  if (a < 0x38100000u) f = 0;
#ifdef __CUDA_ARCH__
  return __uint_as_float(f);
#else
  float r;
  memcpy(&r, &f, 4);
  return r;
#endif
}
JANC_HD double widen(float x) {
#ifdef __CUDA_ARCH__
  const u32 f = __float_as_uint(x);
#else
  u32 f;
  memcpy(&f, &x, 4);
#endif
  return double_of(((u64)((((f & 0x7fffffffu) >> 3) + 0x38000000u) | (f & 0x80000000u)) << 32) | (u64)(f << 29));
}

// 1/x for normal x of either sign, correctly rounded but for near ties; 0
// beyond 2^1021, NaN for 0, denormals, infinities and NaN.
JANC_HD double rcp_double(double x) {
  const Parts p(x);
  const double r = round_double(recip_normal(p.m), 1022 - p.e);
  u32 h = hi32(bits_of(r)) | (p.neg ? 0x80000000u : 0u);
  u32 l = lo32(bits_of(r));
  if (p.e >= 2045) h = l = 0;
  if (p.e == 0 || p.e == 2047) h = 0x7ff80000u;
  return double_of(((u64)h << 32) | l);
}

// e^x for |x| < 708, within 0.6 units in the last place (the exponent in
// units of 2^-54, the power of two to 2^-57).
JANC_HD double exp_double(double x) {
  const Parts p(x);
  // |x| log2 e in units of 2^-54: log2 e = 0xb8.. 2^-63
  constexpr u64 kLog2e = 0xb8aa3b295c17f0bcull;
  u64 a = mulhi_exact(p.m, kLog2e);
  a = p.e > 1031 ? (a << 1) + ((p.m * kLog2e) >> 63) : shr(a, 1031 - p.e);
  int k = (int)(a >> 54);
  if (p.neg && a) {
    a = 0ull - a;
    k = (int)(a >> 54) - 1024;
  }
  return round_double(exp2_frac(a << 10), k);
}

// 2^(a 2^-54), within 0.6 units in the last place.
JANC_HD double exp2_fixed(long long a) { return round_double(exp2_frac((u64)a << 10), (int)(a >> 54)); }

// ln x for x in [2, 2^1023), within 2^-53 before the rounding to nearest.
JANC_HD double log_double(double x) {
  const Parts p(x);
  // log2 x in units of 2^-54, then ln 2 = 0xb1.. 2^-64
  const u64 a = mulhi_exact(((u64)(p.e - 1023) << 54) + (log2_frac(p.m) >> 10), 0xb17217f7d1cf79acull);
  const Num n = normal(a, 0);
  return round_double(n.n, n.e + 9);
}

// a 2^e rounded to nearest, 0 for a = 0. No range check on the exponent.
JANC_HD double signed_double(long long a, int e) {
  const u64 m = a < 0 ? 0ull - (u64)a : (u64)a;
  u32 h = hi32(m), l = lo32(m);
  if (h == 0) {
    h = l;
    l = 0;
    e -= 32;
  }
  const int z = leading_zeros(h);
  const u64 b = bits_of(round_double(shl(((u64)h << 32) | l, z), e - z + 63));
  return a == 0 ? 0.0 : double_of(((u64)(hi32(b) | (a < 0 ? 0x80000000u : 0u)) << 32) | lo32(b));
}

// a 2^e rounded to nearest, 0 below the normal range. No check against overflow.
JANC_HD double scaled_double(long long a, int e) {
  u64 m = a < 0 ? 0ull - (u64)a : (u64)a;
  if (hi32(m) == 0) {
    m <<= 32;
    e -= 32;
  }
  const int z = leading_zeros(hi32(m));  // 158 for 0
  const int x = 1085 + e - z;
  m = shl(m, z);
  const u64 b = (m >> 11) + ((m >> 10) & 1) + ((u64)((u32)x << 20 | ((u32)hi32((u64)a) & 0x80000000u)) << 32);
  return double_of(x < 0 || m == 0 ? 0ull : b);
}

// sqrt(d / 2^64) for d in [2^62, 2^64), in units of 2^-64, within 2^-60: a float
// seed biased down, then two Newton steps on the exact remainder.
JANC_HD u64 sqrt_q(u64 d) {
#ifdef __CUDA_ARCH__
  const float f = __fmul_rn(__uint2float_rz(hi32(d)), 0x1p-32f);  // [1/4, 1)
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  const u32 s0 = __float_as_uint(__fmaf_rn(__fmul_rn(f, r), 1.0f - 0x1p-21f, 1.0f)) << 9;  // 1 + s in [1.5, 2)
  const u32 rr = __float_as_uint(__fmaf_rn(r, 1.0f - 0x1p-21f, 2.0f)) << 9;                // 2 + r in [3, 4)
#else
  const float f = (float)hi32(d & ~0xffffffffffull) * 0x1p-32f, r = 1.0f / sqrtf(f);
  const float sf = fmaf(f * r, 1.0f - 0x1p-21f, 1.0f), rf = fmaf(r, 1.0f - 0x1p-21f, 2.0f);
  u32 s0, rr;
  memcpy(&s0, &sf, 4);
  memcpy(&rr, &rf, 4);
  s0 <<= 9;
  rr <<= 9;
#endif
  // s0: units of 2^-32; rr = 1/s: units of 2^-31
  const u64 e0 = d - (u64)s0 * s0;  // >= 0, below 2^44
  const u64 s1 = ((u64)s0 << 32) + (u64)hi32(e0) * rr + (((u64)lo32(e0) * rr) >> 32);
  const int e1 = (int)(d - sqhi(s1));  // |d - s1^2| < 2^26
  const u32 n1 = e1 < 0 ? 0u - (u32)e1 : (u32)e1;
  const u32 c1 = (u32)(((u64)n1 * rr) >> 32);
  return e1 < 0 ? s1 - c1 : s1 + c1;
}

}  // namespace soft
}  // namespace janc
