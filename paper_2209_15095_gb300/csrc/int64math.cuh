// 64- and 128-bit integer arithmetic for the places where FP64 issue or
// latency bounds a phase (host and device).
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define ETD_HD __host__ __device__ __forceinline__
#else
#define ETD_HD inline
#endif

namespace etd {

typedef unsigned long long u64;
typedef long long i64;

ETD_HD u64 wide(unsigned a, unsigned b, u64 c = 0) { return (u64)a * b + c; }
ETD_HD unsigned hi32(u64 x) { return (unsigned)(x >> 32); }
ETD_HD unsigned lo32(u64 x) { return (unsigned)x; }
ETD_HD int clz32(unsigned x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}
// (h, l) <<< n, the upper word, 0 <= n < 32
ETD_HD unsigned shfl32(unsigned l, unsigned h, int n) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(l, h, n);
#else
  return n ? (h << n) | (l >> (32 - n)) : h;
#endif
}

struct U128 {
  u64 hi, lo;
};
ETD_HD U128 add128(U128 a, U128 b) {
  U128 r;
#ifdef __CUDA_ARCH__
  asm("add.cc.u64 %0, %2, %4;\n\taddc.u64 %1, %3, %5;"
      : "=l"(r.lo), "=l"(r.hi)
      : "l"(a.lo), "l"(a.hi), "l"(b.lo), "l"(b.hi));
#else
  r.lo = a.lo + b.lo;
  r.hi = a.hi + b.hi + (r.lo < a.lo);
#endif
  return r;
}
// t^2, exact
ETD_HD U128 sq128(i64 t) {
  const i64 s = t >> 63;
  const u64 a = (u64)((t ^ s) - s);
  const unsigned h = hi32(a), l = lo32(a);
  const u64 m = wide(h, l);
  return add128(U128{wide(h, h), wide(l, l)}, U128{m >> 31, m << 33});
}
// x y of signed operands, exact (two's complement)
ETD_HD U128 mul128(i64 x, i64 y) {
  const unsigned xh = hi32((u64)x), xl = lo32((u64)x), yh = hi32((u64)y), yl = lo32((u64)y);
  const u64 ll = wide(xl, yl);
  const u64 m1 = wide(xl, yh, ll >> 32);
  const u64 m2 = wide(xh, yl, (u64)lo32(m1));
  u64 hi = wide(xh, yh, m1 >> 32) + (m2 >> 32);
  hi -= (u64)((x >> 63) & y) + (u64)((y >> 63) & x);
  return U128{hi, (m2 << 32) | lo32(ll)};
}
// the upper 64 bits of x y, low by at most 2
ETD_HD u64 mulhi_u(u64 x, u64 y) {
  const u64 m1 = wide(hi32(x), lo32(y)), m2 = wide(lo32(x), hi32(y));
  return wide(hi32(x), hi32(y), m1 >> 32) + (m2 >> 32);
}
ETD_HD u64 sqhi_u(u64 x) {
  const u64 m = wide(hi32(x), lo32(x));
  return wide(hi32(x), hi32(x), m >> 31);
}
ETD_HD u64 shr_sat(u64 x, int n) { return n > 63 ? 0ull : x >> n; }

// leading 64 bits of s >= 2^64 (most significant bit set) and its leading zeros
ETD_HD u64 normalise(U128 s, int& z) {
  const unsigned w3 = hi32(s.hi), w2 = lo32(s.hi), w1 = hi32(s.lo), w0 = lo32(s.lo);
  const bool top = w3 != 0;
  const unsigned a = top ? w3 : w2, b = top ? w2 : w1, c = top ? w1 : w0;
  const int n = clz32(a);
  z = top ? n : n + 32;
  return (u64)shfl32(b, a, n) << 32 | shfl32(c, b, n);
}

// A single-precision seed of a value in (1, 2] as r 2^31, 1 <= r < 2: the
// exponent is dropped, so a seed that ends outside [1, 2) would enter at half
// or twice its value.  The approximations' documented errors (1 ulp of the
// reciprocal, 2^-22.9 of the reciprocal root) allow both sides; a seed moved
// onto the end is within those errors.
ETD_HD unsigned seed_bits(float r) {
  r = fminf(fmaxf(r, 1.0f), 1.9999998f);
#ifdef __CUDA_ARCH__
  const unsigned b = __float_as_uint(r);
#else
  unsigned b;
  memcpy(&b, &r, 4);
#endif
  return (b & 0x7fffffu) << 8 | 0x80000000u;
}

// Reciprocal root and root of x = M 2^-64, 1/4 <= x < 1: r 2^63 and sqrt(x) 2^63,
// to about 2^-60: a single-precision reciprocal root r0, then r = r0 (1 + e/2 +
// 3 e^2 / 8) with e = 1 - x r0^2 (|e| < 2^-21), sqrt(x) = x r.
ETD_HD void root_u(u64 M, u64& r, u64& gx) {
  const unsigned mh = hi32(M);
  const unsigned fb = (mh >> 31) ? 0x3f000000u | ((mh & 0x7fffffffu) >> 8) : 0x3e800000u | ((mh & 0x3fffffffu) >> 7);
  float f, rf;
#ifdef __CUDA_ARCH__
  f = __uint_as_float(fb);
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(f));
#else
  memcpy(&f, &fb, 4);
  rf = 1.0f / sqrtf(f);
#endif
  const unsigned r0 = seed_bits(rf);
  const i64 e = (i64)((1ull << 62) - mulhi_u(M, wide(r0, r0)));  // e 2^62
  const int eh = (int)(e >> 16);
  const i64 e1 = (e >> 1) + ((i64)eh * eh * 3 >> 33);
  const i64 c = ((i64)r0 * (int)(e1 >> 16) + (i64)(wide(r0, (unsigned)e1 & 0xffffu) >> 16)) >> 14;
  r = ((u64)r0 << 32) + (u64)c;
  gx = mulhi_u(M, r);
}

// sqrt(a) and 1 / sqrt(a), each to about an ulp, for a positive normal a; other
// arguments by the FP64 functions.  About 200 cycles where a dependent FP64
// root and division take 1500.
ETD_HD void root_pair(double a, double& s, double& r) {
#ifdef __CUDA_ARCH__
  const u64 b = (u64)__double_as_longlong(a);
#else
  u64 b;
  memcpy(&b, &a, 8);
#endif
  const int be = (int)(b >> 52);
  if (be == 0 || be >= 0x7ff) {  // zero, subnormal, negative, infinite, NaN
    s = sqrt(a);
    r = 1.0 / s;
    return;
  }
  u64 M = (b << 11) | 0x8000000000000000ull;  // a = M 2^-64 2^ex, 1/2 <= M 2^-64 < 1
  int ex = be - 1022;
  if (ex & 1) {
    M >>= 1;
    ex += 1;
  }
  ex /= 2;
  u64 y, gx;
  root_u(M, y, gx);
  const u64 sb = ((u64)(1021 + ex) << 52) + ((gx + 512) >> 10);
  const u64 rb = ((u64)(1022 - ex) << 52) + (y >> 11) + ((y >> 10) & 1);
#ifdef __CUDA_ARCH__
  s = __longlong_as_double((i64)sb);
  r = __longlong_as_double((i64)rb);
#else
  memcpy(&s, &sb, 8);
  memcpy(&r, &rb, 8);
#endif
}

}  // namespace etd
