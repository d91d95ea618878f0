// HJ-WENO5 upwind differences in 64-bit integer arithmetic.
//
// This GPU issues an FP64 warp instruction once per 16 to 19 cycles per SM
// (measured: DFMA 16.0, DADD 19.1), a 32 x 32 + 64 bit multiply-add once per
// 0.55 and a 64-bit add once per 0.5.  The level-set stages are bound by FP64
// issue, and the WENO5 weights are what they issue, so these run on the
// integer pipe, at more than FP64 precision:
//   * phi enters as F = phi 2^S with S = 54 - floor(log2 h) (h 2^S lies in
//     [2^54, 2^55)), rounded once: exact for |phi| >= h / 4, off by at most
//     half a unit 2^-S <= 2^-54 h below.  Differences are then exact, where
//     FP64 rounds them to 2^-53 of their size (about h).
//   * the squared smoothness terms s_k are exact 128-bit integers, their
//     squares, pairwise products and the quotient 64-bit mantissas: the
//     weights carry an error below 2^-53, against about 20 roundings of
//     2^-53 in the FP64 form, and the result one of a few units.
// Only differences enter the arithmetic: it covers adjacent differences in
// [-2^57, 2^57) units (at least 4h) of values below 2^61 units (at least 64h,
// FIX_KMAX; where phi is not clamped, the stencil of a tube node reaches 10h).
// Axes with larger differences go through the same arithmetic in larger units
// (weno_steep12), values out of range through the FP64 form.  With values limited to 2^58 units (8h
// to 16h) 91% of the warps of a 200^3 grid with an unclamped phi took both: an
// advancing launch 1430 us, a reinitialising one 16.4 ms, against 870 us and 3.77 ms.
#pragma once
#include "int64math.cuh"

namespace etd {

struct WenoInt {
  int eh;            // floor(log2 h)
  u64 e4hi, e4lo;    // (3/4) eps' 2^2S = 3e-6 (h 2^S)^2, 128 bits
  double unit;       // 2^-S
  double scale;      // 2^-S / (12 h): the gradient from 12 times itself in units
  float epsf;        // (3/4) eps' in units of 2^eh, squared
};

constexpr i64 FIX_OUT = 1ll << 62;  // stored for a value out of range (either sign)
constexpr int FIX_KMAX = 6;                 // the stages take |phi| < 2^7 2^eh
constexpr unsigned FIX_OWN_HI = 1u << 29;   // |F| < 2^61
constexpr unsigned FIX_DIFF_HI = 1u << 25;  // |difference| < 2^57

inline WenoInt weno_int(double h, double eps) {
  WenoInt w;
  u64 b;
  memcpy(&b, &h, 8);
  w.eh = (int)((b >> 52) & 0x7ff) - 1023;
  if (w.eh < -900 || w.eh > 900) {  // near the ends of the exponent range: nothing is in range
    w.eh = -4000;
    w.e4hi = w.e4lo = 0;
    w.unit = 0.0;
    w.scale = 0.0;
    w.epsf = 0.f;
    return w;
  }
  const u64 one = (b & 0xfffffffffffffull) | (1023ull << 52);
  double m;
  memcpy(&m, &one, 8);  // h = m 2^eh, 1 <= m < 2
  const double e4 = 3.0 * eps * m * m * 18014398509481984.0;  // times 2^54; the other 2^54 below
  w.epsf = (float)(3.0 * eps * m * m);
  const u64 i = (u64)e4;
  w.e4hi = i >> 10;  // e4 2^54 = i 2^54: bits 54 and up
  w.e4lo = i << 54;
  // the fraction of e4 (i holds about 36 bits of its 53)
  w.e4lo += (u64)((e4 - (double)i) * 18014398509481984.0);
  const u64 sb = (u64)(1023 + w.eh - 54) << 52;
  double s;
  memcpy(&s, &sb, 8);  // 2^-S
  w.unit = s;
  w.scale = s / (12.0 * h);
  return w;
}

// phi 2^S as a 64-bit integer, to nearest; FIX_OUT with phi's sign when
// |phi| >= 2^(kmax + 1) 2^eh (kmax <= FIX_KMAX), infinite or NaN.
ETD_HD i64 to_fix(double f, int eh, int kmax = 3) {
#ifdef __CUDA_ARCH__
  const u64 b = (u64)__double_as_longlong(f);
#else
  u64 b;
  memcpy(&b, &f, 8);
#endif
  const int k = (int)((b >> 52) & 0x7ff) - 1023 - eh;
  const i64 sg = (i64)b >> 63;
  if (k > kmax) return (FIX_OUT ^ sg) - sg;
  const int r = 7 - k;  // the mantissa times 2^9, shifted right by r >= 1
  if (r > 62) return 0;
  const u64 m = ((b & 0xfffffffffffffull) | 0x10000000000000ull) << 9;
  const i64 v = (i64)((m + (1ull << (r - 1))) >> r);
  return (v ^ sg) - sg;
}

// |x| as far as its upper word decides: the word, complemented if negative
ETD_HD unsigned hi_mag(i64 x) {
  const int h = (int)hi32((u64)x);
  return (unsigned)(h ^ (h >> 31));
}
// The six differences of seven values; returns a bound of their magnitudes, which
// the integer form takes below FIX_DIFF_HI.  A value out of range (FIX_OUT)
// differs by 2^61 or more from every one in range and from FIX_OUT of the other
// sign: beside a node's own value (FIX_OWN_HI) the differences decide.
ETD_HD unsigned fix_diffs(const i64 (&F)[7], i64 (&q)[6]) {
  unsigned big = 0;
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < 6; ++i) {
    q[i] = (i64)((u64)F[i + 1] - (u64)F[i]);
    big |= hi_mag(q[i]);
  }
  return big;
}

// 2^126 / w for w in [2^62, 2^63), to about 2^-58: a single-precision
// reciprocal r0 of the leading bits, then r0 (1 + e + e^2) with
// e = 1 - w r0 (|e| < 2^-21).
ETD_HD u64 recip_u(u64 w) {
  const unsigned wh = hi32(w);
  float f, rf;
  const unsigned fb = 0x3f000000u | ((wh - 0x40000000u) >> 7);  // w 2^-63, truncated
#ifdef __CUDA_ARCH__
  f = __uint_as_float(fb);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rf) : "f"(f));
#else
  memcpy(&f, &fb, 4);
  rf = 1.0f / f;
#endif
  const unsigned r0 = seed_bits(rf);
  // w r0 2^-32, about 2^62: p = w r0 >> 32 as 64 bits
  const u64 p = wide(hi32(w), r0, wide(lo32(w), r0) >> 32);
  const i64 e = (i64)((1ull << 62) - p);  // e 2^62, |e| < 2^42
  const int eh = (int)(e >> 16);          // e 2^46, below 2^26
  const i64 e1 = e + (((i64)eh * eh) >> 30);  // (e + e^2) 2^62
  // r0 2^32 (1 + e1 2^-62), with |e1| < 2^42: r0 e1 2^-30 in two parts
  const i64 c = ((i64)r0 * (int)(e1 >> 16) + (i64)(wide(r0, (unsigned)e1 & 0xffffu) >> 16)) >> 14;
  return ((u64)r0 << 32) + (u64)c;
}

// 12 Phi(a, b, c, d) of Jiang & Peng's form (levelset.cu, weno5_terms) from
// second differences in units 2^-S:
//   12 Phi = (4 A X + V Y) / W,  A = d1 d2, B = d0 d2, C = d0 d1,
//   W = A + 6 B + 3 C, V = 3 C - A - 6 B, X = a - 2b + c, Y = b - 2c + d,
//   d_k = s_k^2,  s_0 = 4 (a-b)^2 + 3 b (2b-a), s_1 = 4 (b-c)^2 + 3 b c,
//   s_2 = 4 (c-d)^2 + 3 c (2c-d), each plus 3/4 eps':
// 3/4 of eps' + (13/3) t^2 + m^2, with 13 t^2 + 3 m^2 = 16 t^2 + 3 (m-t)(m+t).
ETD_HD i64 weno_phi12(i64 a, i64 b, i64 c, i64 d, const WenoInt& k) {
  const U128 e4{k.e4hi, k.e4lo};
  const i64 t0 = a - b, t1 = b - c, t2 = c - d;
  int z0, z1, z2;
  const u64 s0 = normalise(add128(add128(sq128(2 * t0), mul128(3 * b, 2 * b - a)), e4), z0);
  const u64 s1 = normalise(add128(add128(sq128(2 * t1), mul128(3 * b, c)), e4), z1);
  const u64 s2 = normalise(add128(add128(sq128(2 * t2), mul128(3 * c, 2 * c - d)), e4), z2);
  // squares, normalised; y_k: the larger, the smaller s_k
  u64 d0 = sqhi_u(s0), d1 = sqhi_u(s1), d2 = sqhi_u(s2);
  const int b0 = (i64)d0 >= 0, b1 = (i64)d1 >= 0, b2 = (i64)d2 >= 0;
  d0 <<= b0;
  d1 <<= b1;
  d2 <<= b2;
  const int y0 = 2 * z0 + b0, y1 = 2 * z1 + b1, y2 = 2 * z2 + b2;
  const int y01 = y0 > y1 ? y0 : y1;
  const int ym = (y01 > y2 ? y01 : y2) + 5;
  u64 A = shr_sat(mulhi_u(d1, d2), ym - y0);
  const u64 B = shr_sat(mulhi_u(d0, d2), ym - y1), C = shr_sat(mulhi_u(d0, d1), ym - y2);
  const u64 AB = A + 6 * B, C3 = 3 * C;
  u64 W = AB + C3;       // in [2^57, 2^62.4)
  i64 V = (i64)(C3 - AB);
  const int n = clz32(hi32(W)) - 1;
  W <<= n;
  A <<= n;
  V = (i64)((u64)V << n);
  // (4 A X + V Y) 2^-62, then the quotient
  const i64 X = t0 - t1, Y = t1 - t2;
  const U128 p = add128(mul128((i64)A, 4 * X), mul128(V, Y));
  const i64 N = (i64)(p.hi << 2 | p.lo >> 62);
  const i64 sg = N >> 63;
  const u64 q = mulhi_u((u64)((N ^ sg) - sg), recip_u(W));  // |N| 2^126 / W 2^-64
  return ((i64)q ^ sg) - sg;
}

// max(d, 0)-style upwind value of one axis, 12 max(d-, -d+, 0) for outward
// motion (positive) or its mirror image, from the six differences q (units
// 2^-S; of no use where they are out of range).  Only one side's weights are
// evaluated: the larger of the two candidates a, b is decided on a
// single-precision estimate of a - b = +-(d- + d+), whose error stays below
// `tol` (the second differences enter truncated to 2^-22 2^eh, which moves a
// weight by up to 0.3%: 5.1 2^-22 / sqrt(3e-6) per s_k, four-fold in the
// quotient, rounded up to tolf = 2^-7 of the terms it multiplies); where that
// does not decide, both sides are evaluated.  Equal values (all second
// differences 0) need no decision.
ETD_HD i64 weno_axis(const i64 (&q)[6], bool positive, const WenoInt& k, float tolf = 0x1p-7f) {
  const float epsf = k.epsf;
  i64 e[5];
#ifdef __CUDA_ARCH__
#pragma unroll
#endif
  for (int i = 0; i < 5; ++i) e[i] = q[i + 1] - q[i];
  const i64 cen = 7 * (q[2] + q[3]) - (q[1] + q[4]);
  // the estimate, in units of 2^eh (f = 2^-22 leading words)
  const float f0 = (float)(int)hi32((u64)e[0]) * 0x1p-22f, f1 = (float)(int)hi32((u64)e[1]) * 0x1p-22f,
              f2 = (float)(int)hi32((u64)e[2]) * 0x1p-22f, f3 = (float)(int)hi32((u64)e[3]) * 0x1p-22f,
              f4 = (float)(int)hi32((u64)e[4]) * 0x1p-22f;
  const float ta = f0 - f1, tb = f1 - f2, tc = f2 - f3, td = f4 - f3;
  const float Y = tb - tc, X0 = ta - tb, X1 = td + tc;
  // s_k as in weno_phi12, eps' scaled to match
  const float sb = fmaf(4.f * tb, tb, epsf), sc = fmaf(4.f * tc, tc, epsf);
  const float bc = 3.f * f1, cd = 3.f * f3;
  const float m0 = fmaf(4.f * ta, ta, fmaf(bc, 2.f * f1 - f0, epsf)), m1 = fmaf(bc, f2, sb),
              m2 = fmaf(3.f * f2, 2.f * f2 - f3, sc);
  const float p0 = fmaf(4.f * td, td, fmaf(cd, 2.f * f3 - f4, epsf)), p1 = fmaf(cd, f2, sc),
              p2 = fmaf(3.f * f2, 2.f * f2 - f1, sb);
  const auto phi = [](float s0, float s1, float s2, float X, float Yv) {
    const float d0 = s0 * s0, d1 = s1 * s1, d2 = s2 * s2;
    const float A = d1 * d2, AB = fmaf(6.f, d0 * d2, A), C3 = 3.f * (d0 * d1);
#ifdef __CUDA_ARCH__
    return __fdividef(fmaf(4.f * A, X, (C3 - AB) * Yv), AB + C3);
#else
    return fmaf(4.f * A, X, (C3 - AB) * Yv) / (AB + C3);
#endif
  };
  const float D = 2.f * ((float)(int)hi32((u64)cen) * 0x1p-22f) - phi(m0, m1, m2, X0, Y) + phi(p0, p1, p2, X1, Y);
  const float tol = fmaf(tolf, 4.f * (fabsf(X0) + fabsf(X1)) + 2.f * fabsf(Y), 0x1p-14f);
  const bool flat = (e[0] | e[1] | e[2] | e[3] | e[4]) == 0;  // d- = d+ = cen / 12
  bool minus = (flat ? cen > 0 : D > 0.f) == positive;
  bool both = !flat && !(fabsf(D) > tol);
  i64 best = 0;
  for (;;) {
    const i64 ph = weno_phi12(minus ? e[0] : e[4], minus ? e[1] : e[3], e[2], minus ? e[3] : e[1], k);
    const i64 v = minus ? cen - ph : -cen - ph;  // 12 d- or -12 d+
    const i64 w = positive ? v : -v;
    best = w > best ? w : best;
    if (!both) break;
    both = false;
    minus = !minus;
  }
  return best;
}

// 12 h max(d-, -d+, 0) or its mirror image where the differences (bound `big`,
// fix_diffs) of values in range may leave weno_axis's range: the same in units
// 2^(s-S) in which they fit, so that they are rounded by 2^-57 of the largest at
// most (eps' enters the side's estimate smaller by 2^2s, its truncation 2^s times
// as large): an error below the FP64 form's, but beside a kink that only the
// stencil's far end sees (to 1e-15 of the gradient), and a call's result is as far
// from extended precision as with the FP64 form.  Such nodes are those of a phi
// far from a distance, until it is reinitialised, and their neighbours.  Steps on
// phi = slope (r - R) in 3D, with the FP64 form after the integer one for such
// nodes / with this / with the FP64 form alone: slope 9 at 200^3 952 / 625 / 782 us,
// slope 20 at 160^3 685 / 447 / 594 us, with reinitialisation at 200^3, slope 3 7.66 /
// 3.85 / 6.60 ms, slope 9 5.12 / 3.18 / 3.95 ms.
ETD_HD double weno_steep12(i64 (&q)[6], unsigned big, bool positive, const WenoInt& k) {
  const int z = clz32(big);
  const int s = z < 7 ? 7 - z : 0;  // |q| 2^-s < 2^57; s <= 5 (values in range: z >= 2)
  if (s > 0) {
    const i64 half = 1ll << (s - 1);
    for (int i = 0; i < 6; ++i) q[i] = (q[i] + half) >> s;
  }
  WenoInt ks = k;
  const float f = (float)(1 << s);
  if (s > 0) {
    ks.e4lo = k.e4lo >> (2 * s) | k.e4hi << (64 - 2 * s);
    ks.e4hi = k.e4hi >> (2 * s);
    ks.epsf = k.epsf / (f * f);
  }
  return (double)weno_axis(q, positive, ks, 0x1p-7f * f) * (k.unit * (double)(1 << s));
}

// sqrt(acc) 2^-S / (12 h) as a double: acc = x 2^(128 - z), 1/4 <= x < 1, the
// root rounded to 53 bits.
ETD_HD double grad_of(U128 acc, const WenoInt& k) {
  int z = 0;
  if (acc.hi == 0) {
    if (acc.lo == 0) return 0.0;
    acc.hi = acc.lo;
    acc.lo = 0;
    z = 64;
  }
  int z1;
  u64 M = normalise(acc, z1);
  z += z1;
  M >>= z & 1;
  z &= ~1;
  u64 r, gx;  // sqrt(x) 2^63
  root_u(M, r, gx);
  const u64 bits = ((u64)(1085 - (z >> 1)) << 52) + ((gx + 512) >> 10);
  double v;
#ifdef __CUDA_ARCH__
  v = __longlong_as_double((i64)bits);
#else
  memcpy(&v, &bits, 8);
#endif
  return v * k.scale;
}

}  // namespace etd
