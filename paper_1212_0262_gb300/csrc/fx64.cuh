// Reciprocals and products of doubles on the integer pipe, and 96-bit fixed-point sums.
//
// GB300 issues about 2 FP64 operations per SM and clock, against 64 32 x 32 -> 64 bit
// multiply-adds and 128 integer adds (measured: mad.wide.u32 60, add 120, DFMA 1.9 per SM
// and clock): an FP64 operation costs as much issue time as some 30 multiply-adds.  The
// FP64 pair kernels therefore keep on the FP64 pipe only the coordinate differences (and
// those of w and the dot products of the 2D reverse stages) and do the rest on mantissas held as
// integers.  A term has a relative error below 2^-54 (noted at each function) and is truncated
// at the unit of its sum, which the policies choose (pairs_fx.cuh); the sums themselves are exact.
//
// The header has no GPU-only constructs but the reciprocal seed and the carry chain, so
// that the CPU tests compile it and check it against extended precision.
#pragma once
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN static inline
#endif

namespace fx64 {

typedef uint32_t u32;
typedef uint64_t u64;

FX_FN float as_float(u32 b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  memcpy(&f, &b, 4);
  return f;
#endif
}
FX_FN u32 as_uint(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  u32 b;
  memcpy(&b, &f, 4);
  return b;
#endif
}
FX_FN u32 hi_word(double d) {
#ifdef __CUDA_ARCH__
  return (u32)__double2hiint(d);
#else
  u64 b;
  memcpy(&b, &d, 8);
  return (u32)(b >> 32);
#endif
}
FX_FN u32 lo_word(double d) {
#ifdef __CUDA_ARCH__
  return (u32)__double2loint(d);
#else
  u64 b;
  memcpy(&b, &d, 8);
  return (u32)b;
#endif
}
FX_FN u64 mul_wide(u32 a, u32 b, u64 c) { return (u64)a * b + c; }
FX_FN u32 shf_r(u32 lo, u32 hi, int k) {  // (hi:lo) >> k, low word, 0 <= k < 32
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, k);
#else
  return (u32)((((u64)hi << 32) | lo) >> k);
#endif
}
FX_FN u32 shf_l(u32 lo, u32 hi, int k) {  // (hi:lo) << k, high word, 0 <= k < 32
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, k);
#else
  return (u32)(((((u64)hi << 32) | lo) << k) >> 32);
#endif
}

// Seed of 1/f for f in [1, 2): relative error below 2^-22, result in (0.5, 1).
FX_FN float seed_rcp(float f) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
#else
  float r = 1.0f / f;
#endif
  return r < 0x1.fffffep-1f ? r : 0x1.fffffep-1f;
}

// (hi:lo) >> k and hi >> k for k >= 0; from k = 32 on the pair is below 2^32 (its exact
// value does not matter to the callers)
FX_FN u32 shf_r_clamp(u32 lo, u32 hi, u32 k) {
#ifdef __CUDA_ARCH__
  u32 r;
  asm("shf.r.clamp.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(lo), "r"(hi), "r"(k));
  return r;
#else
  return k >= 32 ? hi : (u32)((((u64)hi << 32) | lo) >> k);
#endif
}
FX_FN u32 shr_clamp(u32 x, u32 k) {
#ifdef __CUDA_ARCH__
  u32 r;
  asm("shr.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(k));
  return r;
#else
  return k >= 32 ? 0u : x >> k;
#endif
}
FX_FN u64 shr64_clamp(u64 x, u32 k) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.b64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(k));
  return r;
#else
  return k >= 64 ? 0 : x >> k;
#endif
}
// float of x, truncated to 24 bits
FX_FN float to_float_rz(u32 x) {
#ifdef __CUDA_ARCH__
  return __uint2float_rz(x);
#else
  int z = 0;
  while (z < 8 && !(x & (0x80000000u >> z))) z++;
  return (float)(x & ~(0xffu >> z));
#endif
}

// A softening eps (normal) as m 2^-58 2^(2 (E - 1023)), m in [2^58, 2^60).
struct Soft {
  u64 m;
  int E;
};
FX_FN Soft soft_of(double eps) {
  const int e = (int)(hi_word(eps) >> 20) - 1023, half = e >> 1;
  const u64 mant = ((u64)((hi_word(eps) & 0x000fffffu) | 0x00100000u) << 32) | lo_word(eps);
  return Soft{mant << (6 + (e - 2 * half)), 1023 + half};
}

// The mantissa of a double (words h, l) as an integer in [2^61, 2^62): yh:yl.  A zero or
// subnormal gets a mantissa too; its exponent field 0 makes its products vanish.
FX_FN void mantissa62(u32 h, u32 l, u32 &yh, u32 &yl) {
  yh = shf_l(l, (h & 0x000fffffu) | 0x00100000u, 9);
  yl = l << 9;
}

// s = x_0^2 + ... + x_(D-1)^2 + eps as Mh:Ml 2^-63 2^(es - 1023) with the top bit of Mh set.
// x_d: mantissa62 integers y and biased exponents ex.  The mantissas are shifted to the
// largest exponent E (at least sqrt(eps)'s) as X_d < 2^62, and the squares added as
// integers: X^2 2^-64 = xh^2 + (xh xl >> 31), the low squares left out; relative error
// below 2^-55.
template <int D>
FX_FN void square_sum(const u32 (&yh)[D], const u32 (&yl)[D], const int (&ex)[D], const Soft &eps, u32 &Mh,
                      u32 &Ml, int &es) {
  int E = eps.E;
  for (int d = 0; d < D; d++) E = ex[d] > E ? ex[d] : E;
  u64 mid = 0, H = shr64_clamp(eps.m, 2u * (u32)(E - eps.E));
  for (int d = 0; d < D; d++) {
    const u32 a = (u32)(E - ex[d]);
    const u32 xl = shf_r_clamp(yl[d], yh[d], a), xh = shr_clamp(yh[d], a);
    mid = mul_wide(xh, xl, mid);
    H = mul_wide(xh, xh, H);
  }
  H += mid >> 31;
  const u32 Hh = (u32)(H >> 32), Hl = (u32)H;
  const int z = 158 - (int)(as_uint(to_float_rz(Hh)) >> 23);  // leading zeros of H
  Mh = shf_l(Hl, Hh, z);
  Ml = Hl << z;
  es = 2 * E - 1018 - z;
}

// -2 / s as a double (rounded), from R = 2^62 / ms and the biased exponent es of s
FX_FN double minus_two_over(u64 R, int es) {
  const u64 b = ((u64)(u32)(2046 - es) << 52) + ((R + 256) >> 9) - (1ull << 52) + (1ull << 63);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// Mantissa of 1/s for s = ms 2^(es - 1023), ms = Mh:Ml 2^-63 in [1, 2): 2^62 / ms as an
// integer in (2^61, 2^62].  Seed r0 (24 bits), its defect n = ms r0 - 1 exact to 2^-62
// (|n| < 2^-21), 1/ms = r0 (1 - n + n^2): relative error below 2^-58 (the n^3 term is below
// 2^-63).
FX_FN u64 rcp_mantissa(u32 Mh, u32 Ml, float r0_bias = 1.0f) {
  float r0 = seed_rcp(as_float((Mh >> 8) + 0x3f000000u));
#ifndef __CUDA_ARCH__
  r0 *= r0_bias;  // tests: a seed off by a chosen amount
  r0 = r0 < 0x1.fffffep-1f ? (r0 > 0.5f ? r0 : 0x1.000002p-1f) : 0x1.fffffep-1f;
#endif
  const u32 Q = as_uint(r0) * 128u + 0xC0000000u;                                   // r0 2^31
  const u64 n = mul_wide(Mh, Q, (mul_wide(Ml, Q, 0) >> 32) | 0xC000000000000000ull);  // (ms r0 - 1) 2^62
  const u32 nh = (u32)(n >> 10);                                                    // n 2^-10: 31 bits, signed
  const u64 nn = (u64)((int64_t)(int)nh * (int)nh);
  const u64 g = (u64)(u32)((u32)(nn >> 32) >> 10) - n;                              // (n^2 - n) 2^62
  // r0 (1 + g) 2^62 = Q 2^31 + 2 Q g_hi + (2 Q g_lo >> 32)
  const u32 c = 0x80000000u + 2u * (u32)(g >> 32);
  return mul_wide(Q, c, mul_wide(2u * Q, (u32)g, 0) >> 32);
}

// |x| / s = (w2 w1 w0) 2^(-91 + ex - es) for the mantissa62 integer y of x and R = 2^62 / ms
// of rcp_mantissa: y R 2^-32, a number in [2^90, 2^92), without the low x low product
// (relative error below 2^-58).
FX_FN void mul_mantissa(u32 yh, u32 yl, u64 R, u32 &w2, u32 &w1, u32 &w0) {
  const u32 Rh = (u32)(R >> 32), Rl = (u32)R;
  const u64 mid = mul_wide(yl, Rh, mul_wide(yh, Rl, 0));
  const u64 P = mul_wide(yh, Rh, mid >> 32);
  w2 = (u32)(P >> 32);
  w1 = (u32)P;
  w0 = (u32)mid;
}

// A signed 96-bit integer (two's complement).
struct Acc96 {
  u32 w0, w1, w2;
};
FX_FN void add96(Acc96 &a, u32 w2, u32 w1, u32 w0) {
#ifdef __CUDA_ARCH__
  asm("add.cc.u32 %0, %0, %3;\n\taddc.cc.u32 %1, %1, %4;\n\taddc.u32 %2, %2, %5;"
      : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2)
      : "r"(w0), "r"(w1), "r"(w2));
#else
  u64 t = (u64)a.w0 + w0;
  a.w0 = (u32)t;
  t = (u64)a.w1 + w1 + (t >> 32);
  a.w1 = (u32)t;
  a.w2 = a.w2 + w2 + (u32)(t >> 32);
#endif
}

// a + w + c, c = 0 or 1
FX_FN void add96_carry(Acc96 &a, u32 w2, u32 w1, u32 w0, u32 c) {
#ifdef __CUDA_ARCH__
  u32 t;
  asm("add.cc.u32 %3, %7, 0xffffffff;\n\taddc.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.u32 %2, %2, %6;"
      : "+r"(a.w0), "+r"(a.w1), "+r"(a.w2), "=&r"(t)
      : "r"(w0), "r"(w1), "r"(w2), "r"(c));
#else
  add96(a, 0u, 0u, c);
  add96(a, w2, w1, w0);
#endif
}

// A lane's column sum (|sum| < 2^85) as limbs of 27, 27 and 27 bits and a sign, each of which
// adds over 32 lanes without overflow (the top one below 2^31: 0.77 2^85 is the largest sum of
// the policies).  The low 5 bits are rounded to nearest, by starting the sum at half of 2^5: but
// for half a unit (ties go up) that error has no sign, so it does not grow with the number of
// sums like a truncation's.
FX_FN Acc96 column_start() { return Acc96{16u, 0u, 0u}; }
FX_FN void column_limbs(const Acc96 &a, u32 &l0, u32 &l1, int &l2) {
  l0 = a.w0 >> 5;
  l1 = a.w1 & 0x07ffffffu;
  l2 = (int)shf_r(a.w1, a.w2, 27);
}
// Sums of limbs as a double in units of 2^5
FX_FN double limbs_total(u64 t0, u64 t1, int64_t t2) {
  return ((double)t2 * 134217728.0 + (double)t1) * 134217728.0 + (double)t0;
}

// ---- sines and cosines (|x| <= 1) as fixed-point numbers ----

typedef int64_t i64;
FX_FN i64 mul_wide_s(int a, int b, i64 c) { return (i64)a * b + c; }

// x 2^62 rounded to an integer, |x| <= 1, as h 2^32 + l with signed l
struct Limbs {
  int h, l;
};
FX_FN Limbs limbs_of(double x) {
  const double y = x * 0x1p62;
#ifdef __CUDA_ARCH__
  const i64 v = __double2ll_rn(y);
#else
  const i64 v = (i64)y;  // exact from 2^53 on; below, truncation by less than one unit
#endif
  return Limbs{(int)((u64)(v + 0x80000000ll) >> 32), (int)(u32)v};
}

// (a c + b d) 2^60, the low x low products left out (error below 1.5 units)
FX_FN i64 dot2(const Limbs &a, const Limbs &b, const Limbs &c, const Limbs &d) {
  const i64 mid = mul_wide_s(a.h, c.l, mul_wide_s(a.l, c.h, mul_wide_s(b.h, d.l, mul_wide_s(b.l, d.h, 0))));
  return mul_wide_s(a.h, c.h, mul_wide_s(b.h, d.h, mid >> 32));
}

// A number as a 96-bit integer w 2^-92
struct Fix92 {
  u32 w2, w1, w0;
};
FX_FN Fix92 fix92_of(double x) {  // 2^-27 <= x < 8
  const int e = (int)(hi_word(x) >> 20) - 1023, sh = e + 40;  // x 2^92 = mant 2^(e + 40)
  const u64 m = ((u64)((hi_word(x) & 0x000fffffu) | 0x00100000u) << 32) | lo_word(x);
  const u64 lo = sh < 32 ? (m << sh) : (m << (sh - 32));
  const u32 top = (u32)(sh == 0 ? 0 : m >> (64 - (sh < 32 ? sh : sh - 32)));
  if (sh < 32) return Fix92{top, (u32)(lo >> 32), (u32)lo};
  return Fix92{(u32)(lo >> 32), (u32)lo, 0u};
}

// x^2 + he for x 2^60 (|x| <= 1): ms 2^(3 - z) with ms = Mh:Ml 2^-63 in [1/4, 1) and z odd.
// he in [2^-27, 4].  |x| as ~x where negative: one unit of 2^-60.
FX_FN void square_plus(i64 x, const Fix92 &he, u32 &Mh, u32 &Ml, int &z) {
  const u32 sg = (u32)((int)(u32)((u64)x >> 32) >> 31);
  const u32 a1 = (u32)((u64)x >> 32) ^ sg, a0 = (u32)x ^ sg;
  const u32 xh = shf_l(a0, a1, 2), xl = a0 << 2;
  const u64 mid = mul_wide(xh, xl, (u64)(u32)(mul_wide(xl, xl, 0) >> 33));  // half of the cross terms
  const u64 H = mul_wide(xh, xh, mid >> 31);
  Acc96 d{he.w0, he.w1, he.w2};
  add96(d, (u32)(H >> 32), (u32)H, (u32)mid << 1);
  z = 156 - (int)(as_uint(to_float_rz(d.w2)) >> 23);  // leading zeros - 2
  z |= 1;
  Mh = shf_l(d.w1, d.w2, z);
  Ml = shf_l(d.w0, d.w1, z);
}

// Seed of ms^(-1/2) 2^30 in [2^30, 2^31) for ms = m 2^-31, 2^29 <= m < 2^31, within 2^-21.
FX_FN u32 seed_rsqrt(u32 m, float bias) {
  const float f = to_float_rz(2u * m);  // ms 2^32
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  (void)bias;
#else
  float r = (float)(1.0 / __builtin_sqrt((double)f)) * bias;
#endif
  r = r > 0x1p-16f ? r : 0x1p-16f;
  r = r < 0x1.fffffep-16f ? r : 0x1.fffffep-16f;
  return as_uint(r) * 128u + 0x80000000u;
}

// 2^60 ms^(-1/2), an integer in (2^60, 2^61]: y the seed, n = ms y^2 - 1 to 2^-58, then
// y (1 - n/2 + 3/8 n^2): relative error below 2^-57.
FX_FN u64 rsqrt_mantissa(u32 Mh, u32 Ml, float bias = 1.0f) {
  const u32 Q = seed_rsqrt(Mh, bias);
  const u64 q2 = mul_wide(Q, Q, 0);  // y^2 2^60
  const u32 qh = (u32)(q2 >> 32), ql = (u32)q2;
  const u64 nm = mul_wide(Ml, qh, mul_wide(Mh, ql, 0));
  const u64 n = mul_wide(Mh, qh, (nm >> 32) | 0xF800000000000000ull);  // n 2^59
  const int nh = (int)(u32)(n >> 8);
  const u32 nn = (u32)((u64)mul_wide_s(nh, nh, 0) >> 32);              // n^2 2^70
  const u64 c = (u64)((nn * 3u) >> 14) - (u64)((i64)n >> 1);           // 2^59 (3/8 n^2 - n/2)
  const u64 C = (c << 3) + 0x4000000000000000ull;
  return mul_wide(Q, (u32)(C >> 32), mul_wide(Q, (u32)C, 0) >> 32);
}

// Mh:Ml 2^-63 in [1, 2) times 2^e as ms 2^(2 g), ms = Mh:Ml 2^-63 in [1/4, 1)
FX_FN int even_exponent(u32 &Mh, u32 &Ml, int e) {
  const int sh = 2 - (e & 1);
  Ml = shf_r(Ml, Mh, sh);
  Mh >>= sh;
  return (e + sh) >> 1;
}

// a b 2^-63 for a, b in [2^62, 2^63), renormalised into that range; the power of two goes
// to e.  Relative error below 2^-60.
FX_FN u64 mul_renorm63(u64 a, u64 b, int &e) {
  const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
  const u64 mid = mul_wide(al, bh, mul_wide(ah, bl, 0));
  u64 P = mul_wide(ah, bh, mid >> 32);  // [2^60, 2^62)
  const int up = (P >> 61) ? 1 : 2;
  e -= up;
  P = (P << up) | ((u32)mid >> (32 - up));
  return P;
}

// 2^58 ms^(-3/2), an integer in [2^58, 2^61): y the seed, n = ms y^2 - 1 to 2^-58, then
// y^3 (1 - 3/2 n + 15/8 n^2): relative error below 2^-56.
FX_FN u64 rsqrt3_mantissa(u32 Mh, u32 Ml, float bias = 1.0f) {
  const u32 Q = seed_rsqrt(Mh, bias);
  const u64 q2 = mul_wide(Q, Q, 0);  // y^2 2^60
  const u32 qh = (u32)(q2 >> 32), ql = (u32)q2;
  const u64 nm = mul_wide(Ml, qh, mul_wide(Mh, ql, 0));
  const u64 n = mul_wide(Mh, qh, (nm >> 32) | 0xF800000000000000ull);  // n 2^59
  const u64 q4 = q2 << 2;
  const u64 Y = mul_wide((u32)(q4 >> 32), Q, mul_wide((u32)q4, Q, 0) >> 32);  // y^3 2^60
  const int nh = (int)(u32)(n >> 8);
  const u32 nn = (u32)((u64)mul_wide_s(nh, nh, 0) >> 32);                     // n^2 2^70
  const u64 c = (u64)(((nn >> 4) * 15u) >> 10) - n - (u64)((i64)n >> 1);             // 2^59 (15/8 n^2 - 3/2 n)
  const u64 C = (c << 3) + 0x4000000000000000ull;                             // 2^62 (1 + ...)
  const u32 Yh = (u32)(Y >> 32), Yl = (u32)Y, Ch = (u32)(C >> 32), Cl = (u32)C;
  return mul_wide(Yh, Ch, mul_wide(Yl, Ch, mul_wide(Yh, Cl, 0)) >> 32);
}

// |x| W as (w2 w1 w0) 2^-86 for x 2^60 and W 2^58 < 2^61; the sign of x in sg (0 or ~0)
FX_FN void mul_fixed(i64 x, u64 W, u32 &sg, u32 &w2, u32 &w1, u32 &w0) {
  sg = (u32)((int)(u32)((u64)x >> 32) >> 31);
  const u32 xh = (u32)((u64)x >> 32) ^ sg, xl = (u32)x ^ sg, Wh = (u32)(W >> 32), Wl = (u32)W;
  const u64 mid = mul_wide(xl, Wh, mul_wide(xh, Wl, mul_wide(xl, Wl, 0) >> 32));
  const u64 P = mul_wide(xh, Wh, mid >> 32);
  w2 = (u32)(P >> 32);
  w1 = (u32)P;
  w0 = (u32)mid;
}

// (w2 w1 w0) >> k for any k >= 0 (a non-negative value)
FX_FN void shift96_any(u32 &w2, u32 &w1, u32 &w0, int k) {
  if (k >= 64) {
    w0 = k >= 96 ? 0u : w2;
    w1 = w2 = 0u;
  } else if (k >= 32) {
    w0 = w1;
    w1 = w2;
    w2 = 0u;
  }
  k &= 31;
  w0 = shf_r(w0, w1, k);
  w1 = shf_r(w1, w2, k);
  w2 >>= k;
}
// The term (w2 w1 w0) >> k, k >= 1, with the sign mask sg, rounded to nearest: what to add,
// and its carry (a negative number as ~w + 1, a term rounded up as w + 1: both of the carry).
template <bool SMALL>  // k < 32
FX_FN u32 signed_shift96(u32 &w2, u32 &w1, u32 &w0, int k, u32 sg) {
  if (!SMALL) {
    shift96_any(w2, w1, w0, k - 1);
    k = 1;
  }
  const u32 c = ((w0 >> (k - 1)) ^ sg) & 1u;
  w0 = shf_r(w0, w1, k) ^ sg;
  w1 = shf_r(w1, w2, k) ^ sg;
  w2 = (w2 >> k) ^ sg;
  return c;
}
// 2^e as a double, -1022 <= e <= 1023
FX_FN double pow2(int e) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((e + 1023) << 20, 0);
#else
  const u64 b = (u64)(e + 1023) << 52;
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}
// value 2^lsb as a double
FX_FN double total96(const Acc96 &a, int lsb) {
  const double hi = (double)(int64_t)(((u64)a.w2 << 32) | a.w1);
  return (hi * 4294967296.0 + (double)a.w0) * pow2(lsb);
}

}  // namespace fx64
