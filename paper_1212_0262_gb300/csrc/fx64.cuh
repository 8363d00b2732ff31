// Reciprocals and products of doubles on the integer pipe, and 96-bit fixed-point sums.
//
// GB300 issues about 2 FP64 operations per SM and clock, against 64 32 x 32 -> 64 bit
// multiply-adds and 128 integer adds (measured: mad.wide.u32 60, add 120, DFMA 1.9 per SM
// and clock): an FP64 operation costs as much issue time as some 30 multiply-adds.  The
// FP64 pair kernels therefore keep on the FP64 pipe only the operations that need a
// floating-point alignment (coordinate differences, squared distance) and do the rest on
// mantissas held as integers.  Every quantity keeps at least the 53 bits of a double
// (errors below 2^-57 relative, noted at each function), and sums are exact.
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
