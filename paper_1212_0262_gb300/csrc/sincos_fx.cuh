// Sine and cosine of FP64 angles as 62-bit fixed-point numbers, on the integer pipe, for the
// FP64 HMF stages (GB300 issues about 2 FP64 operations per SM and clock against 64 integer
// multiply-adds; the table-driven FP64 form of sincos_fp64.cuh spends 8 of them per angle).
//
// As there (Tang's table-driven reduction): theta = k h + r, h = pi/2048, |r| <= h/2 (1 + 1e-4),
//   sin(theta) = S + S cm + C sr,   cos(theta) = C + C cm - S sr,
// (S, C) = (sin, cos)(k h) from a 4096-entry table, sr = sin r, cm = cos r - 1.  Here
// * r 2^72 = theta 2^72 - k (h 2^72) modulo 2^64: the difference is below 2^62, so the bits
//   that overflow cancel; h 2^72 = pi 2^61 is taken to 96 bits, so r is exact to 2^-72 and
//   the 0.3 units that the last 64 bits of k h are short of;
// * r^2, r^3/6 are integer products, r^4/24 (below 2^-45) an FP32 one;
// * the sums S cm + C sr and C cm - S sr are 62-bit dot products (fx64::dot2).
// Results are within 2^-57 of the true values (r^5/5! is left out).  |theta| >= 2^20, infinities and NaN (false
// returned) are left to the caller.
#pragma once
#include "fx64.cuh"
#include "sincos_fp64.cuh"

namespace scfx {

using fx64::i64;
using fx64::Limbs;
using fx64::u32;
using fx64::u64;

// table entry k: sin, cos of k pi/2048 as (sin.h, sin.l, cos.h, cos.l)
struct Entry {
  int sh, sl, ch, cl;
};

FX_FN Limbs split(i64 v) { return Limbs{(int)((u64)(v + 0x80000000ll) >> 32), (int)(u32)v}; }
FX_FN i64 join(int h, int l) { return (i64)((u64)(u32)h << 32) + l; }

// k nearest to theta 2048/pi (off by less than 4e-5 from a nearest integer), |theta| < 2^20,
// from a two-float split of theta, as in sc64::sincos_tab
FX_FN int nearest_k(u32 hi, u32 lo) {
  const u32 sign = hi & 0x80000000u, a = hi & 0x7fffffffu, E = a >> 20;
  float th_hi = sc64::bitsf(sign | (((a - 0x38000000u) << 3) | (lo >> 29)));
  if (a < 0x38100000u) th_hi = 0.0f;
  float th_lo = 0.0f;
  if (E >= 949u) th_lo = sc64::bitsf(sc64::fbits(sc64::fmul(sc64::u2f(lo & 0x1fffffffu), sc64::bitsf((E - 948u) << 23))) | sign);
  const float pr = sc64::fmul(th_hi, sc64::kInvHHi);
  const float pe = fmaf(th_hi, sc64::kInvHHi, -pr);
  const float ps = fmaf(th_hi, sc64::kInvHLo, sc64::fmul(th_lo, sc64::kInvHHi));
  const float kp = sc64::frint(pr);
  const float ka = sc64::frint(sc64::fadd(sc64::fadd(pr, -kp), sc64::fadd(pe, ps)));
  return sc64::f2i_exact(kp) + sc64::f2i_exact(ka);
}

// (sin, cos) 2^62 of th; false (nothing written) for |th| >= 2^20 or not finite
FX_FN bool sincos_fx(double th, const Entry *tab, i64 &s62, i64 &c62) {
  const u32 hi = fx64::hi_word(th), lo = fx64::lo_word(th);
  const int E = (int)((hi >> 20) & 0x7ffu);
  if (E >= (int)sc64::kExpLimit) return false;
  const int k = nearest_k(hi, lo);
  // theta 2^72 modulo 2^64 (bits below 2^-72 dropped)
  const u64 mant = ((u64)((hi & 0x000fffffu) | 0x00100000u) << 32) | lo;
  const int sh = E - 1003;
  u64 t72 = sh >= 0 ? mant << sh : fx64::shr64_clamp(mant, (u32)-sh);
  t72 = (int)hi < 0 ? 0 - t72 : t72;
  // k pi 2^61 to 2^-32
  const u64 kh = (u64)(i64)k * 0x6487ED5110B4611Aull + (u64)((i64)k * 0x62633145 >> 32);
  const i64 r = (i64)(t72 - kh);
  const Limbs R = split(r);
  const i64 r2 = fx64::mul_wide_s(R.h, R.h, fx64::mul_wide_s(R.h, R.l, 0) >> 31);  // r^2 2^80, below 2^60
  const int r2h = (int)(r2 >> 29), rh = (int)(r >> 31);                            // r^2 2^51, r 2^41
  const int r3 = (int)(fx64::mul_wide_s(r2h, rh, 0) >> 32);                        // r^3 2^60
  const int r3_6 = (int)(fx64::mul_wide_s(r3, 715827883, 0) >> 32);                // r^3/6 2^60
  const float r2f = (float)r2h;                                                    // r^2 2^51
  const float q = fmaf(sc64::fmul(r2f, r2f), 0x1p-35f / 24.0f, 12582912.0f);       // r^4/24 2^67 + 3 2^22
  const int r4 = (int)(sc64::fbits(q) - 0x4b400000u);
  const Limbs sr = split(r - ((i64)r3_6 << 12));
  const Limbs cm = split(((i64)r4 << 5) - (r2 >> 9));
  const Limbs nsr = split(((i64)r3_6 << 12) - r);
  const Entry e = tab[k & 4095];
  const Limbs S{e.sh, e.sl}, C{e.ch, e.cl};
  s62 = join(e.sh, e.sl) + (fx64::dot2(S, C, cm, sr) >> 8);
  c62 = join(e.ch, e.cl) + (fx64::dot2(C, S, cm, nsr) >> 8);
  return true;
}

// v 2^-60 as a double (rounded to nearest), |v| < 2^62
FX_FN double to_double60(i64 v) {
  const u32 sg = (u32)((int)(u32)((u64)v >> 32) >> 31);
  const u64 a = (u64)(v < 0 ? -v : v);
  u32 h = (u32)(a >> 32), l = (u32)a;
  int z = 0;
  if (h == 0u) {  // below 2^-28
    if (l == 0u) return 0.0;
    h = l;
    l = 0u;
    z = 32;
  }
  const int lz = sc64::clz32(h);  // normalise to bit 63
  const u32 nh = fx64::shf_l(l, h, lz & 31), nl = l << lz;
  // value = (nh:nl) 2^-(60 + z + lz): exponent of bit 63 is 3 - z - lz
  const u32 oh = (sg & 0x80000000u) | ((u32)(1023 + 3 - z - lz - 1) << 20);
  const u64 m = (((((u64)nh << 32) | nl) >> 10) + 1) >> 1;  // 53 bits; the leading one adds 1 to the exponent
  return sc64::bitsd(((u64)oh << 32) + m);
}

}  // namespace scfx
