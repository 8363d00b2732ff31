// FP64 pair policies of the Newton's-third-law stages with the pair arithmetic on the
// integer pipe (fx64.cuh).  A unit (i-rows x one j-tile) keeps its sums as 96-bit
// integers whose unit 2^lsb follows from the softening: |d| / (d^2 + eps) <= 1 / (2 sqrt
// eps), so no sum can overflow, and what is added is added exactly, whatever the order.  Terms
// are truncated at the unit.  Row sums are moved into doubles (shared memory) every kFxFlush
// units; column sums are added over the warp with redux.sync on 27-bit limbs (rounded to 2^5
// units), over the warps as integers, and stored as doubles.
//
// A unit with a particle beyond RANGE, 2^26 sqrt(eps) (3D: 2^15), of its first row in some
// coordinate, or with a non-finite one runs the FP64 policy's tile instead: at twice that
// distance in every component a 2D term is still 2^54 units long and a 3D term 2^50, so that
// half a unit per term stays below the rounding of FP64 sums.  So does a unit all of whose
// particles lie within 2^-24 sqrt(eps) (CLOSE) of its first row, whose terms, about d / eps, are
// as small: that is a system, or a group in one, whose extent is nothing against its softening
// length.  The CTA decides per unit with one vote, which replaces the barrier after the
// tile's load, and with a second one where its rows are close to each other.
// Error against 64 bits of 1,024 particles in a disk or ball of radius R, rms over the particles
// of |error| / sum of |terms|, column sums truncated to 2^11 units, rounded to 2^5, and all in
// FP64: 2D R = 1000, eps = 1e-8 1.7e-15, 3.8e-17, 4.3e-16; 3D R = 30, eps = 1e-6 2.7e-14, 4.6e-17,
// 4.2e-16.
#pragma once
#include "fx64.cuh"
#include "pairs_impl.cuh"

namespace {

constexpr int kFxFlush = 16;        // units between moves of the row sums into doubles
// What stage() finds in a 16-byte chunk of a tile, and load() in a thread's rows (State::flags)
constexpr int kFxWild = 1;    // out of the fixed-point range
constexpr int kFxNarrow = 2;  // Ring: so small that the fixed-point form has fewer bits than a double
constexpr int kFxBroad = 4;   // 2D, 3D: far enough from the unit's first row for the fixed-point form

// Row sums of a thread in shared memory: [value][thread]
template <int V>
struct FxRowSums {
  double *p;  // this thread's column
  __device__ double &at(int v) const { return p[v * NT]; }
};

// Warp total of 96-bit sums from column_start() (|sum| < 2^85 per lane) to the nearest 2^5: three
// limbs, each added over the 32 lanes without overflow.
__device__ __forceinline__ uint4 fx_warp_sum(const fx64::Acc96 &a) {
  unsigned l0, l1;
  int l2;
  fx64::column_limbs(a, l0, l1, l2);
  uint4 r;
  r.x = __reduce_add_sync(0xffffffffu, l0);
  r.y = __reduce_add_sync(0xffffffffu, l1);
  r.z = (unsigned)__reduce_add_sync(0xffffffffu, l2);
  r.w = 0u;
  return r;
}
// and exactly (|sum| < 2^85 per lane): the low 5 bits as a fourth limb.
__device__ __forceinline__ uint4 fx_warp_sum_exact(const fx64::Acc96 &a) {
  uint4 r;
  r.x = __reduce_add_sync(0xffffffffu, a.w0 >> 5);
  r.y = __reduce_add_sync(0xffffffffu, a.w1 & 0x07ffffffu);
  r.z = (unsigned)__reduce_add_sync(0xffffffffu, (int)fx64::shf_r(a.w1, a.w2, 27));
  r.w = __reduce_add_sync(0xffffffffu, a.w0 & 31u);
  return r;
}
// Sum of n warps' limbs `stride` apart, as a double in units of 2^(lsb + 5)
template <int n>
__device__ __forceinline__ double fx_limb_total(const uint4 *s, int stride) {
  unsigned long long t0 = 0, t1 = 0;
  unsigned t3 = 0;
  long long t2 = 0;
#pragma unroll
  for (int w = 0; w < n; w++) {
    const uint4 v = s[w * stride];
    t0 += v.x;
    t1 += v.y;
    t2 += (int)v.z;
    t3 += v.w;
  }
  return fx64::limbs_total(t0, t1, t2) + (double)t3 * 0.03125;
}

// Rows, flushes and columns shared by the policies: State has acc[R][NACC] and rows.
template <class State, int R, int NACC>
__device__ __forceinline__ void fx_flush(State &st, int lsb) {
#pragma unroll
  for (int r = 0; r < R; r++)
#pragma unroll
    for (int d = 0; d < NACC; d++) {
      st.rows.at(r * NACC + d) += fx64::total96(st.acc[r][d], lsb);
      st.acc[r][d] = fx64::Acc96{0u, 0u, 0u};
    }
  st.units = 0;
}
template <class State, int R, int NACC>
__device__ __forceinline__ void fx_clear(State &st, double *rowsm) {
  st.rows.p = rowsm + threadIdx.x;
  st.units = 0;
#pragma unroll
  for (int r = 0; r < R; r++)
#pragma unroll
    for (int d = 0; d < NACC; d++) {
      st.acc[r][d] = fx64::Acc96{0u, 0u, 0u};
      st.rows.at(r * NACC + d) = 0.0;
    }
}
// column idx of a finished unit: the warps' integer limbs, or (FP64 tile) their doubles
template <int TJ, int NACC>
__device__ __forceinline__ double fx_column(const unsigned char *colraw, int idx, bool wild, int lsb) {
  if (!wild) return fx_limb_total<NT / 32>((const uint4 *)colraw + idx, TJ * NACC) * fx64::pow2(lsb + 5);
  const double *c = (const double *)colraw;
  double v = c[idx];
#pragma unroll
  for (int w = 1; w < NT / 32; w++) v += c[w * TJ * NACC + idx];
  return v;
}
// -v as ~v (one unit of the 96 bits below): the term w with sign mask sg into a row and a column
template <bool COL>
__device__ __forceinline__ void fx_add(unsigned sg, unsigned w2, unsigned w1, unsigned w0, fx64::Acc96 &row,
                                       fx64::Acc96 &col) {
  w2 ^= sg;
  w1 ^= sg;
  w0 ^= sg;
  fx64::add96(row, w2, w1, w0);
  if (COL) fx64::add96(col, w2, w1, w0);
}

// ------------------------------------------------------------ forward 2D and 3D
// Terms d / s (2D) and d s^(-3/2) (3D), s = |d|^2 + eps.  Per pair only the coordinate
// differences are FP64 operations (2 instead of 14, 3 instead of 23.4); the squared distance,
// its inverse power, the products and the sums are integers: 137 instructions per 2D pair and
// 213 per 3D pair, 57% of the integer pipe and of the FP64 pipe (4 warps per scheduler; dependent
// instructions are what is left).  One 2D force at N = 49,152: 28.1 ms with GravF64, 9.74 with
// s on the FP64 pipe, 7.07 as it stands; 3D 49.6 and 11.3.
// eps of the fixed-point form: below, the unit 2^lsb of the sums would grow too large; far above,
// it would lie below the smallest double, and the terms of padding above it
inline bool fx_grav_applies(double eps) { return eps >= 0x1p-28 && eps <= 0x1p600; }

template <int D>
struct FxGravTraits;
template <>
struct FxGravTraits<2> {
  static constexpr int MODEL = MD_GRAV2D, MINB = 4;
  static constexpr int RANGE = 26;  // coordinates within 2^RANGE sqrt(eps) of the first row's
  template <int R, int TJ>
  using Wild = GravF64<R, TJ, STAGE_KICK_DRIFT>;
  using Vec = double2;
  // |d| / s <= 1 / (2 sqrt eps) <= 2^(-half - 1): unit 2^lsb of the sums
  __device__ static int lsb(int half) { return -82 - half; }
  // inverse power of s = ms 2^(es - 1023) as an integer and the shift of a term with exponent ex
  __device__ static unsigned long long power(unsigned Mh, unsigned Ml, int es, int half, int &k) {
    k = es + 9 - half;  // y R 2^-32 = |d| / s 2^(91 - ex + es); at least 9, so 2^12 terms fit
    return fx64::rcp_mantissa(Mh, Ml);
  }
};
template <>
struct FxGravTraits<3> {
  static constexpr int MODEL = MD_GRAV3D, MINB = 4;
  static constexpr int RANGE = 15;  // terms fall as 1 / r^2
  template <int R, int TJ>
  using Wild = Grav3DF64<R, TJ, STAGE_KICK_DRIFT>;
  using Vec = double4_16a;
  // |d| s^(-3/2) <= 0.385 / eps <= 2^(-2 half - 1)
  __device__ static int lsb(int half) { return -84 - 2 * half; }
  __device__ static unsigned long long power(unsigned Mh, unsigned Ml, int es, int half, int &k) {
    const int g = fx64::even_exponent(Mh, Ml, es - 1023);
    k = 3 * g + 1026 - 2 * half;  // y W 2^-32 = |d| s^(-3/2) 2^(87 - (ex - 1023) + 3 g); at least 4
    return fx64::rsqrt3_mantissa(Mh, Ml);
  }
};
__device__ __forceinline__ double fx_coord(const double2 &v, int d) { return d == 0 ? v.x : v.y; }
__device__ __forceinline__ double fx_coord(const double4_16a &v, int d) { return d == 0 ? v.x : d == 1 ? v.y : v.z; }

template <int D, int R_, int TJ_>
struct FxGrav {
  using Tr = FxGravTraits<D>;
  using Vec = typename Tr::Vec;
  static constexpr bool FX = true;
  static constexpr int THREADS = NT, MINB = Tr::MINB;
  using ColT = double;
  using Wild = typename Tr::template Wild<R_, TJ_>;  // units out of the fixed-point range
  static constexpr int R = R_, TJ = TJ_, NACC = D, JB = RecordBytes<Tr::MODEL, false, false>::value;
  static_assert(JB == (int)sizeof(Vec), "one record per particle");
  static constexpr bool MASK = false;
  static constexpr int NR = R;
  static constexpr int FMT = 0;
  static constexpr int COL_BYTES = (NT / 32) * TJ * NACC * (int)sizeof(uint4);
  static constexpr int STAGE_BYTES = 16;  // nothing is staged
  __device__ static int row_of(int r) { return r * NT + (int)threadIdx.x; }
  struct State {
    double x[R][D];
    fx64::Acc96 acc[R][NACC];
    FxRowSums<R * NACC> rows;
    int units;     // since the last flush
    int flags;     // kFxWild, kFxBroad: of the rows of this thread
  };
  // floor(log2(eps) / 2)
  __device__ static int half_exp(const PairArgs &a) { return ((int)(fx64::hi_word(a.epsd) >> 20) - 1023) >> 1; }
  __device__ static int lsb(const PairArgs &a) { return Tr::lsb(half_exp(a)); }
  // Where a coordinate lies from the unit's first row's: kFxWild from 2^range sqrt(eps) on (or
  // not finite), kFxBroad from 2^-CLOSE on.  Padding's terms vanish.
  static constexpr int CLOSE = 24;
  __device__ static int place(double v, double ref, int half, int range = Tr::RANGE) {
    const unsigned h = fx64::hi_word(v - ref) & 0x7fffffffu;
    if ((fx64::hi_word(v) & 0x7fffffffu) == fx64::hi_word(1.0e150)) return 0;
    return (h >= ((unsigned)(1023 + range + half) << 20) ? kFxWild : 0) |
           (h >= ((unsigned)(1023 - CLOSE + half) << 20) ? kFxBroad : 0);
  }
  __device__ static void load(State &st, const void *mirror, int64_t i0, const PairArgs &a, double *rowsm) {
    const int half = half_exp(a);
    const Vec ref = ((const Vec *)mirror)[i0];
    st.flags = 0;
    fx_clear<State, R, NACC>(st, rowsm);
#pragma unroll
    for (int r = 0; r < R; r++) {
      const Vec m = ((const Vec *)mirror)[i0 + row_of(r)];
#pragma unroll
      for (int d = 0; d < D; d++) {
        st.x[r][d] = fx_coord(m, d);
        st.flags |= place(st.x[r][d], fx_coord(ref, d), half);
      }
    }
  }
  __device__ static void flush(State &st, const PairArgs &a) { fx_flush<State, R, NACC>(st, lsb(a)); }
  __device__ static void total(const State &st, int r, double *out) {
#pragma unroll
    for (int d = 0; d < NACC; d++) out[d] = st.rows.at(r * NACC + d);
  }
  // a 16-byte chunk of the tile, all or half of a record (3D: (x, y) or (z, 0)), and the same of the
  // unit's first row
  __device__ static int stage(const unsigned char *tile, int ch, unsigned char *, const PairArgs &a, int64_t i0) {
    constexpr int PER = JB / 16;
    const double2 v = ((const double2 *)tile)[ch], ref = ((const double2 *)a.mirror_in)[i0 * PER + ch % PER];
    const int half = half_exp(a);
    return place(v.x, ref.x, half) | place(v.y, ref.y, half);
  }
  template <bool COL>
  __device__ static void unit(State &st, const unsigned char *smb, const unsigned char *, const PairArgs &a,
                              unsigned char *colraw, int64_t, int64_t) {
    const Vec *sm = (const Vec *)smb;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = half_exp(a);
    const fx64::Soft eps = fx64::soft_of(a.epsd);
    uint4 *colsm = (uint4 *)colraw + w * TJ * NACC;
#pragma unroll(4 / R)
    for (int j = 0; j < TJ; j++) {
      const Vec o = sm[j];
      fx64::Acc96 col[D];
#pragma unroll
      for (int c = 0; c < D; c++) col[c] = fx64::column_start();
      unsigned h[R][D], yh[R][D], yl[R][D];
      unsigned long long pw[R];
      int k[R][D];
      unsigned kor = 0u;
#pragma unroll
      for (int r = 0; r < R; r++) {
        int ex[D], es, kc;
#pragma unroll
        for (int c = 0; c < D; c++) {
          const double d = st.x[r][c] - fx_coord(o, c);
          h[r][c] = fx64::hi_word(d);
          ex[c] = (int)((h[r][c] >> 20) & 0x7ffu);
          fx64::mantissa62(h[r][c], fx64::lo_word(d), yh[r][c], yl[r][c]);
        }
        unsigned Mh, Ml;
        fx64::square_sum<D>(yh[r], yl[r], ex, eps, Mh, Ml, es);
        pw[r] = Tr::power(Mh, Ml, es, half, kc);
#pragma unroll
        for (int c = 0; c < D; c++) {
          k[r][c] = kc - ex[c];
          kor |= (unsigned)k[r][c];
        }
      }
      // one branch for the rows: a component far below the distance (2D: 2^-14) is rare
      if (__builtin_expect(kor < 32u, 1)) {
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
          for (int c = 0; c < D; c++) {
            unsigned w2, w1, w0;
            fx64::mul_mantissa(yh[r][c], yl[r][c], pw[r], w2, w1, w0);
            w0 = fx64::shf_r(w0, w1, k[r][c]);
            w1 = fx64::shf_r(w1, w2, k[r][c]);
            w2 >>= k[r][c];
            fx_add<COL>((unsigned)((int)h[r][c] >> 31), w2, w1, w0, st.acc[r][c], col[c]);
          }
      } else {
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
          for (int c = 0; c < D; c++) {
            unsigned w2, w1, w0;
            fx64::mul_mantissa(yh[r][c], yl[r][c], pw[r], w2, w1, w0);
            fx64::shift96_any(w2, w1, w0, k[r][c]);
            // a zero term adds exactly zero (~0 would be -1 unit)
            fx_add<COL>((w2 | w1 | w0) == 0u ? 0u : (unsigned)((int)h[r][c] >> 31), w2, w1, w0, st.acc[r][c], col[c]);
          }
      }
      if (COL) {
#pragma unroll
        for (int c = 0; c < D; c++) {
          const uint4 s = fx_warp_sum(col[c]);
          if (lane == 0) colsm[D * j + c] = s;
        }
      }
    }
    if (++st.units == kFxFlush) flush(st, a);
  }
  // the unit in FP64: sums of its rows straight into the doubles, columns as doubles
  template <bool COL>
  __device__ static void unit_wild(State &st, const unsigned char *smb, const PairArgs &a, unsigned char *colraw,
                                   int64_t i0, int64_t j0) {
    typename Wild::State ws;
    Wild::load(ws, a.mirror_in, i0);
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int d = 0; d < NACC; d++) ws.accd[r][d] = st.rows.at(r * NACC + d);
    if (COL) Wild::tile_sym(ws, smb, a, (double *)colraw);
    else Wild::template tile<true>(ws, smb, a, i0, j0);
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int d = 0; d < NACC; d++) st.rows.at(r * NACC + d) = ws.accd[r][d];
  }
  __device__ static double column(const unsigned char *colraw, int idx, bool wild, const PairArgs &a) {
    return fx_column<TJ, NACC>(colraw, idx, wild, lsb(a));
  }
};

template <int R, int TJ>
using FxGrav2D = FxGrav<2, R, TJ>;
template <int R, int TJ>
using FxGrav3D = FxGrav<3, R, TJ>;

// ------------------------------------------------------------ forward Ring
// Sines and cosines are numbers of at most 1, so the whole pair term is fixed-point: S and
// sin(d/2) as 62-bit dot products, sin^2 + eps/2 in 96 bits, its power -3/2 from an FP32 seed
// and one third-order step, no FP64 operation (15.5 in RingF64).  The tile's records are
// turned into integers once per unit, by the thread that loaded them.  132 instructions per
// pair; one force at N = 49,152: 36.3 ms with RingF64, 7.10 here (bound by the integer pipe,
// 51%, and by dependent instructions at 4 warps per scheduler).
// The sine of a difference has an error of some 2^-59 here, a product of two doubles' one of
// 2^-53 of the larger sine: less where both angles lie within 2^-6 of 0 (or of pi).  One such
// pair beside N others does not matter to a particle's sum, a system or cluster of such angles
// does (extent 1e-6: forces to 1e-12): a unit with narrow rows and a quarter or more of its
// columns narrow runs RingF64's tile.
// eps of the fixed-point form: shifts of 0 .. 31 bits, sums below 2^95
inline bool fx_ring_applies(double eps) { return eps >= 0x1p-17 && eps <= 4.0; }

template <int R_, int TJ_>
struct RingFx {
  static constexpr bool FX = true;
  static constexpr int THREADS = NT, MINB = 4;
  using ColT = double;
  using Wild = RingF64<R_, TJ_, STAGE_KICK_DRIFT>;
  static constexpr int R = R_, TJ = TJ_, NACC = 1, JB = RecordBytes<MD_RING, false, false>::value;
  static constexpr bool MASK = true;
  static constexpr int NR = R;
  static constexpr int FMT = 0;
  static constexpr int COL_BYTES = (NT / 32) * TJ * NACC * (int)sizeof(uint4);
  static constexpr int STAGE_BYTES = TJ * JB;
  static constexpr int NARROW = TJ / 4;  // narrow columns from which a unit with narrow rows runs in FP64
  __device__ static int row_of(int r) { return r * NT + (int)threadIdx.x; }
  struct State {
    fx64::Limbs s[R], c[R], a[R], g[R];
    fx64::Acc96 acc[R][NACC];
    FxRowSums<R * NACC> rows;
    int units;
    int flags;
  };
  // |term| <= 0.77 / he <= 2^T for he = eps/2; T also makes the shift of the closest pairs,
  // whose power -3/2 is the largest, non-negative
  __device__ static int top(const PairArgs &a) {
    const int h = (int)(fx64::hi_word(a.epsd) >> 20) - 1023;
    const int t = (-8 - 3 * h) >> 1;  // ceil(-4.5 - 1.5 h)
    return -h > t ? -h : t;
  }
  __device__ static int lsb(const PairArgs &a) { return top(a) - 83; }
  __device__ static bool out_of_range(double v) { return (fx64::hi_word(v) & 0x7fffffffu) > 0x3ff00000u; }
  // |sin theta| below 2^-6 (a padding record's cosine is zero)
  __device__ static bool narrow(double s, double c) {
    return (fx64::hi_word(s) & 0x7fffffffu) < (1017u << 20) && c != 0.0;
  }
  __device__ static void load(State &st, const void *mirror, int64_t i0, const PairArgs &a, double *rowsm) {
    st.flags = 0;
    fx_clear<State, R, NACC>(st, rowsm);
#pragma unroll
    for (int r = 0; r < R; r++) {
      const double *m = (const double *)mirror + (i0 + row_of(r)) * 4;
      if (out_of_range(m[0]) || out_of_range(m[1]) || out_of_range(m[2]) || out_of_range(m[3])) st.flags |= kFxWild;
      if (narrow(m[0], m[1])) st.flags |= kFxNarrow;
      st.s[r] = fx64::limbs_of(m[0]);
      st.c[r] = fx64::limbs_of(m[1]);
      st.a[r] = fx64::limbs_of(m[2]);
      st.g[r] = fx64::limbs_of(m[3]);
    }
  }
  __device__ static void flush(State &st, const PairArgs &a) { fx_flush<State, R, NACC>(st, lsb(a)); }
  __device__ static void total(const State &st, int r, double *out) { out[0] = st.rows.at(r); }
  // half a record, (s, c) or (a, g): as (-s, c) or (-a, g) limbs
  __device__ static int stage(const unsigned char *tile, int ch, unsigned char *out, const PairArgs &, int64_t) {
    const double2 v = ((const double2 *)tile)[ch];
    const fx64::Limbs x = fx64::limbs_of(-v.x), y = fx64::limbs_of(v.y);
    ((int4 *)out)[ch] = make_int4(x.h, x.l, y.h, y.l);
    return (out_of_range(v.x) || out_of_range(v.y) ? kFxWild : 0) | ((ch & 1) == 0 && narrow(v.x, v.y) ? kFxNarrow : 0);
  }
  template <bool COL>
  __device__ static void unit(State &st, const unsigned char *, const unsigned char *staged, const PairArgs &a,
                              unsigned char *colraw, int64_t i0, int64_t j0) {
    const int4 *sm = (const int4 *)staged;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const fx64::Fix92 he = fx64::fix92_of(a.epsd);
    const int kc = 3 + top(a);
    uint4 *colsm = (uint4 *)colraw + w * TJ * NACC;
#pragma unroll(4 / R)
    for (int j = 0; j < TJ; j++) {
      const int4 p = sm[2 * j], q = sm[2 * j + 1];
      const fx64::Limbs ns{p.x, p.y}, c{p.z, p.w}, na{q.x, q.y}, g{q.z, q.w};
      fx64::Acc96 col = fx64::column_start();
#pragma unroll
      for (int r = 0; r < R; r++) {
        const long long S = fx64::dot2(st.s[r], st.c[r], c, ns);     // sin(theta_i - theta_j) 2^60
        const long long sh = fx64::dot2(st.a[r], st.g[r], g, na);    // sin((theta_i - theta_j)/2) 2^60
        unsigned Mh, Ml, sg, w2, w1, w0;
        int z;
        fx64::square_plus(sh, he, Mh, Ml, z);
        fx64::mul_fixed(S, fx64::rsqrt3_mantissa(Mh, Ml), sg, w2, w1, w0);
        const int k = kc - 3 * ((z - 3) >> 1);
        w0 = fx64::shf_r(w0, w1, k);
        w1 = fx64::shf_r(w1, w2, k);
        w2 >>= k;
        if (!COL && i0 + row_of(r) == j0 + j) w2 = w1 = w0 = sg = 0u;
        fx_add<COL>(sg, w2, w1, w0, st.acc[r][0], col);
      }
      if (COL) {
        const uint4 sum = fx_warp_sum(col);
        if (lane == 0) colsm[j] = sum;
      }
    }
    if (++st.units == kFxFlush) flush(st, a);
  }
  template <bool COL>
  __device__ static void unit_wild(State &st, const unsigned char *smb, const PairArgs &a, unsigned char *colraw,
                                   int64_t i0, int64_t j0) {
    typename Wild::State ws;
    Wild::load(ws, a.mirror_in, i0);
#pragma unroll
    for (int r = 0; r < R; r++) ws.accd[r][0] = st.rows.at(r);
    if (COL) Wild::tile_sym(ws, smb, a, (double *)colraw);
    else Wild::template tile<true>(ws, smb, a, i0, j0);
#pragma unroll
    for (int r = 0; r < R; r++) st.rows.at(r) = ws.accd[r][0];
  }
  __device__ static double column(const unsigned char *colraw, int idx, bool wild, const PairArgs &a) {
    return fx_column<TJ, NACC>(colraw, idx, wild, lsb(a));
  }
};

// ------------------------------------------------------------ reverse 2D
// Reverse and tangent stages of 2D (w = v_i - v_j, v = lambda_p or dq) in the
// Newton's-third-law form: per pair
//   f = d / s,  j = (w - 2 d (d.w) / s) / s,  e = d / s^2,
// all antisymmetric.  d, w, d.w, and w - 2 d (d.w)/s are FP64 (9 operations; 22 per ordered
// pair in GravF64Adj); the reciprocal, the products and the sums are integers.
//
// f falls as 1 / r, j as 1 / r^2, e as 1 / r^3, each against a unit that its largest term,
// at r = sqrt(eps), sets: RANGE is where a term of e is still 2^52 units long (coordinates
// within 2^9 sqrt(eps) of the first row's; e at 2^26, the forward range, would be 2^5 units).  The
// unit of j also follows from the v: from W, the largest |v_k - v_0| (found before the stage).
// Every particle has a partner whose w is at least W / 2, however the other w are spread, so
// the sum of its |j| is at least 2^58 units within RANGE; terms of j are rounded to
// nearest and its column sums are exact, so that N small terms beside that one add no bias.  Error
// against 64 bits of 1,024 particles in a disk of radius R, rms of |error| / sum of |terms|,
// one-sided in FP64 and here: R = 1, eps = 1e-3 (2^5 sqrt(eps)) j 1.1e-16, 4.7e-17, e 1.5e-16,
// 9.5e-17; eps = 4e-6 (2^9) j 2.1e-16, 9.3e-17, e 2.9e-16, 1.5e-16; eps = 1e-8 (FP64 units here)
// j 2.2e-16, 1.4e-16, e 2.9e-16, 2.1e-16.
//
// Bound by the FP64 pipe (78% at N = 16,384).  A stage of N = 1,000, 8,192 and 16,385: one-sided in
// FP64 220, 3040, 10750 us, here 81, 696, 2880; all units out of range, as in GravF64Adj but with
// columns, 123, 2580, 9550.
template <int R_, int TJ_>
struct FxGrav2DAdj {
  using Fwd = FxGrav<2, R_, TJ_>;
  static constexpr bool FX = true;
  static constexpr int THREADS = NT, MINB = R_ == 1 ? 4 : 3;
  using ColT = double;
  static constexpr int R = R_, TJ = TJ_, NACC = 6, JB = RecordBytes<MD_GRAV2D, false, true>::value;
  static constexpr bool MASK = false;
  static constexpr int NR = R;
  static constexpr int FMT = 0;
  static constexpr int COL_BYTES = (NT / 32) * TJ * NACC * (int)sizeof(uint4);
  static constexpr int STAGE_BYTES = 16;
  __device__ static int row_of(int r) { return r * NT + (int)threadIdx.x; }
  struct State {
    double x[R][2], v[R][2];
    fx64::Acc96 acc[R][NACC];
    FxRowSums<R * NACC> rows;
    int units;
    int flags;
  };
  static constexpr int RANGE = 9;
  static constexpr int CLOSE = Fwd::CLOSE;
  // |w_d| <= 2 W < 2^vexp.  All v equal: any exponent will do (the w of padding, up to 2^299,
  // divided by its s must vanish)
  __device__ static int vexp(const PairArgs &a) { return *a.vrange == 0u ? 299 : (int)(*a.vrange >> 20) - 1021; }
  // the v too large (or not finite) or, not all equal, too close for the exponents used here
  // (the unit of j from 2^-1022 on)
  __device__ static bool v_wild(const PairArgs &a) {
    const unsigned m = *a.vrange;
    return m >= (1322u << 20) || (m != 0u && m < (unsigned)max(223, 2 * Fwd::half_exp(a) + 83) << 20);
  }
  // units of the sums of f, j, e: |f| <= 2^(-half - 1), |j| <= 2^(vexp + 1/2 - 2 half),
  // |e| <= 0.325 eps^(-3/2) <= 2^(-3 half - 1), each 2^83 units at most
  __device__ static int lsb_of(int kind, int half, int ev) {
    return kind == 0 ? -82 - half : kind == 1 ? ev - 82 - 2 * half : -84 - 3 * half;
  }
  __device__ static int lsb(const PairArgs &a, int d) { return lsb_of(d >> 1, Fwd::half_exp(a), vexp(a)); }
  __device__ static void load(State &st, const void *mirror, int64_t i0, const PairArgs &a, double *rowsm) {
    const int half = Fwd::half_exp(a);
    const double2 ref = *(const double2 *)((const double4_16a *)mirror + i0);
    st.flags = v_wild(a) ? kFxWild : 0;
    fx_clear<State, R, NACC>(st, rowsm);
#pragma unroll
    for (int r = 0; r < R; r++) {
      const double4_16a m = ((const double4_16a *)mirror)[i0 + row_of(r)];
      st.x[r][0] = m.x;
      st.x[r][1] = m.y;
      st.v[r][0] = m.z;
      st.v[r][1] = m.w;
      st.flags |= Fwd::place(m.x, ref.x, half, RANGE) | Fwd::place(m.y, ref.y, half, RANGE);
    }
  }
  __device__ static void flush(State &st, const PairArgs &a) {
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int d = 0; d < NACC; d++) {
        st.rows.at(r * NACC + d) += fx64::total96(st.acc[r][d], lsb(a, d));
        st.acc[r][d] = fx64::Acc96{0u, 0u, 0u};
      }
    st.units = 0;
  }
  __device__ static void total(const State &st, int r, double *out) {
#pragma unroll
    for (int d = 0; d < NACC; d++) out[d] = st.rows.at(r * NACC + d);
  }
  // half a record, (x, y) or (vx, vy)
  __device__ static int stage(const unsigned char *tile, int ch, unsigned char *, const PairArgs &a, int64_t i0) {
    if (ch & 1) return 0;
    const double2 m = ((const double2 *)tile)[ch], ref = ((const double2 *)a.mirror_in)[2 * i0];
    const int half = Fwd::half_exp(a);
    return Fwd::place(m.x, ref.x, half, RANGE) | Fwd::place(m.y, ref.y, half, RANGE);
  }
  template <bool COL>
  __device__ static void unit(State &st, const unsigned char *smb, const unsigned char *, const PairArgs &a,
                              unsigned char *colraw, int64_t, int64_t) {
    const double4_16a *sm = (const double4_16a *)smb;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, half = Fwd::half_exp(a);
    const fx64::Soft eps = fx64::soft_of(a.epsd);
    // shifts: f k = es - ex + kf, j k = es - ex(g) + kj, e k = 2 es - ex + ke
    const int kf = 9 - half, kj = vexp(a) + 9 - 2 * half, ke = -1018 - 3 * half;
    uint4 *colsm = (uint4 *)colraw + w * TJ * NACC;
#pragma unroll 1
    for (int j = 0; j < TJ; j++) {
      const double4_16a o = sm[j];
      fx64::Acc96 col[NACC];
#pragma unroll
      for (int c = 0; c < NACC; c++) col[c] = c >> 1 == 1 ? fx64::Acc96{0u, 0u, 0u} : fx64::column_start();
#pragma unroll
      for (int r = 0; r < R; r++) {
        const double d[2] = {st.x[r][0] - o.x, st.x[r][1] - o.y}, v[2] = {st.v[r][0] - o.z, st.v[r][1] - o.w};
        unsigned yh[2], yl[2], Mh, Ml;
        int ex[2], es;
#pragma unroll
        for (int c = 0; c < 2; c++) {
          ex[c] = (int)((fx64::hi_word(d[c]) >> 20) & 0x7ffu);
          fx64::mantissa62(fx64::hi_word(d[c]), fx64::lo_word(d[c]), yh[c], yl[c]);
        }
        fx64::square_sum<2>(yh, yl, ex, eps, Mh, Ml, es);
        const unsigned long long inv = fx64::rcp_mantissa(Mh, Ml);
        const double m2q = fma(d[1], v[1], d[0] * v[0]) * fx64::minus_two_over(inv, es);
        unsigned gh[2], gl[2], hg[2];
        int k[6];
#pragma unroll
        for (int c = 0; c < 2; c++) {
          const double g = fma(m2q, d[c], v[c]);
          hg[c] = fx64::hi_word(g);
          fx64::mantissa62(hg[c], fx64::lo_word(g), gh[c], gl[c]);
          k[c] = es + kf - ex[c];
          k[2 + c] = es + kj - (int)((hg[c] >> 20) & 0x7ffu);
          k[4 + c] = 2 * es + ke - ex[c];
        }
        const bool small = ((unsigned)(k[0] | k[1] | k[2] | k[3] | k[4] | k[5])) < 32u;
#pragma unroll
        for (int c = 0; c < 2; c++) {
          unsigned w2[3], w1[3], w0[3];
          fx64::mul_mantissa(yh[c], yl[c], inv, w2[0], w1[0], w0[0]);
          fx64::mul_mantissa(gh[c], gl[c], inv, w2[1], w1[1], w0[1]);
          fx64::mul_mantissa(w2[0], w1[0], inv, w2[2], w1[2], w0[2]);  // the product of f again
          const unsigned sd = (unsigned)((int)fx64::hi_word(d[c]) >> 31), sg = (unsigned)((int)hg[c] >> 31);
#pragma unroll
          for (int t = 0; t < 3; t++) {
            const int kk = k[2 * t + c];
            if (t == 1) {
              const unsigned cy = __builtin_expect(small, 1)
                                      ? fx64::signed_shift96<true>(w2[t], w1[t], w0[t], kk, sg)
                                      : fx64::signed_shift96<false>(w2[t], w1[t], w0[t], kk, sg);
              fx64::add96_carry(st.acc[r][2 + c], w2[t], w1[t], w0[t], cy);
              if (COL) fx64::add96_carry(col[2 + c], w2[t], w1[t], w0[t], cy);
              continue;
            }
            unsigned sgn = sd;
            if (__builtin_expect(small, 1)) {
              w0[t] = fx64::shf_r(w0[t], w1[t], kk);
              w1[t] = fx64::shf_r(w1[t], w2[t], kk);
              w2[t] >>= kk;
            } else {
              fx64::shift96_any(w2[t], w1[t], w0[t], kk);
              if ((w2[t] | w1[t] | w0[t]) == 0u) sgn = 0u;
            }
            fx_add<COL>(sgn, w2[t], w1[t], w0[t], st.acc[r][2 * t + c], col[2 * t + c]);
          }
        }
      }
      if (COL) {
#pragma unroll
        for (int c = 0; c < NACC; c++) {
          const uint4 s = c >> 1 == 1 ? fx_warp_sum_exact(col[c]) : fx_warp_sum(col[c]);
          if (lane == 0) colsm[NACC * j + c] = s;
        }
      }
    }
    if (++st.units == kFxFlush) flush(st, a);
  }
  // the unit in FP64 (GravF64Adj's terms); a column's six sums are reduced over the warp
  // together, by a butterfly over 8 values
  template <bool COL>
  __device__ static void unit_wild(State &st, const unsigned char *smb, const PairArgs &a, unsigned char *colraw,
                                   int64_t, int64_t) {
    const double4_16a *sm = (const double4_16a *)smb;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    double *colsm = (double *)colraw + w * TJ * NACC;
    flush(st, a);  // frees the integer sums' registers
    double row[R][NACC] = {};
#pragma unroll 1
    for (int j = 0; j < TJ; j++) {
      const double4_16a o = sm[j];
      double col[8] = {};
#pragma unroll
      for (int r = 0; r < R; r++) {
        const double dx = st.x[r][0] - o.x, dy = st.x[r][1] - o.y, wx = st.v[r][0] - o.z, wy = st.v[r][1] - o.w;
        const double inv = rcp_nr(fma(dx, dx, fma(dy, dy, a.epsd))), inv2 = inv * inv;
        const double m2u = -2.0 * fma(dy, wy, dx * wx) * inv2;
        const double t[NACC] = {dx * inv, dy * inv, fma(m2u, dx, wx * inv), fma(m2u, dy, wy * inv), dx * inv2, dy * inv2};
#pragma unroll
        for (int c = 0; c < NACC; c++) {
          row[r][c] += t[c];
          if (COL) col[c] += t[c];
        }
      }
      if (COL) {
        double s = butterfly_sum<8, 16>(col, lane);  // value number: bits 4, 3, 2 of the lane
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        const int c = lane >> 2;
        if ((lane & 3) == 0 && c < NACC) colsm[NACC * j + c] = s;
      }
    }
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
      for (int c = 0; c < NACC; c++) st.rows.at(r * NACC + c) += row[r][c];
  }
  __device__ static double column(const unsigned char *colraw, int idx, bool wild, const PairArgs &a) {
    return fx_column<TJ, NACC>(colraw, idx, wild, lsb(a, idx % NACC));
  }
};

// The largest |v_k - v_0| over both components as the high word of a double into *cur (zero
// before; at least 1 unless all v are equal, ~0 for |v| from 2^299 on or not finite); *next = 0
// for the next stage's.
__global__ void fx_vrange_kernel(const double *__restrict__ v, int64_t N, unsigned *cur, unsigned *next) {
  unsigned m = 0u;
  const int64_t G = (int64_t)gridDim.x * blockDim.x;
  const double v0[2] = {v[0], v[N]};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += G)
#pragma unroll
    for (int c = 0; c < 2; c++) {
      const double x = v[c * N + i], d = x - v0[c];
      m = max(m, max(fx64::hi_word(d) & 0x7fffffffu, d != 0.0 ? 1u : 0u));
      if ((fx64::hi_word(x) & 0x7fffffffu) >= (1322u << 20)) m = ~0u;
    }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(cur, m);
  if (blockIdx.x == 0 && threadIdx.x == 0) *next = 0u;
}

}  // namespace
