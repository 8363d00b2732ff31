// HMF model (Sec. 3.1): one fused, memory-bound pass per integrator stage.
//
// The force of Eq. 6 needs the magnetization of Eq. 7 of the *current* angles.
// Each stage kernel reads the sums (sum cos, sum sin) that the previous stage
// left behind, and per particle
//     f = cos(theta) My - sin(theta) Mx                  (Eq. 6)
//     p += kick * f ;  theta += drift * p                (Sec. 3 step list)
//     accumulate cos(theta_new), sin(theta_new)          (Eq. 7 for the next stage)
// so the state is read once and written once per stage (32 B per particle).
// The paper stores sin and cos in global memory and reloads them.  The mixed
// path recomputes them instead (FP32 polynomials are cheaper than 32 B more
// traffic); the FP64 path keeps (cos, sin) of the current angles in a buffer, as the
// paper does, and computes one sine and cosine per particle-stage instead of two.
//
// Consecutive stages sweep the particles in opposite directions: the last part of
// a stage's writes is still in L2 when the next stage starts on it.
//
// Reduction: per-thread sums, warp shuffles and a block tree give one FP64
// partial per CTA; the last CTA to finish (atomic ticket, no waiting) adds the
// partials in CTA order, so the result is deterministic.
#include <cooperative_groups.h>
#include <math.h>

#include <mutex>

#include "md_internal.cuh"
#include "sincos_fp64.cuh"
#include "sincos_fx.cuh"

namespace {

constexpr int kMaxDevicesTab = 64;

constexpr int NT = kStreamThreads;
constexpr int UNROLL = 2;  // double2 loads of theta and of p in flight per thread
// Mixed sums: a thread adds at most kFlush angles' cosines and sines in FP32 before moving
// them into its FP64 partial, so their rounding does not grow with N / (threads).
constexpr int kFlush = 256;

// ------------------------------------------------ FP64 sine and cosine ------
//
// Table-driven (sincos_fp64.cuh): theta = k pi/2048 + r, a 4096-entry FP64 table of
// (sin, cos)(k pi/2048) in dynamic shared memory (64 KB) of the kernels that use it,
// k and the terms of sin r and cos r below 2^-33 in FP32, 8 FP64 operations per angle;
// |theta| >= 2^20, infinities and NaN use sincos.
constexpr int kTabN = sc64::kTabN;
constexpr int kTabBytes = kTabN * (int)sizeof(double2);

__device__ double2 g_sincos_tab[kTabN];  // (sin, cos)(k pi / 2048), k = 0 .. 4095

__device__ __forceinline__ void sincos_tab(double th, const double2 *__restrict__ tab, double *sp, double *cp) {
  sc64::sincos_tab(th, tab, sp, cp);
}

// The table into shared memory (every thread of the CTA takes part).
__device__ __forceinline__ void load_sincos_tab(double2 *sm) {
  for (int k = threadIdx.x; k < kTabN; k += blockDim.x) sm[k] = g_sincos_tab[k];
  __syncthreads();
}

// The FP64 stages hold (cos, sin) of the current angles as 62-bit fixed-point numbers
// (sincos_fx.cuh), 16 bytes per particle, so that the stage's force, its sine and cosine and
// the magnetization sums are integer arithmetic; the kick and the drift are its FP64
// operations (12 with the sine and cosine of sincos_fp64.cuh and an FP64 force, which bound
// the stage).  Per stage at N = 5e7: 1149 -> 565 us, 3.2 GB at 84% of the copy rate; the
// integer pipe is half busy, the next pair's loads run ahead of the arithmetic (22 us more without).
// A non-finite angle is marked by kNoAngle and makes the sums NaN, and with them every force.
// Cold systems hold doubles instead (hmf_sweep64).
__device__ scfx::Entry g_sincos_fx[kTabN];
constexpr int kNoAngle = (int)0x80000000;

// Set by a thread of this CTA that met a non-finite angle.  In shared memory: as a NaN in the
// thread's FP64 sums it would keep registers through the sweep (12 bytes of spills).
__device__ __forceinline__ volatile int &no_angle_flag() {
  __shared__ int flag;
  return flag;
}

__device__ __forceinline__ void load_sincos_fx(scfx::Entry *sm) {
  if (threadIdx.x == 0) no_angle_flag() = 0;
  for (int k = threadIdx.x; k < kTabN; k += blockDim.x) sm[k] = g_sincos_fx[k];
  __syncthreads();
}

// (cos, sin) as stored: (cos.h, cos.l, sin.h, sin.l)
__device__ __forceinline__ int4 angle_fx_of(double s, double c) {
  if (!(fabs(s) <= 1.0)) return make_int4(kNoAngle, 0, 0, 0);
  const fx64::Limbs lc = fx64::limbs_of(c), ls = fx64::limbs_of(s);
  return make_int4(lc.h, lc.l, ls.h, ls.l);
}

// (cos, sin) of th as stored, and their sums in units of 2^-54.
__device__ __forceinline__ int4 angle_fx(double th, const scfx::Entry *tab, long long &aci, long long &asi) {
  fx64::i64 s62, c62;
  if (!scfx::sincos_fx(th, tab, s62, c62)) {
    if (!(fabs(th) <= 1.7976931348623157e308)) {
      no_angle_flag() = 1;
      return make_int4(kNoAngle, 0, 0, 0);
    }
    double s, c;
    sincos(th, &s, &c);
    s62 = __double2ll_rn(s * 0x1p62);
    c62 = __double2ll_rn(c * 0x1p62);
  }
  aci += (c62 + 128) >> 8;
  asi += (s62 + 128) >> 8;
  const fx64::Limbs c = scfx::split(c62), s = scfx::split(s62);
  return make_int4(c.h, c.l, s.h, s.l);
}

// The FP64 stages' magnetization: (My, -Mx) 2^e as limbs for the integer force, the larger of
// them in [1/2, 1), so that a force has the bits of a double relative to |M|, however small.  The
// kicks' coefficient takes the 2^-e.
struct HmfM {
  fx64::Limbs my, nmx;
  double unit;  // 2^-e
};
// high word of the larger of |Mx|, |My|
__device__ __forceinline__ unsigned hmf_top(double mx, double my) {
  return max(fx64::hi_word(mx) & 0x7fffffffu, fx64::hi_word(my) & 0x7fffffffu);
}
constexpr unsigned kTopMin = (1023u - 200u) << 20, kTopMax = 0x3ff80000u;  // 2^-200, 1.5
// M that the integer force takes: not those that are not finite (some angle is not), or too small.
__device__ __forceinline__ bool hmf_ordinary(double mx, double my) {
  const unsigned top = hmf_top(mx, my);
  return top >= kTopMin && top < kTopMax;
}
// of an ordinary M; lone: N = 1, whose particle's force, its self-term, is exactly zero
__device__ __forceinline__ HmfM hmf_m_of(double mx, double my, bool lone) {
  HmfM m;
  const int e = 1022 - (int)(hmf_top(mx, my) >> 20);
  const double scale = __hiloint2double(lone ? 0 : (1023 + 62 + e) << 20, 0);
  m.unit = __hiloint2double((1023 - e) << 20, 0);
  m.my = scfx::split(__double2ll_rn(my * scale));
  m.nmx = scfx::split(__double2ll_rn(-mx * scale));
  return m;
}

struct HmfArgs {
  double *q, *p;
  int64_t N;
  double invN;
  const double *m_in;  // (sum cos, sum sin) of the current angles
  double kick, drift;
  double *partials;  // 2 per CTA
  double *m_out;     // (sum cos, sum sin) of the new angles
  unsigned *ticket;
  double *fout;  // STAGE_FORCE_ONLY output
  int4 *cs;      // FP64 path: (cos, sin) of the current angles, rewritten by drifts
  unsigned *fmt; // FP64 path: whether cs holds doubles (hmf_sweep64)
  int rev;       // sweep the particles from the top end down
  int nsum;      // row shard: m_in holds nsum (sum cos, sum sin) pairs, one per rank
};

// FP64 mean-field force cos(th) My - sin(th) Mx (Eq. 6): one product and one FMA.  A lone
// particle's force, its own self-term, is exactly zero (N = 1: My = sin th, Mx = cos th),
// which the FMA would leave as a rounding residual of the product.
__device__ __forceinline__ double hmf_force_fp64(double c, double s, double mx, double my, double invN) {
  return invN == 1.0 ? 0.0 : fma(c, my, -(s * mx));
}

// One particle of a mixed stage: FP64 state update, FP32 sine/cosine of the
// FP64-range-reduced angle; the new angle's reduced value is carried in FP32.
// Only the kick and the drift use the FP64 pipe (two DFMA per particle): range
// reduction and float<->double conversions move bits on the integer pipe, and the
// sines and cosines are FP32 polynomials.
template <int MODE>
__device__ __forceinline__ void hmf_particle_mixed(double &th, double &pp, const HmfArgs &a, float mxf, float myf,
                                                   float dtf, float &acf, float &asf, int64_t i) {
  float r = reduce_2pi_f(th);
  float s, c;
  sincos_small(r, &s, &c);
  float f = __fsub_rn(__fmul_rn(c, myf), __fmul_rn(s, mxf));
  if (MODE == STAGE_FORCE_ONLY) {
    a.fout[i] = f2d_bits(f);
    return;
  }
  pp = fma(a.kick, f2d_bits(f), pp);
  if (MODE == STAGE_KICK_DRIFT) {
    th = fma(a.drift, pp, th);
    float r2 = fmaf(dtf, d2f_trunc_bits(pp), r);
    sincos_small(r2, &s, &c);
    acf += c;
    asf += s;
  }
}

// One particle of an FP64 stage; cs: its (cos, sin), rewritten by a drift; kick: a.kick m.unit.
template <int MODE>
__device__ __forceinline__ void hmf_particle_fp64(double &th, double &pp, int4 &cs, const HmfArgs &a, const HmfM &m,
                                                  double kick, long long &aci, long long &asi, int64_t i,
                                                  const scfx::Entry *tab) {
  const fx64::Limbs c{cs.x, cs.y}, s{cs.z, cs.w};
  const double f = scfx::to_double60(fx64::dot2(c, s, m.my, m.nmx));  // (cos My - sin Mx) 2^e
  if (MODE == STAGE_FORCE_ONLY) {
    a.fout[i] = f * m.unit;
    return;
  }
  pp = fma(kick, f, pp);
  if (MODE == STAGE_KICK_DRIFT) {
    th = fma(a.drift, pp, th);
    cs = angle_fx(th, tab, aci, asi);
  }
}

// Grid finish: write this CTA's partial; the last CTA sums all partials in order
// (true in that one).
__device__ __forceinline__ bool grid_finish(double sc, double ss, double *partials, double *m_out,
                                            unsigned *ticket) {
  __shared__ double2 red[NT / 32];
  __shared__ bool last;
  double2 b = block_sum2<NT>(sc, ss, red);
  if (threadIdx.x == 0) {
    partials[2 * blockIdx.x] = b.x;
    partials[2 * blockIdx.x + 1] = b.y;
    __threadfence();
    unsigned t = atomicAdd(ticket, 1u);
    last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double c0 = 0.0, c1 = 0.0;
  for (int j = threadIdx.x; j < (int)gridDim.x; j += NT) {
    c0 += __ldcg(partials + 2 * j);
    c1 += __ldcg(partials + 2 * j + 1);
  }
  __syncthreads();
  double2 t = block_sum2<NT>(c0, c1, red);
  if (threadIdx.x == 0) {
    m_out[0] = t.x;
    m_out[1] = t.y;
    *ticket = 0u;
  }
  return true;
}

// Cold systems, whose angles all lie near 0, pi / 2, pi or 3 pi / 2 (|Mx| or |My| above 1 - 2^-24:
// within some 3e-4): the forces are differences of sines (cosines) and a magnetization component
// that are small themselves, where doubles have more bits than fixed-point numbers.  Their
// stages are all FP64: (cos, sin) kept as doubles (*HmfArgs::fmt = 1), the table-driven sines and
// cosines of sincos_fp64.cuh, FP64 sums; 12 FP64 operations per particle-stage, 8.0 us at
// N = 10,007, 1.31 ms at N = 5e7.  So are stages whose M is not finite, or below 2^-200.
// Wider systems are more exact in fixed point (N = 50,000, angles up to 1e-3, rms of |error| /
// scale of a force 9e-16 against 2.8e-15, whose table sine rounds r^3 / 6 to FP32), narrower ones
// as doubles (up to 1e-6 7e-13 against 7e-17).  A stage whose predecessor's M was cold reads
// doubles, one whose own M is cold writes them.
__device__ __forceinline__ bool hmf_near_one(double m) {
  const unsigned h = fx64::hi_word(m) & 0x7fffffffu;
  return h >= 0x3fefffffu && h < kTopMax && (h > 0x3fefffffu || fx64::lo_word(m) > 0xe0000000u);
}
__device__ __forceinline__ bool hmf_cold(double mx, double my) {
  return (hmf_near_one(mx) && hmf_top(0.0, my) < kTopMax) || (hmf_near_one(my) && hmf_top(mx, 0.0) < kTopMax);
}
template <int MODE, bool CG>
__device__ __noinline__ double2 hmf_sweep64(double *q, double *p, int4 *cs, double *fout, int64_t N, double invN,
                                            double kick, double drift, double mx, double my, const double2 *tab,
                                            int in64, int out64) {
  auto load = [](const auto *ptr) {
    if constexpr (CG) return __ldcg(ptr);
    else return *ptr;
  };
  double2 sum = make_double2(0.0, 0.0);
  auto particle = [&](double &th, double &pp, int4 &w, int64_t i) {
    double c, s;
    if (in64) {
      c = __hiloint2double(w.y, w.x);
      s = __hiloint2double(w.w, w.z);
    } else {
      c = (double)scfx::join(w.x, w.y) * 0x1p-62;
      s = (double)scfx::join(w.z, w.w) * 0x1p-62;
    }
    const double f = hmf_force_fp64(c, s, mx, my, invN);
    if (MODE == STAGE_FORCE_ONLY) {
      fout[i] = f;
      return;
    }
    pp = fma(kick, f, pp);
    if (MODE == STAGE_KICK_DRIFT) {
      th = fma(drift, pp, th);
      sincos_tab(th, tab, &s, &c);
      sum.x += c;
      sum.y += s;
      w = out64 ? make_int4(__double2loint(c), __double2hiint(c), __double2loint(s), __double2hiint(s)) : angle_fx_of(s, c);
    }
  };
  constexpr int UN = CG ? 1 : UNROLL;  // the cluster kernel has no registers for two pairs
  const int64_t G = (int64_t)gridDim.x * NT, npairs = N >> 1;
  const int64_t t0 = (int64_t)blockIdx.x * NT + threadIdx.x;
  for (int64_t k = t0; k < npairs; k += UN * G) {
    double2 qv[UN], pv[UN];
    int4 w[UN][2];
#pragma unroll
    for (int u = 0; u < UN; u++)
      if (k + u * G < npairs) {
        const int64_t ix = k + u * G;
        qv[u] = load((const double2 *)q + ix);
        pv[u] = load((const double2 *)p + ix);
        w[u][0] = load(cs + 2 * ix);
        w[u][1] = load(cs + 2 * ix + 1);
      }
#pragma unroll
    for (int u = 0; u < UN; u++)
      if (k + u * G < npairs) {
        const int64_t ix = k + u * G;
        particle(qv[u].x, pv[u].x, w[u][0], 2 * ix);
        particle(qv[u].y, pv[u].y, w[u][1], 2 * ix + 1);
        if (MODE != STAGE_FORCE_ONLY) ((double2 *)p)[ix] = pv[u];
        if (MODE == STAGE_KICK_DRIFT) {
          ((double2 *)q)[ix] = qv[u];
          cs[2 * ix] = w[u][0];
          cs[2 * ix + 1] = w[u][1];
        }
      }
  }
  if ((N & 1) && t0 == 0) {
    double th = load(q + N - 1), pp = load(p + N - 1);
    int4 w = load(cs + N - 1);
    particle(th, pp, w, N - 1);
    if (MODE != STAGE_FORCE_ONLY) p[N - 1] = pp;
    if (MODE == STAGE_KICK_DRIFT) {
      q[N - 1] = th;
      cs[N - 1] = w;
    }
  }
  return sum;
}
template <int MODE, bool CG>
__device__ __forceinline__ void hmf_sweep64(const HmfArgs &a, double mx, double my, const void *tab, bool in64, bool out64,
                                            double &acd, double &asd) {
  const double2 sum = hmf_sweep64<MODE, CG>(a.q, a.p, a.cs, a.fout, a.N, a.invN, a.kick, a.drift, mx, my,
                                            (const double2 *)tab, in64, out64);
  acd = sum.x;
  asd = sum.y;
}

// One sweep over the particles: the stage's work of this thread, its sums of the new angles'
// cosines and sines into acd, asd.  CG: the loads bypass L1 (a kernel of several stages reads
// what other CTAs wrote in its previous stage).
template <bool MIXED, int MODE, bool CG>
__device__ __forceinline__ void hmf_sweep(const HmfArgs &a, double mx, double my, const scfx::Entry *tab, double &acd,
                                          double &asd) {
  auto load = [](const auto *ptr) {
    if constexpr (CG) return __ldcg(ptr);
    else return *ptr;
  };
  const HmfM m = hmf_m_of(mx, my, a.invN == 1.0);
  const double kick = a.kick * m.unit;
  const float mxf = (float)mx, myf = (float)my, dtf = (float)a.drift;
  float acf = 0.f, asf = 0.f;
  long long aci = 0, asi = 0;
  const int64_t npairs = a.N >> 1;
  const int64_t G = (int64_t)gridDim.x * NT;
  const int64_t t0 = (int64_t)blockIdx.x * NT + threadIdx.x;
  double2 *q2 = reinterpret_cast<double2 *>(a.q);
  double2 *p2 = reinterpret_cast<double2 *>(a.p);
  // blocks of kFlush / 2 double2 pairs per thread; the FP32 sums move into FP64 after each
  // block (a counter tested inside the loop instead made the stage a fifth slower)
  const int64_t block = (int64_t)(kFlush / (2 * UNROLL)) * UNROLL * G;
  for (int64_t kb = t0; kb < npairs; kb += block) {
  const int64_t kend = kb + block < npairs ? kb + block : npairs;
  if constexpr (MIXED) {
    for (int64_t k = kb; k < kend; k += UNROLL * G) {
      double2 qv[UNROLL], pv[UNROLL];
#pragma unroll
      for (int u = 0; u < UNROLL; u++) {
        const int64_t kk = k + u * G;
        const int64_t ix = a.rev ? npairs - 1 - kk : kk;
        if (kk < npairs) {
          qv[u] = load(q2 + ix);
          pv[u] = load(p2 + ix);
        }
      }
#pragma unroll
      for (int u = 0; u < UNROLL; u++) {
        const int64_t kk = k + u * G;
        const int64_t ix = a.rev ? npairs - 1 - kk : kk;
        if (kk < npairs) {
          hmf_particle_mixed<MODE>(qv[u].x, pv[u].x, a, mxf, myf, dtf, acf, asf, 2 * ix);
          hmf_particle_mixed<MODE>(qv[u].y, pv[u].y, a, mxf, myf, dtf, acf, asf, 2 * ix + 1);
          if (MODE == STAGE_KICK_DRIFT) q2[ix] = qv[u];
          if (MODE != STAGE_FORCE_ONLY) p2[ix] = pv[u];
        }
      }
    }
  } else {
    // one pair ahead: the next pair's 64 bytes are on their way while this one is computed
    auto at = [&](int64_t kk) { return a.rev ? npairs - 1 - kk : kk; };
    double2 qn = load(q2 + at(kb)), pn = load(p2 + at(kb));
    int4 an = load(a.cs + 2 * at(kb)), bn = load(a.cs + 2 * at(kb) + 1);
    for (int64_t k = kb; k < kend; k += G) {
      const int64_t ix = at(k);
      double2 qv = qn, pv = pn;
      int4 ca = an, cb = bn;
      if (k + G < kend) {
        const int64_t nx = at(k + G);
        qn = load(q2 + nx);
        pn = load(p2 + nx);
        an = load(a.cs + 2 * nx);
        bn = load(a.cs + 2 * nx + 1);
      }
      hmf_particle_fp64<MODE>(qv.x, pv.x, ca, a, m, kick, aci, asi, 2 * ix, tab);
      hmf_particle_fp64<MODE>(qv.y, pv.y, cb, a, m, kick, aci, asi, 2 * ix + 1, tab);
      if (MODE == STAGE_KICK_DRIFT) {
        a.cs[2 * ix] = ca;
        a.cs[2 * ix + 1] = cb;
        q2[ix] = qv;
      }
      if (MODE != STAGE_FORCE_ONLY) p2[ix] = pv;
    }
  }
  if constexpr (MIXED && MODE == STAGE_KICK_DRIFT) {
    acd += (double)acf;
    asd += (double)asf;
    acf = asf = 0.f;
  }
  if constexpr (!MIXED && MODE == STAGE_KICK_DRIFT) {
    acd += (double)aci * 0x1p-54;
    asd += (double)asi * 0x1p-54;
    aci = asi = 0;
  }
  }
  if ((a.N & 1) && t0 == 0) {
    int64_t i = a.N - 1;
    double th = load(a.q + i), pp = load(a.p + i);
    if constexpr (MIXED) {
      hmf_particle_mixed<MODE>(th, pp, a, mxf, myf, dtf, acf, asf, i);
    } else {
      int4 c = load(a.cs + i);
      hmf_particle_fp64<MODE>(th, pp, c, a, m, kick, aci, asi, i, tab);
      if (MODE == STAGE_KICK_DRIFT) a.cs[i] = c;
    }
    if (MODE == STAGE_KICK_DRIFT) a.q[i] = th;
    if (MODE != STAGE_FORCE_ONLY) a.p[i] = pp;
  }
  if (MODE == STAGE_KICK_DRIFT) {
    if (MIXED) {  // the odd last particle, if any
      acd += (double)acf;
      asd += (double)asf;
    } else {
      acd += (double)aci * 0x1p-54;
      asd += (double)asi * 0x1p-54;
      if (no_angle_flag()) acd = asd = __longlong_as_double(0x7ff8000000000000LL);
    }
  }
}

// SHARD: the magnetization is the sum of every rank's pair in m_in, added in rank
// order (the same value on every rank), over the whole system's N (invN).
// Register budgets of the kick-drift stages: mixed 4 CTAs per SM (64 registers; 80 and 3 CTAs: 262
// against 248 us per stage at N = 5e7), FP64 3 (80; 112 and 2 CTAs: 750 against 566 us).
template <bool MIXED, int MODE, bool SHARD = false>
__global__ void __launch_bounds__(NT, MODE != STAGE_KICK_DRIFT ? 1 : MIXED ? 4 : 3) hmf_stage_kernel(HmfArgs a) {
  double sx = a.m_in[0], sy = a.m_in[1];
  if constexpr (SHARD)
    for (int r = 1; r < a.nsum; r++) {
      sx += a.m_in[2 * r];
      sy += a.m_in[2 * r + 1];
    }
  const double mx = sx * a.invN, my = sy * a.invN;
  extern __shared__ __align__(16) unsigned char tabraw[];  // FP64 kick-drift stages: a sine/cosine table (kTabBytes)
  scfx::Entry *tab = (scfx::Entry *)tabraw;
  double acd = 0.0, asd = 0.0;
  if constexpr (!MIXED) {
    const bool in64 = *a.fmt != 0u, out64 = MODE == STAGE_KICK_DRIFT && hmf_cold(mx, my);
    if (in64 || out64 || !hmf_ordinary(mx, my)) {
      if (MODE == STAGE_KICK_DRIFT) load_sincos_tab((double2 *)tabraw);
      hmf_sweep64<MODE, false>(a, mx, my, tabraw, in64, out64, acd, asd);
      // the last CTA to finish: every other has read *a.fmt
      if (MODE == STAGE_KICK_DRIFT && grid_finish(acd, asd, a.partials, a.m_out, a.ticket) && threadIdx.x == 0) *a.fmt = out64;
      return;
    }
    if (MODE == STAGE_KICK_DRIFT) load_sincos_fx(tab);
  }
  hmf_sweep<MIXED, MODE, false>(a, mx, my, tab, acd, asd);
  if (MODE == STAGE_KICK_DRIFT) grid_finish(acd, asd, a.partials, a.m_out, a.ticket);
}

// Small systems: the 3 n kick-drift stages of n steps in one launch of one cluster.  A stage of
// these sizes is all latency, so the stages follow one another behind a cluster barrier instead
// of a kernel boundary, with the grid, the sweep directions and the groupings of the launched
// stages, and so with their results.  Microseconds per stage at N = 300, 3,000, 10,007:
// mixed 5.9, 6.7, 7.8 launched, 1.7, 2.0, 2.2 here; FP64 7.9, 10.8, 12.3 and 4.2, 5.9, 6.2 (the
// state through L2: 4.5 us in mixed, too).
constexpr int kRunCtas = 16;  // CTAs of the largest cluster

struct HmfRun {
  int64_t begin, end;            // kick-drift stages: (b0, d0) (b1, d1) (b1, d0), b0 = first, then b0
  double first, b0, b1, d0, d1;  // times dt
  // sweep directions: stages [3, 3 + fixed) alternate from rev_fixed on (the captured blocks of
  // steps, whose directions stay as captured), the others from HmfArgs::rev
  int64_t fixed;
  int rev_fixed;
  __device__ int rev(int64_t st, int rev0) const {
    if (st >= 3 && st < 3 + fixed) return rev_fixed ^ (int)((st - 3) & 1);
    return rev0 ^ (int)((st < 3 ? st : st - fixed) & 1);
  }
};

// FP64: the sweep of the launched stage; the CTAs exchange their partial sums through
// distributed shared memory and every CTA adds them, in grid_finish's order.
__global__ void __launch_bounds__(NT, 3) hmf_run_fp64_kernel(HmfArgs a, HmfRun r) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(16) unsigned char tabraw[];
  scfx::Entry *tab = (scfx::Entry *)tabraw;
  __shared__ double2 part[2], msum;
  __shared__ double2 red[NT / 32];
  int table = -1;  // the one in shared memory: of hmf_sweep (0) or hmf_sweep64 (1)
  bool in64 = *a.fmt != 0u;
  const int rev0 = a.rev;
  double2 s = make_double2(a.m_in[0], a.m_in[1]);
  for (int64_t st = r.begin; st < r.end; st++) {
    const int ph = (int)(st % 3);
    a.kick = ph == 0 ? (st == 0 ? r.first : r.b0) : r.b1;
    a.drift = ph == 1 ? r.d1 : r.d0;
    a.rev = r.rev(st, rev0);
    double acd = 0.0, asd = 0.0;
    const double mx = s.x * a.invN, my = s.y * a.invN;
    const bool out64 = hmf_cold(mx, my);
    const int want = in64 || out64 || !hmf_ordinary(mx, my);
    if (table != want) {  // every thread is past its last look-up: it has been at the cluster barrier since
      if (want) load_sincos_tab((double2 *)tabraw);
      else load_sincos_fx(tab);
      table = want;
    }
    if (want) hmf_sweep64<STAGE_KICK_DRIFT, true>(a, mx, my, tabraw, in64, out64, acd, asd);
    else hmf_sweep<false, STAGE_KICK_DRIFT, true>(a, mx, my, tab, acd, asd);
    in64 = out64;
    const double2 b = block_sum2<NT>(acd, asd, red);
    if (threadIdx.x == 0) part[st & 1] = b;
    cluster.sync();  // the partial sums and the state of every CTA are visible
    if (threadIdx.x < 32) {
      double2 v = make_double2(0.0, 0.0);
      if (threadIdx.x < gridDim.x) v = *cluster.map_shared_rank(&part[st & 1], threadIdx.x);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        v.x += __shfl_down_sync(0xffffffffu, v.x, o);
        v.y += __shfl_down_sync(0xffffffffu, v.y, o);
      }
      if (threadIdx.x == 0) msum = v;
    }
    __syncthreads();
    s = msum;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.m_out[0] = s.x;
    a.m_out[1] = s.y;
    *a.fmt = in64;
  }
  cluster.sync();  // no CTA leaves while another reads its partial sums
}

// Sum of a thread's at most five cosines (or sines), below 8, in units of 2^-38: exact for an
// FP32 sum of 2^-15 and more, within 2^-39 below.
__device__ __forceinline__ long long fix38(float v) {
  const float h = rintf(v * 0x1p28f);  // below 2^31
  return ((long long)__float2int_rn(h) << 10) + __float2int_rn((v - h * 0x1p-28f) * 0x1p38f);
}

// Mixed: a thread keeps its particles (at most two pairs, UNROLL of the launched grid, and the
// odd one) in registers through all stages.  A reverse sweep groups the same pairs, p and
// p + G, in the other order.  The groups' FP32 sums are added as integers (the launched stages
// add them in FP64, where they are exact too, but for sums below 2^-16 whose last bits are
// beyond M's FP32): every warp puts its total into every CTA's shared memory, and after the
// cluster barrier every warp adds them for itself.  A drift of some 2^23 and more in one stage
// leaves the FP32 reduction's range: its cosine can be of any size, infinite or NaN.  A warp
// that holds one puts kWildSum in place of its total, every CTA sees it in the sum, and the
// stage's sums are added in FP64, as the launched stages do.  So they are where a sum is below
// 2^-13 per group (all sines or cosines small, or as many of either sign): there the groups'
// 2^-39 could reach M's FP32.
constexpr long long kWildSum = 1ll << 54;  // the particles' own sums stay below 2^53, 128 of these below 2^62
__global__ void __launch_bounds__(NT, 1) hmf_run_mixed_kernel(HmfArgs a, HmfRun r) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  cluster.barrier_arrive();  // here: waited for before the first store into another CTA's shared memory
  constexpr int NW = NT / 32;
  __shared__ longlong2 part[2][kRunCtas * NW];
  __shared__ double2 wide, red[NW];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t npairs = a.N >> 1, G = (int64_t)gridDim.x * NT;
  const int64_t t0 = (int64_t)blockIdx.x * NT + threadIdx.x;
  double2 *q2 = reinterpret_cast<double2 *>(a.q), *p2 = reinterpret_cast<double2 *>(a.p);
  const bool has[2] = {t0 < npairs, t0 + G < npairs}, odd = (a.N & 1) && t0 == 0;
  double2 q[2], p[2];
  double qo = 0.0, po = 0.0;
#pragma unroll
  for (int u = 0; u < 2; u++) {
    q[u] = has[u] ? q2[t0 + u * G] : make_double2(0.0, 0.0);
    p[u] = has[u] ? p2[t0 + u * G] : make_double2(0.0, 0.0);
  }
  if (odd) {
    qo = a.q[a.N - 1];
    po = a.p[a.N - 1];
  }
  double sx = a.m_in[0], sy = a.m_in[1];
  cluster.barrier_wait();  // every CTA of the cluster has started
  for (int64_t st = r.begin; st < r.end; st++) {
    const int ph = (int)(st % 3);
    a.kick = ph == 0 ? (st == 0 ? r.first : r.b0) : r.b1;
    a.drift = ph == 1 ? r.d1 : r.d0;
    const float mxf = (float)(sx * a.invN), myf = (float)(sy * a.invN), dtf = (float)a.drift;
    float c[2][2] = {}, s[2][2] = {};
#pragma unroll
    for (int u = 0; u < 2; u++)
      if (has[u]) {
        hmf_particle_mixed<STAGE_KICK_DRIFT>(q[u].x, p[u].x, a, mxf, myf, dtf, c[u][0], s[u][0], 0);
        hmf_particle_mixed<STAGE_KICK_DRIFT>(q[u].y, p[u].y, a, mxf, myf, dtf, c[u][1], s[u][1], 0);
      }
    // the group's FP32 sums in its sweep's order (a missing pair adds zeros first or last)
    const bool f = r.rev(st, a.rev) != 0;
    const float ac = (((f ? c[1][0] : c[0][0]) + (f ? c[1][1] : c[0][1])) + (f ? c[0][0] : c[1][0])) + (f ? c[0][1] : c[1][1]);
    const float as = (((f ? s[1][0] : s[0][0]) + (f ? s[1][1] : s[0][1])) + (f ? s[0][0] : s[1][0])) + (f ? s[0][1] : s[1][1]);
    float co = 0.f, so = 0.f;
    if (odd) hmf_particle_mixed<STAGE_KICK_DRIFT>(qo, po, a, mxf, myf, dtf, co, so, 0);
    const bool tame = fabsf(ac) + fabsf(as) + fabsf(co) + fabsf(so) < 8.f;  // five angles: at most 5 sqrt(2)
    longlong2 v = make_longlong2(fix38(ac) + fix38(co), fix38(as) + fix38(so));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    if (!__all_sync(0xffffffffu, tame)) v.x = kWildSum;
    longlong2 *slot = &part[st & 1][blockIdx.x * NW + w];
    if (lane < (int)gridDim.x) *cluster.map_shared_rank(slot, lane) = v;
    cluster.sync();
    v = make_longlong2(0, 0);
    for (int k = lane; k < (int)gridDim.x * NW; k += 32) {
      v.x += part[st & 1][k].x;
      v.y += part[st & 1][k].y;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
      v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
    }
    sx = (double)v.x * 0x1p-38;
    sy = (double)v.y * 0x1p-38;
    // kWildSum, or a total below G 2^25 (t in the high word); the same in every thread of the cluster
    const int hx = (int)(v.x >> 32), hy = (int)(v.y >> 32), t = (int)(G >> 7);
    if (hx > (int)(kWildSum >> 33) || (unsigned)(hx + t) < 2u * t || (unsigned)(hy + t) < 2u * t) {
      const double2 b = block_sum2<NT>((double)ac + (double)co, (double)as + (double)so, red);
      if (threadIdx.x == 0) wide = b;
      cluster.sync();
      double2 d = make_double2(0.0, 0.0);
      if (lane < (int)gridDim.x) d = *cluster.map_shared_rank(&wide, lane);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        d.x += __shfl_down_sync(0xffffffffu, d.x, o);
        d.y += __shfl_down_sync(0xffffffffu, d.y, o);
      }
      sx = __shfl_sync(0xffffffffu, d.x, 0);
      sy = __shfl_sync(0xffffffffu, d.y, 0);
      cluster.sync();  // every CTA has read them before the next such stage writes
    }
  }
#pragma unroll
  for (int u = 0; u < 2; u++)
    if (has[u]) {
      q2[t0 + u * G] = q[u];
      p2[t0 + u * G] = p[u];
    }
  if (odd) {
    a.q[a.N - 1] = qo;
    a.p[a.N - 1] = po;
  }
  if (t0 == 0) {
    a.m_out[0] = sx;
    a.m_out[1] = sy;
  }
  cluster.sync();  // no CTA leaves while another writes into its shared memory
}

// (cos, sin) of every angle as the FP64 stages read them, and their sums.  A non-finite angle
// makes the sums NaN.
__global__ void __launch_bounds__(NT) hmf_prime_fp64_kernel(const double *__restrict__ q, int64_t N, double *partials,
                                                            double *m_out, unsigned *ticket, int4 *__restrict__ cs) {
  extern __shared__ __align__(16) unsigned char tabraw[];
  scfx::Entry *tab = (scfx::Entry *)tabraw;
  load_sincos_fx(tab);
  double acd = 0.0, asd = 0.0;
  const int64_t G = (int64_t)gridDim.x * NT;
  const int64_t block = (int64_t)kFlush * G;  // kFlush angles per thread, then the FP64 move
  for (int64_t ib = (int64_t)blockIdx.x * NT + threadIdx.x; ib < N; ib += block) {
    const int64_t iend = ib + block < N ? ib + block : N;
    long long aci = 0, asi = 0;
    for (int64_t i = ib; i < iend; i += G) {
      cs[i] = angle_fx(q[i], tab, aci, asi);
    }
    acd += (double)aci * 0x1p-54;
    asd += (double)asi * 0x1p-54;
  }
  if (no_angle_flag()) acd = asd = __longlong_as_double(0x7ff8000000000000LL);
  grid_finish(acd, asd, partials, m_out, ticket);
}

// After it: a cold system's (cos, sin) once more as doubles, and their FP64 sums (others leave at
// once; the whole grid decides alike, as the last CTA alone writes m_out and fmt).
__global__ void __launch_bounds__(NT) hmf_prime_cold_kernel(const double *__restrict__ q, int64_t N, double *partials,
                                                            double *m_out, unsigned *ticket, int4 *__restrict__ cs,
                                                            unsigned *fmt) {
  const double inv = 1.0 / (double)N;
  const bool cold = hmf_cold(m_out[0] * inv, m_out[1] * inv);
  if (!cold) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *fmt = 0u;
    return;
  }
  double acd = 0.0, asd = 0.0;
  const int64_t G = (int64_t)gridDim.x * NT;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < N; i += G) {
    double s, c;
    sincos(q[i], &s, &c);
    acd += c;
    asd += s;
    cs[i] = make_int4(__double2loint(c), __double2hiint(c), __double2loint(s), __double2hiint(s));
  }
  if (grid_finish(acd, asd, partials, m_out, ticket) && threadIdx.x == 0) *fmt = 1u;
}

// (sum cos, sum sin) of the given angles.  MIXED: FP32 sine/cosine after FP64
// range reduction, FP32 per-thread sums; otherwise FP64 throughout.
// FP64: use_tab selects the table-driven sine and cosine of the FP64 stages (the table
// in kTabBytes of dynamic shared memory) over sincos.
template <bool MIXED>
__global__ void __launch_bounds__(NT) hmf_sums_kernel(const double *__restrict__ q, int64_t N,
                                                      double *partials, double *m_out, unsigned *ticket,
                                                      int use_tab) {
  extern __shared__ double2 tab[];
  if (!MIXED && use_tab) load_sincos_tab(tab);  // use_tab is the same for the whole grid
  float acf = 0.f, asf = 0.f;
  double acd = 0.0, asd = 0.0;
  const int64_t G = (int64_t)gridDim.x * NT;
  const int64_t block = (int64_t)kFlush * G;  // kFlush angles per thread, then the FP64 move
  for (int64_t ib = (int64_t)blockIdx.x * NT + threadIdx.x; ib < N; ib += block) {
  const int64_t iend = ib + block < N ? ib + block : N;
  for (int64_t i = ib; i < iend; i += G) {
    double th = q[i];
    if (MIXED) {
      float s, c;
      sincos_small(reduce_2pi_f(th), &s, &c);
      acf += c;
      asf += s;
    } else {
      double s, c;
      if (use_tab)
        sincos_tab(th, tab, &s, &c);
      else
        sincos(th, &s, &c);
      acd += c;
      asd += s;
    }
  }
  if (MIXED) {
    acd += (double)acf;
    asd += (double)asf;
    acf = asf = 0.f;
  }
  }
  grid_finish(acd, asd, partials, m_out, ticket);
}

// Grid of a streaming kernel: CTAs per SM = the occupancy limit, or `cap` when
// given (0: none), or the tuning key when set.
int grid_for(md_ctx *c, const void *kern, int64_t work_items, int cap = 0, size_t dyn_smem = 0) {
  int lim = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&lim, kern, NT, dyn_smem);
  int occ = (cap > 0 && cap < lim) ? cap : lim;
  if (c->ht.ctas_per_sm > 0) occ = c->ht.ctas_per_sm < lim ? c->ht.ctas_per_sm : lim;
  int64_t g = (int64_t)c->nsm * (occ > 0 ? occ : 1);
  int64_t need = (work_items + NT - 1) / NT;
  if (need < 1) need = 1;
  if (g > need) g = need;
  if (g > c->hmf_grid_max) g = c->hmf_grid_max;
  return (int)g;
}

// The word that says how hmf_cs holds (cos, sin).
unsigned *hmf_fmt(md_ctx *c) { return (unsigned *)(c->hmf_m + 4); }

template <bool MIXED, int MODE>
int launch_stage(md_ctx *c, double kick, double drift, double *fout) {
  HmfArgs a;
  a.q = c->q;
  a.p = c->p;
  a.N = c->N;
  a.invN = 1.0 / (double)c->N;
  a.m_in = c->hmf_m + 2 * c->hmf_cur;
  a.kick = kick;
  a.drift = drift;
  a.partials = c->hmf_partials;
  a.m_out = c->hmf_m + 2 * (1 - c->hmf_cur);
  a.ticket = c->hmf_ticket;
  a.fout = fout;
  a.cs = (int4 *)c->hmf_cs;
  a.fmt = hmf_fmt(c);
  // Consecutive stages sweep the state in opposite directions, so a stage starts on
  // the lines the previous one wrote last, which are still in L2 (dirty lines that
  // are overwritten before eviction are never written back either).
  a.rev = c->hmf_rev;
  a.nsum = 1;
  c->hmf_rev ^= 1;
  auto kern = hmf_stage_kernel<MIXED, MODE>;
  const size_t dyn = (!MIXED && MODE == STAGE_KICK_DRIFT) ? kTabBytes : 0;
  // Mixed stages: 4 CTAs of 256 threads per SM measured fastest on GB300 at N = 5e7
  // (0.252 ms per stage; 0.269 at 3, 0.307 at 2 and 0.271 at 5, the register limit).
  int g = grid_for(c, (const void *)kern, (c->N + 1) / 2 / UNROLL + 1, MIXED ? 4 : 0, dyn);
  kern<<<g, NT, dyn, c->stream>>>(a);
  MD_LAUNCHED(c);
  if (MODE == STAGE_KICK_DRIFT) c->hmf_cur = 1 - c->hmf_cur;
  return MD_OK;
}

}  // namespace

// The sine/cosine table of this device (made on the host in long double, rounded to
// double) and the shared-memory attribute of the kernels that hold it: set up once per
// device, and again if (probe) a read of one entry finds the device copy gone (a device
// reset drops both).  Synchronous; not to be called inside a stream capture.
int hmf_sincos_table(md_ctx *c, bool probe) {
  static std::mutex mu;
  static bool done[kMaxDevicesTab] = {};
  static double2 t[kTabN];
  if (c->device < 0 || c->device >= kMaxDevicesTab) return set_err(c, MD_EINVAL, "device %d", c->device);
  std::lock_guard<std::mutex> lk(mu);
  if (done[c->device]) {
    if (!probe) return MD_OK;
    double2 e1;
    MD_CUDA(c, cudaMemcpyFromSymbol(&e1, g_sincos_tab, sizeof e1, sizeof(double2)));
    if (e1.x == t[1].x && e1.y == t[1].y) return MD_OK;
    done[c->device] = false;
  }
  const long double pi = 3.141592653589793238462643383279502884L;
  for (int k = 0; k < kTabN; k++) {
    const long double x = (long double)k * pi / (long double)(kTabN / 2);
    t[k] = make_double2((double)sinl(x), (double)cosl(x));
  }
  MD_CUDA(c, cudaMemcpyToSymbol(g_sincos_tab, t, sizeof t));
  static scfx::Entry tf[kTabN];
  for (int k = 0; k < kTabN; k++) {
    const long double x = (long double)k * pi / (long double)(kTabN / 2);
    const fx64::Limbs s = scfx::split(llrintl(sinl(x) * 0x1p62L)), co = scfx::split(llrintl(cosl(x) * 0x1p62L));
    tf[k] = scfx::Entry{s.h, s.l, co.h, co.l};
  }
  MD_CUDA(c, cudaMemcpyToSymbol(g_sincos_fx, tf, sizeof tf));
  // the kernels that hold the table in dynamic shared memory (64 KB, above the 48 KB default)
  MD_CUDA(c, cudaFuncSetAttribute(hmf_stage_kernel<false, STAGE_KICK_DRIFT, false>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, kTabBytes));
  MD_CUDA(c, cudaFuncSetAttribute(hmf_stage_kernel<false, STAGE_KICK_DRIFT, true>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, kTabBytes));
  MD_CUDA(c, cudaFuncSetAttribute(hmf_sums_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kTabBytes));
  MD_CUDA(c, cudaFuncSetAttribute(hmf_prime_fp64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kTabBytes));
  done[c->device] = true;
  return MD_OK;
}

// FP64 (sum cos, sum sin) of q[0..N) into device out2, with caller-supplied
// partials (>= grid_cap doubles x 2) and a zeroed ticket.
void hmf_sums_raw(cudaStream_t st, int nsm, int grid_cap, const double *q, int64_t N, double *partials,
                  double *out2, unsigned *ticket) {
  int occ = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, hmf_sums_kernel<false>, NT, 0);
  int64_t g = (int64_t)nsm * (occ > 0 ? occ : 1);
  const int64_t need = (N + NT - 1) / NT;
  if (g > need) g = need;
  if (g > grid_cap) g = grid_cap;
  if (g < 1) g = 1;
  hmf_sums_kernel<false><<<(int)g, NT, 0, st>>>(q, N, partials, out2, ticket, 0);
}

int hmf_sums_fp64_of(md_ctx *c, const double *q, double *d_out2) {
  int rc = hmf_sincos_table(c, false);  // HMF contexts have it already; Ring ones (md_magnetization) may not
  if (rc) return rc;
  auto kern = hmf_sums_kernel<false>;
  int g = grid_for(c, (const void *)kern, c->N, 0, kTabBytes);
  kern<<<g, NT, kTabBytes, c->stream>>>(q, c->N, c->hmf_partials, d_out2, c->hmf_ticket, 1);
  MD_LAUNCHED(c);
  return MD_OK;
}

int hmf_sums_fp64(md_ctx *c, double *d_out2) { return hmf_sums_fp64_of(c, c->q, d_out2); }

// Sums of the current angles into the current magnetization slot.
int hmf_prime(md_ctx *c) {
  double *out = c->hmf_m + 2 * c->hmf_cur;
  if (c->prec == MD_MIXED) {
    auto kern = hmf_sums_kernel<true>;
    int g = grid_for(c, (const void *)kern, c->N);
    kern<<<g, NT, 0, c->stream>>>(c->q, c->N, c->hmf_partials, out, c->hmf_ticket, 0);
    MD_LAUNCHED(c);
  } else {
    // FP64: the sums and the (cos, sin) buffer the FP64 stages read
    const size_t need = sizeof(int4) * (size_t)c->N;
    if (need > c->hmf_cs_bytes) {
      dev_free(c->hmf_cs);
      c->hmf_cs = (double *)dev_alloc(need);
      c->hmf_cs_bytes = c->hmf_cs ? need : 0;
      if (!c->hmf_cs) return set_err(c, MD_ENOMEM, "HMF (cos, sin) buffer: %zu bytes", need);
    }
    int g = grid_for(c, (const void *)hmf_prime_fp64_kernel, c->N, 0, kTabBytes);
    hmf_prime_fp64_kernel<<<g, NT, kTabBytes, c->stream>>>(c->q, c->N, c->hmf_partials, out, c->hmf_ticket,
                                                           (int4 *)c->hmf_cs);
    MD_LAUNCHED(c);
    hmf_prime_cold_kernel<<<g, NT, 0, c->stream>>>(c->q, c->N, c->hmf_partials, out, c->hmf_ticket, (int4 *)c->hmf_cs,
                                                   hmf_fmt(c));
    MD_LAUNCHED(c);
  }
  c->hmf_m_valid = true;
  c->hmf_m_prec = c->prec;
  return MD_OK;
}

// ------------------------------------------------------------ row shards ---
//
// A row shard (md_shard_*) holds rows [row0, row0 + N) of a system of n_total
// particles.  Its stages read the magnetization from every rank's partial sums
// (shard_sums[cur][rank], in rank order) and write the sums of their own new angles
// to shard_sums[1 - cur][rank]; the exchange between stages copies the other ranks'
// pairs in (Sec. 3.1, last paragraph: partial magnetizations per GPU, summed).

int hmf_shard_prime(md_ctx *c) {
  const size_t sums_bytes = sizeof(double) * 4 * (size_t)c->shard_nranks;
  if (!c->shard_sums) {
    c->shard_sums = (double *)dev_alloc(sums_bytes);
    if (!c->shard_sums) return set_err(c, MD_ENOMEM, "HMF shard sums: %zu bytes", sums_bytes);
  }
  MD_CUDA(c, cudaMemsetAsync(c->shard_sums, 0, sums_bytes, c->stream));
  c->shard_cur = 0;
  double *out = c->shard_sums + 2 * c->shard_rank;
  if (c->prec == MD_MIXED) {
    auto kern = hmf_sums_kernel<true>;
    int g = grid_for(c, (const void *)kern, c->N);
    kern<<<g, NT, 0, c->stream>>>(c->q, c->N, c->hmf_partials, out, c->hmf_ticket, 0);
  } else {
    const size_t need = sizeof(int4) * (size_t)c->N;
    if (need > c->hmf_cs_bytes) {
      dev_free(c->hmf_cs);
      c->hmf_cs = (double *)dev_alloc(need);
      c->hmf_cs_bytes = c->hmf_cs ? need : 0;
      if (!c->hmf_cs) return set_err(c, MD_ENOMEM, "HMF (cos, sin) buffer: %zu bytes", need);
    }
    int g = grid_for(c, (const void *)hmf_prime_fp64_kernel, c->N, 0, kTabBytes);
    hmf_prime_fp64_kernel<<<g, NT, kTabBytes, c->stream>>>(c->q, c->N, c->hmf_partials, out, c->hmf_ticket,
                                                           (int4 *)c->hmf_cs);
    MD_LAUNCHED(c);
    hmf_prime_cold_kernel<<<g, NT, 0, c->stream>>>(c->q, c->N, c->hmf_partials, out, c->hmf_ticket, (int4 *)c->hmf_cs,
                                                   hmf_fmt(c));
  }
  MD_LAUNCHED(c);
  c->hmf_m_valid = false;  // md_step's own sums are not kept on a shard
  return MD_OK;
}

namespace {
template <bool MIXED, int MODE>
int launch_shard_stage(md_ctx *c, double kick, double drift, double *fout) {
  const int P = c->shard_nranks;
  HmfArgs a;
  a.q = c->q;
  a.p = c->p;
  a.N = c->N;
  a.invN = 1.0 / (double)c->n_total;
  a.m_in = c->shard_sums + 2 * P * c->shard_cur;
  a.nsum = P;
  a.kick = kick;
  a.drift = drift;
  a.partials = c->hmf_partials;
  a.m_out = c->shard_sums + 2 * (P * (1 - c->shard_cur) + c->shard_rank);
  a.ticket = c->hmf_ticket;
  a.fout = fout;
  a.cs = (int4 *)c->hmf_cs;
  a.fmt = hmf_fmt(c);
  a.rev = c->hmf_rev;
  c->hmf_rev ^= 1;
  auto kern = hmf_stage_kernel<MIXED, MODE, true>;
  const size_t dyn = (!MIXED && MODE == STAGE_KICK_DRIFT) ? kTabBytes : 0;
  int g = grid_for(c, (const void *)kern, (c->N + 1) / 2 / UNROLL + 1, MIXED ? 4 : 0, dyn);
  kern<<<g, NT, dyn, c->stream>>>(a);
  MD_LAUNCHED(c);
  if (MODE == STAGE_KICK_DRIFT) c->shard_cur = 1 - c->shard_cur;
  return MD_OK;
}
}  // namespace

int hmf_shard_stage(md_ctx *c, int mode, double kick, double drift, double *fout) {
  const bool mixed = c->prec == MD_MIXED;
  if (mode == STAGE_FORCE_ONLY)
    return mixed ? launch_shard_stage<true, STAGE_FORCE_ONLY>(c, 0.0, 0.0, fout)
                 : launch_shard_stage<false, STAGE_FORCE_ONLY>(c, 0.0, 0.0, fout);
  return mixed ? launch_shard_stage<true, STAGE_KICK_DRIFT>(c, kick, drift, nullptr)
               : launch_shard_stage<false, STAGE_KICK_DRIFT>(c, kick, drift, nullptr);
}

// The kick-drift stages of nsteps steps as one cluster launch, when the stages' grid is at
// most one cluster and the device can hold it (*done = false, nothing launched, otherwise).
// block_steps of them (after the first step) would be replayed blocks.
int hmf_run(md_ctx *c, int64_t nsteps, int64_t block_steps, const double *k4, double h, bool *done) {
  *done = false;
  const bool mixed = c->prec == MD_MIXED;
  const void *stage = mixed ? (const void *)hmf_stage_kernel<true, STAGE_KICK_DRIFT>
                            : (const void *)hmf_stage_kernel<false, STAGE_KICK_DRIFT>;
  const size_t dyn = mixed ? 0 : kTabBytes;
  const int g = grid_for(c, stage, (c->N + 1) / 2 / UNROLL + 1, mixed ? 4 : 0, dyn);
  if (g > kRunCtas) return MD_OK;
  auto kern = mixed ? hmf_run_mixed_kernel : hmf_run_fp64_kernel;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(g);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = dyn;
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = g;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (g > 8) MD_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  if (dyn) MD_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn));
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, (const void *)kern, &cfg) != cudaSuccess || clusters < 1) {
    cudaGetLastError();
    return MD_OK;
  }
  if (!c->hmf_m_valid || c->hmf_m_prec != c->prec) {
    int rc = hmf_prime(c);
    if (rc) return rc;
  }
  HmfArgs a{};
  a.q = c->q;
  a.p = c->p;
  a.N = c->N;
  a.invN = 1.0 / (double)c->N;
  a.cs = (int4 *)c->hmf_cs;
  a.fmt = hmf_fmt(c);
  a.m_in = c->hmf_m + 2 * c->hmf_cur;
  a.rev = c->hmf_rev;
  // launched stages alternate the direction, replayed blocks keep the one they were captured with
  const int64_t launched = 3 * (nsteps - block_steps);
  const int cur1 = 1 - c->hmf_cur;  // parity after the first step
  HmfRun r{0, 0, k4[0] * h, 2.0 * k4[0] * h, k4[1] * h, k4[2] * h, k4[3] * h, 3 * block_steps, 0};
  if (block_steps) r.rev_fixed = run_direction(c, cur1, h, 1 - c->hmf_rev);
  if (nsteps & 1) c->hmf_cur = 1 - c->hmf_cur;
  if (launched & 1) c->hmf_rev ^= 1;
  a.m_out = c->hmf_m + 2 * c->hmf_cur;
  // pieces of kRunStages, so that a launch stays in the milliseconds
  constexpr int64_t kRunStages = 768;
  for (; r.begin < 3 * nsteps; r.begin = r.end) {
    r.end = r.begin + kRunStages < 3 * nsteps ? r.begin + kRunStages : 3 * nsteps;
    MD_CUDA(c, cudaLaunchKernelEx(&cfg, kern, a, r));
    MD_LAUNCHED(c);
    a.m_in = a.m_out;
  }
  *done = true;
  return MD_OK;
}

int hmf_stage(md_ctx *c, int mode, double kick, double drift, double *fout) {
  if (!c->hmf_m_valid || c->hmf_m_prec != c->prec) {
    int rc = hmf_prime(c);
    if (rc) return rc;
  }
  const bool mixed = c->prec == MD_MIXED;
  switch (mode) {
  case STAGE_KICK_DRIFT:
    return mixed ? launch_stage<true, STAGE_KICK_DRIFT>(c, kick, drift, fout)
                 : launch_stage<false, STAGE_KICK_DRIFT>(c, kick, drift, fout);
  case STAGE_KICK_ONLY:
    return mixed ? launch_stage<true, STAGE_KICK_ONLY>(c, kick, drift, fout)
                 : launch_stage<false, STAGE_KICK_ONLY>(c, kick, drift, fout);
  default:
    return mixed ? launch_stage<true, STAGE_FORCE_ONLY>(c, kick, drift, fout)
                 : launch_stage<false, STAGE_FORCE_ONLY>(c, kick, drift, fout);
  }
}

// ---------------------------------------------------------------- adjoint --
//
// Reverse stages of md_grad for HMF.  With Eqs. 6-7, J = df/dtheta gives
//   (J v)_i = -(sin t_i My + cos t_i Mx) v_i + cos t_i A + sin t_i B,
//   A = (1/N) sum cos t_k v_k,  B = (1/N) sum sin t_k v_k,
// so each reverse stage needs the four sums (sum cos, sum sin, sum cos v,
// sum sin v) of the current angles and lambda_p, which the previous reverse
// stage leaves behind (same deterministic grid finish as the forward).

namespace {

struct HmfAdjArgs {
  double *q, *p, *lq, *lp;
  int64_t N;
  double invN;
  const double *s_in;  // 4 sums of the current (theta, lambda_p)
  double b_adj, b_undo, drift;
  double *partials;  // 4 per CTA
  double *s_out;
  unsigned *ticket;
};

__device__ __forceinline__ void grid_finish4(double v0, double v1, double v2, double v3, double *partials,
                                             double *out, unsigned *ticket) {
  __shared__ double2 red[NT / 32];
  __shared__ bool last;
  double2 b01 = block_sum2<NT>(v0, v1, red);
  __syncthreads();
  double2 b23 = block_sum2<NT>(v2, v3, red);
  if (threadIdx.x == 0) {
    partials[4 * blockIdx.x] = b01.x;
    partials[4 * blockIdx.x + 1] = b01.y;
    partials[4 * blockIdx.x + 2] = b23.x;
    partials[4 * blockIdx.x + 3] = b23.y;
    __threadfence();
    last = (atomicAdd(ticket, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double c[4] = {0.0, 0.0, 0.0, 0.0};
  for (int j = threadIdx.x; j < (int)gridDim.x; j += NT)
#pragma unroll
    for (int k = 0; k < 4; k++) c[k] += __ldcg(partials + 4 * j + k);
  __syncthreads();
  double2 t01 = block_sum2<NT>(c[0], c[1], red);
  __syncthreads();
  double2 t23 = block_sum2<NT>(c[2], c[3], red);
  if (threadIdx.x == 0) {
    out[0] = t01.x;
    out[1] = t01.y;
    out[2] = t23.x;
    out[3] = t23.y;
    *ticket = 0u;
  }
}

template <bool MIXED>
__device__ __forceinline__ void sc_of(double th, double &s, double &c) {
  if (MIXED) {
    float sf, cf;
    sincos_small(reduce_2pi_f(th), &sf, &cf);
    s = f2d_bits(sf);
    c = f2d_bits(cf);
  } else {
    sincos(th, &s, &c);
  }
}

template <bool MIXED>
__global__ void __launch_bounds__(NT) hmf_adj_sums_kernel(const double *__restrict__ q, const double *__restrict__ lp,
                                                          int64_t N, double *partials, double *out, unsigned *ticket) {
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  const int64_t G = (int64_t)gridDim.x * NT;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < N; i += G) {
    double s, c;
    sc_of<MIXED>(q[i], s, c);
    const double v = lp[i];
    a0 += c;
    a1 += s;
    a2 = fma(c, v, a2);
    a3 = fma(s, v, a3);
  }
  grid_finish4(a0, a1, a2, a3, partials, out, ticket);
}

template <bool MIXED>
__global__ void __launch_bounds__(NT) hmf_adj_stage_kernel(HmfAdjArgs a) {
  const double mx = a.s_in[0] * a.invN, my = a.s_in[1] * a.invN;
  const double A = a.s_in[2] * a.invN, B = a.s_in[3] * a.invN;
  const float mxf = (float)mx, myf = (float)my;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  const int64_t G = (int64_t)gridDim.x * NT;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < a.N; i += G) {
    double th = a.q[i], pp = a.p[i], lq = a.lq[i], lp = a.lp[i];
    double s, c, f;
    sc_of<MIXED>(th, s, c);
    if (MIXED)  // the same FP32 force as the forward stage, so the reversal undoes it
      f = f2d_bits(__fsub_rn(__fmul_rn((float)c, myf), __fmul_rn((float)s, mxf)));
    else
      f = hmf_force_fp64(c, s, mx, my, a.invN);
    const double jv = fma(-fma(s, my, c * mx), lp, fma(c, A, s * B));
    lq = fma(a.b_adj, jv, lq);
    pp = fma(-a.b_undo, f, pp);
    if (a.drift != 0.0) {
      lp = fma(a.drift, lq, lp);
      th = fma(-a.drift, pp, th);
      sc_of<MIXED>(th, s, c);
      a0 += c;
      a1 += s;
      a2 = fma(c, lp, a2);
      a3 = fma(s, lp, a3);
      a.q[i] = th;
      a.lp[i] = lp;
    }
    a.p[i] = pp;
    a.lq[i] = lq;
  }
  if (a.drift != 0.0) grid_finish4(a0, a1, a2, a3, a.partials, a.s_out, a.ticket);
}

// lambda_q of the |M| observable: d|M|/dtheta_i = (My cos t_i - Mx sin t_i) / (N |M|).
__global__ void hmf_mag_terminal_kernel(const double *__restrict__ q, int64_t N, double cx, double cy,
                                        double *__restrict__ lq) {
  const int64_t G = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += G) {
    double s, c;
    sincos(q[i], &s, &c);
    lq[i] = fma(cx, c, -cy * s);
  }
}

}  // namespace

// Four sums of the current (theta, lambda_p) into the current adjoint slot.
int hmf_adjoint_prime(md_ctx *c, const double *lp, double *sums) {
  const int g = grid_for(c, (const void *)hmf_adj_sums_kernel<true>, c->N);
  if (c->prec == MD_MIXED)
    hmf_adj_sums_kernel<true><<<g, NT, 0, c->stream>>>(c->q, lp, c->N, c->hmf_partials, sums, c->hmf_ticket);
  else
    hmf_adj_sums_kernel<false><<<g, NT, 0, c->stream>>>(c->q, lp, c->N, c->hmf_partials, sums, c->hmf_ticket);
  MD_LAUNCHED(c);
  return MD_OK;
}

int hmf_adjoint_stage(md_ctx *c, double b_adj, double b_undo, double drift, double *lq, double *lp,
                      const double *s_in, double *s_out) {
  HmfAdjArgs a;
  a.q = c->q;
  a.p = c->p;
  a.lq = lq;
  a.lp = lp;
  a.N = c->N;
  a.invN = 1.0 / (double)c->N;
  a.s_in = s_in;
  a.b_adj = b_adj;
  a.b_undo = b_undo;
  a.drift = drift;
  a.partials = c->hmf_partials;
  a.s_out = s_out;
  a.ticket = c->hmf_ticket;
  const int g = grid_for(c, (const void *)hmf_adj_stage_kernel<false>, c->N);
  if (c->prec == MD_MIXED)
    hmf_adj_stage_kernel<true><<<g, NT, 0, c->stream>>>(a);
  else
    hmf_adj_stage_kernel<false><<<g, NT, 0, c->stream>>>(a);
  MD_LAUNCHED(c);
  return MD_OK;
}

int hmf_magnetization_terminal(md_ctx *c, double cx, double cy, double *lq) {
  int64_t b = (c->N + 255) / 256;
  if (b > (int64_t)c->nsm * 16) b = (int64_t)c->nsm * 16;
  hmf_mag_terminal_kernel<<<(int)b, 256, 0, c->stream>>>(c->q, c->N, cx, cy, lq);
  MD_LAUNCHED(c);
  return MD_OK;
}

// ---------------------------------------------------------------- tangent --
//
// Forward tangent (linearised) dynamics for HMF:  p += kick f, dp += kick J dq,
// then theta += drift p, dq += drift dp, with (J dq)_i from the four sums of the
// current (theta, dq) as in the adjoint above.

namespace {

template <bool MIXED>
__global__ void __launch_bounds__(NT) hmf_tangent_stage_kernel(HmfAdjArgs a) {
  const double mx = a.s_in[0] * a.invN, my = a.s_in[1] * a.invN;
  const double A = a.s_in[2] * a.invN, B = a.s_in[3] * a.invN;
  const float mxf = (float)mx, myf = (float)my;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  const int64_t G = (int64_t)gridDim.x * NT;
  for (int64_t i = (int64_t)blockIdx.x * NT + threadIdx.x; i < a.N; i += G) {
    double th = a.q[i], pp = a.p[i], dq = a.lq[i], dp = a.lp[i];
    double s, c, f;
    sc_of<MIXED>(th, s, c);
    if (MIXED)
      f = f2d_bits(__fsub_rn(__fmul_rn((float)c, myf), __fmul_rn((float)s, mxf)));
    else
      f = hmf_force_fp64(c, s, mx, my, a.invN);
    const double jv = fma(-fma(s, my, c * mx), dq, fma(c, A, s * B));
    pp = fma(a.b_adj, f, pp);
    dp = fma(a.b_adj, jv, dp);
    if (a.drift != 0.0) {
      th = fma(a.drift, pp, th);
      dq = fma(a.drift, dp, dq);
      sc_of<MIXED>(th, s, c);
      a0 += c;
      a1 += s;
      a2 = fma(c, dq, a2);
      a3 = fma(s, dq, a3);
      a.q[i] = th;
      a.lq[i] = dq;
    }
    a.p[i] = pp;
    a.lp[i] = dp;
  }
  if (a.drift != 0.0) grid_finish4(a0, a1, a2, a3, a.partials, a.s_out, a.ticket);
}

}  // namespace

int hmf_tangent_stage(md_ctx *c, double kick, double drift, double *dq, double *dp, const double *s_in,
                      double *s_out) {
  HmfAdjArgs a;
  a.q = c->q;
  a.p = c->p;
  a.lq = dq;
  a.lp = dp;
  a.N = c->N;
  a.invN = 1.0 / (double)c->N;
  a.s_in = s_in;
  a.b_adj = kick;
  a.b_undo = 0.0;
  a.drift = drift;
  a.partials = c->hmf_partials;
  a.s_out = s_out;
  a.ticket = c->hmf_ticket;
  const int g = grid_for(c, (const void *)hmf_tangent_stage_kernel<false>, c->N);
  if (c->prec == MD_MIXED)
    hmf_tangent_stage_kernel<true><<<g, NT, 0, c->stream>>>(a);
  else
    hmf_tangent_stage_kernel<false><<<g, NT, 0, c->stream>>>(a);
  MD_LAUNCHED(c);
  return MD_OK;
}
