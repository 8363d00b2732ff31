// Newton's-third-law variant of the Ring and 2D force stages: every
// unordered pair is evaluated once and its term added to both particles.  The
// paper evaluates every ordered pair (Sec. 3.2, tile algorithm) and leaves this
// variant out; it is one of the extensions its conclusion names.
//
// The summands are antisymmetric: with q_ij the term of particle i's sum,
//   Ring:  q_ij = S_ij dd_ij^(-3/2),  S_ji = -S_ij (sine of the opposite angle),
//          dd_ji = dd_ij (sin^2 of the half angle is even);
//   2D:    q_ij = r_ij / (|r_ij|^2 + eps),  r_ji = -r_ij;
// so f_j receives -q_ij from the evaluation of (i, j).
//
// Units.  i-tiles of TI = m TJ particles (m = TI/TJ), j-tiles of TJ.  Row I of
// the unit table holds the j-tiles J = m I .. n_jt - 1 (n_jt = m n_it), so
// rowstart(I) = I n_jt - m I (I - 1) / 2 and U = rowstart(n_it).  A unit whose
// j-tile lies inside its i-tile (J < m (I + 1), "diagonal") holds pairs of the
// tile's own particles: the FP32 Ring and 2D policies (tile_diag) evaluate the
// pairs above the diagonal once, as below, and only the squares on the diagonal
// (16 x 16 for Ring, 256 x 256 for 2D) for the i-rows alone; the other policies
// evaluate the whole TI x TJ block for the i-rows only, self pairs masked.  Every
// other unit evaluates its block once: the i-rows accumulate in registers across
// the CTA's consecutive units of the row (as in the one-sided kernel), and the sums over
// the block's i-rows for each of its TJ j's (warp butterflies, then the warps in
// a fixed order through shared memory) are stored as that unit's column partial
// (FP32, [U][TJ][NACC]).
//
// Pair phase (sym_pairs_kernel, stream-K).  Virtual CTA c (taken by the
// persistent CTAs in increasing order, take_vcta) covers units
// [U c / P, U (c+1) / P) in row-major order and writes the row partials of the
// rows it covers (rowfull[T] when it covered all of row T, else the one-sided
// kernel's two slots per virtual CTA) and the column partial of each off-diagonal
// unit (and of each diagonal one, with tile_diag).
//
// Finish phase (sym_finish_kernel).  Tile T needs its row partials and the
// column partials of the units (I', J), J in tile T, I' < T (I' <= T with
// tile_diag).  One CTA per (128 particles of a tile, chunk of rows I' or of row
// partials) sums its chunk per particle and component (column partials in compensated
// FP32, then one double); the last chunk to arrive (atomic ticket, no waiting) adds the
// chunk sums in order and runs the stage epilogue (kick, drift, new mirror record) for
// the 128 particles.  Every sum has a fixed order, so results are
// deterministic.  The finish phase spreads the O(N^2 / TJ) column reads over the
// whole GPU; finishing a tile inside the pair kernel instead serialised them on
// the few CTAs that cover the many short rows at the end of the order.
// Column partials take U TJ NACC floats: beyond kSymMaxColBytes the one-sided
// kernel runs instead.
#include <mutex>

#include "pairs_fx.cuh"
#include "pairs_impl.cuh"

namespace {

constexpr size_t kSymMaxColBytes = (size_t)16 << 30;  // Ring and 2D at N = 1e6 fit

struct SymArgs {
  int m;             // TI / TJ
  int nc;            // chunk slots per block in the finish phase
  int ch;            // column-partial rows or row segments per chunk
  double *rowfull;   // [n_it][NACC][TI] row partials of rows covered by one CTA
  void *colslot;     // [U][TJ][NACC] column partials of the units (Pol::ColT:
                     // FP32 for the mixed policies, FP64 for the FP64 ones)
  double *chunks;    // [blocks][nc][kFinishBlock][NACC] chunk sums
};

// Policies with integer pair arithmetic (pairs_fx.cuh): their row sums partly in shared
// memory, a unit's columns as integer limbs, and an FP64 form for units out of range.
template <class P, class = void>
struct IsFx : std::false_type {};
template <class P>
struct IsFx<P, std::void_t<decltype(P::FX)>> : std::true_type {};
// and with a rule on units of close particles, or on narrow records
template <class P, class = void>
struct HasClose : std::false_type {};
template <class P>
struct HasClose<P, std::void_t<decltype(P::CLOSE)>> : std::true_type {};
template <class P, class = void>
struct HasNarrow : std::false_type {};
template <class P>
struct HasNarrow<P, std::void_t<decltype(P::NARROW)>> : std::true_type {};

// Shared-memory bytes of a unit's column sums.
template <class Pol>
constexpr int sym_col_bytes() {
  if constexpr (IsFx<Pol>::value) return Pol::COL_BYTES;
  else return Pol::THREADS / 32 * Pol::TJ * Pol::NACC * (int)sizeof(typename Pol::ColT);
}

// Bytes of a tile turned into integers (FX).
template <class Pol>
constexpr int sym_stage_bytes() {
  if constexpr (IsFx<Pol>::value) return Pol::STAGE_BYTES;
  else return 16;
}

// Pair phase: every unit's block, row partials per CTA segment, column partials per unit.
template <class Pol>
__global__ void __launch_bounds__(Pol::THREADS, Pol::MINB) sym_pairs_kernel(PairArgs a, SymArgs s) {
  constexpr int THR = Pol::THREADS, NW = THR / 32;
  constexpr int TJ = Pol::TJ, NACC = Pol::NACC;
  constexpr int TILE_BYTES = TJ * Pol::JB;
  constexpr int CHUNKS = TILE_BYTES / 16;
  constexpr int64_t TI = (int64_t)THR * Pol::R;
  static_assert(TILE_BYTES % 16 == 0, "tile must be a whole number of 16-byte chunks");
  static_assert(TI % TJ == 0, "i-tiles must be whole numbers of j-tiles");
  using ColT = typename Pol::ColT;
  constexpr bool DIAG_SYM = HasDiagSym<Pol>::value;
  __shared__ __align__(16) unsigned char sbuf[2][TILE_BYTES];
  constexpr bool FX = IsFx<Pol>::value;
  __shared__ __align__(16) unsigned char colraw[sym_col_bytes<Pol>()];
  __shared__ double rowsm[FX ? THR * Pol::R * NACC : 1];
  __shared__ __align__(16) unsigned char staged[sym_stage_bytes<Pol>()];
  ColT *colsm = (ColT *)colraw;
  __shared__ unsigned s_vc;
  const int m = s.m;
  const unsigned char *mir = (const unsigned char *)a.mirror_in;
  auto prefetch = [&](int buf, int64_t jt) {
    const unsigned char *src = mir + jt * (int64_t)TILE_BYTES;
    for (int ch = threadIdx.x; ch < CHUNKS; ch += THR) cp_async16(&sbuf[buf][ch * 16], src + ch * 16);
    cp_async_commit();
  };
  bool rows_broad = true;  // FX: some row is broad, whatever the columns are
  auto load_rows = [&](typename Pol::State &st, int64_t i0) {
    if constexpr (FX) Pol::load(st, a.mirror_in, i0, a, rowsm);
    else Pol::load(st, a.mirror_in, i0);
    if constexpr (HasClose<Pol>::value) rows_broad = __syncthreads_or(st.flags & kFxBroad);
  };

  for (;;) {
    const int64_t cta = take_vcta(a.sched, s_vc);  // virtual CTA: its range and slots
    if (cta >= a.P) break;
    const int64_t u0 = unit_begin(a.U, a.P, cta), u1 = unit_begin(a.U, a.P, cta + 1);
    if (u0 >= u1) continue;

    typename Pol::State st;
    int64_t it = sym_row_of_unit(u0, a.n_it, a.n_jt, m);
    const int64_t first_row = it;
    int64_t jt = (int64_t)m * it + (u0 - sym_rowstart(it, a.n_jt, m));
    bool row_from_start = (jt == (int64_t)m * it);
    int64_t i0 = it * TI;
    load_rows(st, i0);
    prefetch(0, jt);

    for (int64_t u = u0; u < u1; u++) {
      const int buf = (int)((u - u0) & 1);
      const bool row_end = (jt + 1 == a.n_jt);
      const int64_t next_jt = row_end ? (int64_t)m * (it + 1) : jt + 1;
      if (u + 1 < u1) {
        prefetch(buf ^ 1, next_jt);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      bool wild = false;  // FX: a coordinate of the unit lies out of the fixed-point range
      if constexpr (FX) {
        int flags = 0, narrow = 0;
        for (int ch = threadIdx.x; ch < CHUNKS; ch += THR) {
          const int f = Pol::stage(sbuf[buf], ch, staged, a, i0);
          flags |= f;
          narrow += (f & kFxNarrow) != 0;
        }
        wild = __syncthreads_or((flags | st.flags) & kFxWild);
        if constexpr (HasClose<Pol>::value) {
          if (!rows_broad && !__syncthreads_or(flags & kFxBroad)) {
            const int64_t rows = a.N - i0, cols = a.N - jt * TJ;  // particles, padding follows
            if (cols > 0 && !(rows == 1 && cols == 1)) wild = true;
          }
        }
        if constexpr (HasNarrow<Pol>::value) {
          static_assert(CHUNKS <= 2 * THR, "at most two chunks per thread");
          int n = __syncthreads_count(narrow > 0);
          if (CHUNKS > THR) n += __syncthreads_count(narrow > 1);
          if (n >= Pol::NARROW && __syncthreads_or(st.flags & kFxNarrow)) wild = true;
        }
      } else {
        __syncthreads();
      }
      const bool diag = jt < (int64_t)m * (it + 1);
      if constexpr (FX) {
        if (!wild && diag) Pol::template unit<false>(st, sbuf[buf], staged, a, colraw, i0, jt * TJ);
        else if (!wild) Pol::template unit<true>(st, sbuf[buf], staged, a, colraw, i0, jt * TJ);
        else if (diag) Pol::template unit_wild<false>(st, sbuf[buf], a, colraw, i0, jt * TJ);
        else Pol::template unit_wild<true>(st, sbuf[buf], a, colraw, i0, jt * TJ);
      } else if (!diag) Pol::tile_sym(st, sbuf[buf], a, colsm);
      else if constexpr (DIAG_SYM) Pol::tile_diag(st, sbuf[buf], a, colsm, (int)(jt - (int64_t)m * it));
      else Pol::template tile<true>(st, sbuf[buf], a, i0, jt * TJ);
      __syncthreads();
      if (!diag || DIAG_SYM) {
        // column partial of this unit: the warps' sums in a fixed order (colsm is
        // rewritten only after the next unit's first barrier)
        ColT *dst = (ColT *)s.colslot + u * (int64_t)(TJ * NACC);
        for (int idx = threadIdx.x; idx < TJ * NACC; idx += THR) {
          if constexpr (FX) {
            dst[idx] = Pol::column(colraw, idx, wild, a);
          } else {
            ColT v = colsm[idx];
  #pragma unroll
            for (int w = 1; w < NW; w++) v += colsm[w * TJ * NACC + idx];
            dst[idx] = v;
          }
        }
      }
      if (row_end || u + 1 == u1) {
        // this CTA's part of row it
        if constexpr (FX) Pol::flush(st, a);
        double *sp = (row_end && row_from_start)
                         ? s.rowfull + it * NACC * TI
                         : a.slots + ((cta * 2 + (it == first_row ? 0 : 1)) * NACC) * TI;
  #pragma unroll
        for (int r = 0; r < Pol::NR; r++) {
          double ex[NACC];
          Pol::total(st, r, ex);
          const int lr = Pol::row_of(r);  // row offset in the tile, -1: another lane's
          if (lr >= 0)
  #pragma unroll
            for (int d = 0; d < NACC; d++) sp[d * TI + lr] = ex[d];
        }
        if (row_end && u + 1 < u1) {
          it++;
          row_from_start = true;
          i0 = it * TI;
          load_rows(st, i0);
        }
      }
      jt = next_jt;
    }
  }
  vcta_done(a.sched);
}

// Finish phase, one CTA per (block b of kFinishBlock particles, chunk c).  The force of a
// particle of tile T is the sum of its row's segments (one per virtual CTA that covers part of
// row T) minus the column partials of the rows I' < T (I' <= T with tile_diag).  A chunk CTA
// sums s.ch column partials (compensated FP32, or FP64) or s.ch segments per particle and
// component into one double; the last chunk of the block to arrive (atomic ticket, no
// waiting) adds the chunk sums, segments first, and runs the stage epilogue.
// Small tiles of few rows are all latency: with one CTA per tile, which added up to 64 segments
// one after the other for 1024 particles, this phase took 290 us at N = 16,385 (2D, mixed)
// beside 73 us for the pair phase; split by blocks and segments it takes 13.  Microseconds per
// force, before and after: mixed Ring N = 4,096 31.8, 22.6; 2D N = 4,096 71.7, 33.3, N = 16,385
// 282, 86, N = 65,536 763, 700; 3D N = 16,385 163, 110; FP64 Ring N = 4,096 107, 84.  At N = 131,072
// (Ring) and 262,144 (2D), where it is bound by the column reads, 87 -> 41 and 180 -> 135 us.
constexpr int kFinishBlock = 128;

template <class Pol, int MODEL, bool MIXED, int MODE>
__global__ void __launch_bounds__(kFinishBlock * Pol::NACC) sym_finish_kernel(PairArgs a, SymArgs s) {
  constexpr int NACC = Pol::NACC, TJ = Pol::TJ;
  constexpr int64_t TI = (int64_t)Pol::THREADS * Pol::R;
  constexpr int FT = kFinishBlock * NACC;          // threads: one per (particle, component)
  constexpr int SB = (int)(TI / kFinishBlock);     // blocks per tile
  static_assert(TI % kFinishBlock == 0, "whole blocks per tile");
  __shared__ bool s_last;
  const int64_t b = blockIdx.x / s.nc, T = b / SB;
  const int c = (int)(blockIdx.x % s.nc), sb = (int)(b % SB);
  const int m = s.m;
  const int64_t rows = T + (HasDiagSym<Pol>::value ? 1 : 0);  // column-partial rows I of tile T
  const RowChunks rc = row_chunks(a.U, a.P, 0, a.n_jt, m, T, rows, s.ch, 0);
  const int64_t cf = rc.cf, cl = rc.cl;
  const int nchc = rc.cols, nch = nchc + rc.segs;
  if (c >= nch) return;
  double *chunk = s.chunks + b * s.nc * FT;
  const int lr = sb * kFinishBlock + threadIdx.x / NACC, d = threadIdx.x % NACC;
  double v = 0.0;
  if (c < nchc) {
    using ColT = typename Pol::ColT;
    const ColT *col = (const ColT *)s.colslot;
    const int64_t I_lo = (int64_t)c * s.ch, I_hi = min(rows, I_lo + s.ch);
    const int jsub = lr / TJ, rest = (lr % TJ) * NACC + d;
    CompSum cs{0.f, 0.f};  // FP32 column partials: compensated FP32 sum
    // unit (I2, T m + jsub) = rowstart(I2) + T m + jsub - m I2; from I2 to I2 + 1 it
    // advances by the length of row I2 minus m, i.e. n_jt - m (I2 + 1)
    int64_t off = (sym_rowstart(I_lo, a.n_jt, m) + (T * m + jsub - (int64_t)m * I_lo)) * (TJ * NACC) + rest;
    int64_t step = (a.n_jt - (int64_t)m * (I_lo + 1)) * (TJ * NACC);
    const int64_t dstep = (int64_t)m * (TJ * NACC);
#pragma unroll 8
    for (int64_t I2 = I_lo; I2 < I_hi; I2++) {
      if constexpr (sizeof(ColT) == 4) csum_add(cs, __ldcg(col + off));
      else v += __ldcg(col + off);
      off += step;
      step -= dstep;
    }
    v = sizeof(ColT) == 4 ? -csum_total(cs) : -v;
  } else if (cf == cl) {
    v = __ldcg(s.rowfull + (T * NACC + d) * TI + lr);
  } else {
    // virtual CTA c2 > cf begins inside row T: its first slot; cf may begin in an earlier row
    const int64_t lo = cf + (int64_t)(c - nchc) * s.ch, hi = min(cl + 1, lo + s.ch);
    const bool cf_first = unit_begin(a.U, a.P, cf) >= rc.ubeg;
    const double *src = a.slots + d * TI + lr;
#pragma unroll 8
    for (int64_t c2 = lo; c2 < hi; c2++)
      v += __ldcg(src + (c2 * 2 + (c2 > cf || cf_first ? 0 : 1)) * (NACC * TI));
  }
  chunk[(int64_t)c * FT + threadIdx.x] = v;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&a.tickets[b], 1u) + 1u == (unsigned)nch;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int64_t i = b * kFinishBlock + threadIdx.x;
  if (threadIdx.x < kFinishBlock && i < a.N) {
    double tot[NACC];
#pragma unroll
    for (int e = 0; e < NACC; e++) tot[e] = 0.0;
    const double *mine = chunk + threadIdx.x * NACC;
#pragma unroll 2
    for (int k = 0; k < nch; k++) {
      const int64_t at = (int64_t)(k < nch - nchc ? nchc + k : k - (nch - nchc)) * FT;
#pragma unroll
      for (int e = 0; e < NACC; e++) tot[e] += __ldcg(mine + at + e);
    }
    finish<Pol, MODEL, MIXED, MODE>(a, i, tot);
  }
  if (threadIdx.x == 0) a.tickets[b] = 0u;
}

// ------------------------------------------------------------ host side ---

template <class Pol, int MODEL, bool MIXED, int MODE>
int launch_sym(md_ctx *c, PairArgs a) {
  constexpr int THR = Pol::THREADS;
  constexpr int64_t TI = (int64_t)THR * Pol::R;
  constexpr int TJ = Pol::TJ, NACC = Pol::NACC;
  auto kern = sym_pairs_kernel<Pol>;
  // the grid is sized for the occupancy limit: make the shared-memory carveout allow it
  // (once per kernel, on the first call, which runs before any stream capture)
  static std::once_flag carveout_once;
  std::call_once(carveout_once, [&] {
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  });
  int occ = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, THR, 0);
  if (occ < 1) occ = 1;
  if (c->pt.ctas_per_sm > 0 && c->pt.ctas_per_sm < occ) occ = c->pt.ctas_per_sm;
  SymArgs s{};
  s.m = (int)(TI / TJ);
  a.N = c->N;
  a.n_it = (c->N + TI - 1) / TI;
  a.n_jt = s.m * a.n_it;
  a.U = sym_rowstart(a.n_it, a.n_jt, s.m);
  const int64_t G = std::min<int64_t>((int64_t)c->nsm * occ, a.U);  // CTAs
  // virtual CTAs per CTA, measured at the bench sizes (sweeps of 1-16 show sharp dips at
  // single values, 4 for these two among them): 8 for the Ring tensor-core kernel, 3 for
  // the FP64 3D kernel, 4 for the others
  int kv = c->pt.vcta > 0 ? c->pt.vcta : Pol::FMT == 1 ? 8 : (MODEL == MD_GRAV3D && !MIXED) ? 3 : 4;
  // integer policies, whose units are long: below 16 per CTA one range each.  Neither is best
  // throughout; microseconds per force with one range and with four at N = 4,096, 8,192, 12,000,
  // 16,385: Ring 86, 83; 261, 266; 508, 501; 916, 926; 2D 85, 80; 254, 268; 492, 481; 910, 911;
  // 3D 124, 115; 390, 412; 797, 774; 1470, 1459.
  if (IsFx<Pol>::value && c->pt.vcta == 0 && a.U < 16 * G) kv = 1;
  a.P = (int)vcta_count(G, a.U, kv, IsFx<Pol>::value ? 1 : 16);
  int rc = ensure_pair_buffers(c, (int)TI, a.P, NACC);
  if (rc) return rc;
  // Chunks: the tile with the most sizes the grid (spare CTAs of the others leave at once).
  // Longer chunks where the column partials are many and narrow (Ring FP32: the chunk sums
  // would cost an eighth of their traffic).
  s.ch = Pol::NACC == 1 && a.n_it >= 256 ? 64 : 16;
  s.nc = most_chunks(a.U, a.P, 0, a.n_it, s.m, HasDiagSym<Pol>::value, s.ch, 0);
  const int64_t blocks = a.n_it * (TI / kFinishBlock);
  const size_t need_row = (size_t)a.n_it * NACC * TI * sizeof(double);
  const size_t need_col = (size_t)a.U * TJ * NACC * sizeof(typename Pol::ColT);
  const size_t need_chunk = (size_t)blocks * s.nc * NACC * kFinishBlock * sizeof(double);
  if (need_row > c->sym_rowfull_bytes) {
    dev_free(c->sym_rowfull);
    c->sym_rowfull = (double *)dev_alloc(need_row);
    c->sym_rowfull_bytes = c->sym_rowfull ? need_row : 0;
    if (!c->sym_rowfull) return set_err(c, MD_ENOMEM, "symmetric row partials: %zu bytes", need_row);
  }
  if (need_col > c->sym_colslot_bytes) {
    dev_free(c->sym_colslot);
    c->sym_colslot = dev_alloc(need_col);
    c->sym_colslot_bytes = c->sym_colslot ? need_col : 0;
    if (!c->sym_colslot) return set_err(c, MD_ENOMEM, "symmetric column partials: %zu bytes", need_col);
  }
  if (need_chunk > c->sym_chunk_bytes) {
    dev_free(c->sym_chunks);
    c->sym_chunks = (double *)dev_alloc(need_chunk);
    c->sym_chunk_bytes = c->sym_chunks ? need_chunk : 0;
    if (!c->sym_chunks) return set_err(c, MD_ENOMEM, "symmetric chunk sums: %zu bytes", need_chunk);
  }
  s.rowfull = c->sym_rowfull;
  s.colslot = c->sym_colslot;
  s.chunks = c->sym_chunks;
  a.mirror_in = c->mirror[c->mirror_cur];
  a.mirror_out = c->mirror[1 - c->mirror_cur];
  a.q = c->q;
  a.p = c->p;
  a.epsd = MODEL == MD_RING ? 0.5 * c->eps : c->eps;  // 2D, 3D, sheets: eps
  a.slots = c->sk_slots;
  a.tickets = c->sk_tickets;
  a.sched = pair_sched(c);
  if constexpr (MODE == STAGE_ADJOINT || MODE == STAGE_TANGENT) {
    // the spread of the v of the records (lambda_p, or dq), for the unit of the sums of j
    if (!c->fx_vrange) {
      c->fx_vrange = (unsigned *)dev_alloc(2 * sizeof(unsigned));
      if (!c->fx_vrange) return set_err(c, MD_ENOMEM, "reverse stage scratch");
      MD_CUDA(c, cudaMemsetAsync(c->fx_vrange, 0, 2 * sizeof(unsigned), c->stream));
    }
    const int64_t g = std::min<int64_t>((c->N + 255) / 256, c->nsm);
    a.vrange = c->fx_vrange + c->fx_vcur;
    fx_vrange_kernel<<<(int)g, 256, 0, c->stream>>>(MODE == STAGE_ADJOINT ? a.lp : a.lq, c->N, c->fx_vrange + c->fx_vcur,
                                                   c->fx_vrange + (1 - c->fx_vcur));
    MD_LAUNCHED(c);
    c->fx_vcur = 1 - c->fx_vcur;
  }
  kern<<<(int)G, THR, 0, c->stream>>>(a, s);
  MD_LAUNCHED(c);
  sym_finish_kernel<Pol, MODEL, MIXED, MODE><<<blocks * s.nc, kFinishBlock * NACC, 0, c->stream>>>(a, s);
  MD_LAUNCHED(c);
  if (MODE == STAGE_KICK_DRIFT || ((MODE == STAGE_ADJOINT || MODE == STAGE_TANGENT) && a.drift != 0.0))
    c->mirror_cur = 1 - c->mirror_cur;
  return MD_OK;
}

// Bytes of the column partials: one per unit, column and component.
size_t column_bytes(int64_t N, int64_t TI, int64_t TJ, int nacc, int col) {
  const int64_t m = TI / TJ, n_it = (N + TI - 1) / TI;
  return (size_t)sym_rowstart(n_it, m * n_it, (int)m) * TJ * nacc * col;
}

// The context's column buffer made this large; false if the memory is not to be had, the old
// buffer then kept (other stages, and graphs of them, use it).  Inside a caller's capture, where
// nothing can be allocated, the stage itself reports what is missing.
bool reserve_columns(md_ctx *c, size_t need) {
  if (need <= c->sym_colslot_bytes) return true;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(c->stream, &st) != cudaSuccess) cudaGetLastError();
  else if (st != cudaStreamCaptureStatusNone) return true;
  void *buf = dev_alloc(need);
  if (!buf) return false;
  dev_free(c->sym_colslot);
  c->sym_colslot = buf;
  c->sym_colslot_bytes = need;
  return true;
}

// FP64 stages with integer pair arithmetic: Fx<rows per thread, j-tile>.  A unit is one
// CTA's work of 128 rows x tile, 256 x tile, 512 x tile pairs, and a pair takes thousands of
// cycles of latency, so small systems want small units (N = 1,000, microseconds per force,
// 2D: 45 with <1, 64>, 58 with <2, 64>, 147 with <4, 128>), larger ones more rows to share
// the column reductions (N = 16,385: 967, 915, 1020; N = 8,192: 264, 281, 343).  <4, 128> needs
// half the column storage of <2, 64> and is 2-5% slower.
constexpr int64_t kFxSmall = 10000, kFxLarge = 262144;
// Where it does not fit (the caller's allocator may be bounded), <4, 128> runs at every size.
template <template <int, int> class Fx, int MODEL, int MODE>
int fx_dispatch(md_ctx *c, PairArgs a) {
  constexpr int NACC = Fx<4, 128>::NACC, COL = (int)sizeof(typename Fx<4, 128>::ColT);
  if (c->N <= kFxLarge && !c->fx_wide_units) {
    const int rows = c->N <= kFxSmall ? 128 : 256;
    if (!reserve_columns(c, column_bytes(c->N, rows, 64, NACC, COL)))
      c->fx_wide_units = true;  // kept: the choice must not change inside a capture
    else if (rows == 128)
      return launch_sym<Fx<1, 64>, MODEL, false, MODE>(c, a);
    else
      return launch_sym<Fx<2, 64>, MODEL, false, MODE>(c, a);
  }
  return launch_sym<Fx<4, 128>, MODEL, false, MODE>(c, a);
}

template <int MODEL, bool MIXED, int MODE>
int sym_dispatch(md_ctx *c, PairArgs a) {
  if constexpr (MODEL == MD_GRAV3D) {
    if constexpr (MIXED) return launch_sym<Grav3DMixed<4, 256, MODE>, MODEL, true, MODE>(c, a);
    else if (fx_grav_applies(c->eps)) return fx_dispatch<FxGrav3D, MODEL, MODE>(c, a);
    else return launch_sym<Grav3DF64<4, 128, MODE>, MODEL, false, MODE>(c, a);
  } else if constexpr (MODEL == MD_SHEET1D) {
    // registers for 5 CTAs per SM (96, no spills): 1.4% faster than for 4 at N = 262,144
    if constexpr (MIXED) return launch_sym<SheetMixed<8, 256, MODE, 5>, MODEL, true, MODE>(c, a);
    else return launch_sym<SheetF64<4, 128, MODE>, MODEL, false, MODE>(c, a);
  } else if constexpr (!MIXED) {
    // FP64 tiles: 4 rows per thread, so that the column butterflies' FP64 adds are shared
    if constexpr (MODEL == MD_RING) {
      if (fx_ring_applies(c->eps)) return fx_dispatch<RingFx, MODEL, MODE>(c, a);
      return launch_sym<RingF64<4, 128, MODE>, MODEL, false, MODE>(c, a);
    } else {
      if (fx_grav_applies(c->eps)) return fx_dispatch<FxGrav2D, MODEL, MODE>(c, a);
      return launch_sym<GravF64<4, 128, MODE>, MODEL, false, MODE>(c, a);
    }
  } else if constexpr (MODEL == MD_RING) {
    return launch_sym<RingTC<4, 256, MODE>, MODEL, true, MODE>(c, a);
  } else {
    return launch_sym<GravMixed<8, 256, MODE>, MODEL, true, MODE>(c, a);
  }
}

template <int MODEL, bool MIXED>
int sym_mode(md_ctx *c, int mode, PairArgs a) {
  switch (mode) {
  case STAGE_KICK_DRIFT: return sym_dispatch<MODEL, MIXED, STAGE_KICK_DRIFT>(c, a);
  case STAGE_KICK_ONLY: return sym_dispatch<MODEL, MIXED, STAGE_KICK_ONLY>(c, a);
  default: return sym_dispatch<MODEL, MIXED, STAGE_FORCE_ONLY>(c, a);
  }
}

}  // namespace

// Column partials need U TJ NACC floats, U ~ N^2 / (2 TI TJ): the variant runs
// while they fit in kSymMaxColBytes.
bool sym_applies(const md_ctx *c) {
  if (!c->pt.symmetric) return false;
  int64_t TI, TJ, nacc = c->dim, colbytes;
  if (c->model == MD_HMF) return false;
  if (c->prec == MD_FP64 && c->pt.r_fp64 != 2) return false;
  if (sheet_rank_applies(c)) return true;  // no column partials
  if (c->prec == MD_FP64) {
    TI = 512, TJ = 128, colbytes = 8;
  } else if (c->model == MD_GRAV3D) {
    TI = 512, TJ = 256, colbytes = 4;
  } else if (c->model == MD_SHEET1D) {
    TI = 1024, TJ = 256, colbytes = 4;
  } else if (c->model == MD_RING) {
    if (!c->pt.ring_tc || c->pt.ring_tc == 2 || c->pt.r_mixed == 4) return false;
    TI = 256, TJ = 256, colbytes = 4;
  } else if (c->model == MD_GRAV2D) {
    if (c->pt.r_mixed == 4) return false;
    TI = 1024, TJ = 256, colbytes = 4;
  } else {
    return false;
  }
  const int64_t m = TI / TJ, n_it = (c->N + TI - 1) / TI, n_jt = m * n_it;
  const int64_t U = n_it * n_jt - m * n_it * (n_it - 1) / 2;
  return (size_t)U * TJ * nacc * colbytes <= kSymMaxColBytes;
}

int sym_pair_stage(md_ctx *c, int mode, double kick, double drift, double *fout) {
  if (sheet_rank_applies(c)) return sheet_rank_stage(c, mode, kick, drift, fout);
  PairArgs a{};
  a.kick = kick;
  a.drift = drift;
  a.fout = fout;
  const bool mixed = c->prec == MD_MIXED;
  if (c->model == MD_RING) return mixed ? sym_mode<MD_RING, true>(c, mode, a) : sym_mode<MD_RING, false>(c, mode, a);
  if (c->model == MD_GRAV3D)
    return mixed ? sym_mode<MD_GRAV3D, true>(c, mode, a) : sym_mode<MD_GRAV3D, false>(c, mode, a);
  if (c->model == MD_SHEET1D)
    return mixed ? sym_mode<MD_SHEET1D, true>(c, mode, a) : sym_mode<MD_SHEET1D, false>(c, mode, a);
  return mixed ? sym_mode<MD_GRAV2D, true>(c, mode, a) : sym_mode<MD_GRAV2D, false>(c, mode, a);
}

// Reverse and tangent stages in the symmetric form: FP64 2D with the integer pair arithmetic,
// while its six column partials fit, also in the memory there is (one-sided stages need none).
bool sym_reverse_applies(md_ctx *c) {
  if (!c->pt.symmetric || c->prec != MD_FP64 || c->pt.r_fp64 != 2 || c->sym_reverse_off) return false;
  if (c->model != MD_GRAV2D || !fx_grav_applies(c->eps)) return false;
  const size_t need = column_bytes(c->N, c->N <= kFxSmall ? 128 : 256, 64, 6, sizeof(double));
  if (need > kSymMaxColBytes) return false;
  c->sym_reverse_off = !reserve_columns(c, need);
  return !c->sym_reverse_off;
}

template <int MODE>
int sym_reverse(md_ctx *c, const PairArgs &a) {
  if (c->N <= kFxSmall) return launch_sym<FxGrav2DAdj<1, 64>, MD_GRAV2D, false, MODE>(c, a);
  return launch_sym<FxGrav2DAdj<2, 64>, MD_GRAV2D, false, MODE>(c, a);
}

int sym_reverse_stage(md_ctx *c, int mode, double kick, double undo, double drift, double *lq, double *lp,
                      double *epsacc) {
  PairArgs a{};
  a.kick = kick;
  a.undo = undo;
  a.drift = drift;
  a.lq = lq;
  a.lp = lp;
  a.epsacc = epsacc;
  return mode == STAGE_ADJOINT ? sym_reverse<STAGE_ADJOINT>(c, a) : sym_reverse<STAGE_TANGENT>(c, a);
}
