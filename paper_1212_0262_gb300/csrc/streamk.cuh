// Unit ranges of the stream-K launches and the chunks of the finish phases: whole-number
// arithmetic shared by the kernels, the host code that sizes their grids and buffers, and the
// CPU tests, so that a launch and its kernels cannot disagree.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define SK_FN __host__ __device__ __forceinline__
#else
#define SK_FN static inline
#endif

// First unit of range c of U units cut into P ranges.
SK_FN int64_t unit_begin(int64_t U, int P, int64_t c) { return (U * c) / P; }
// CTA whose range holds unit u: max c with U c / P <= u.
SK_FN int64_t cta_of_unit(int64_t U, int P, int64_t u) { return ((u + 1) * P - 1) / U; }

// Triangular unit table of the Newton's-third-law form: row I (i-tile of m
// j-tiles) holds the j-tiles J = m I .. n_jt - 1.
SK_FN int64_t sym_rowstart(int64_t I, int64_t n_jt, int m) { return I * n_jt - (int64_t)m * I * (I - 1) / 2; }

// What the finish phase adds up for tile T of a system whose first unit is ubeg: `rows` rows of
// column partials and the row's segments, those of the ranges cf .. cl, each in chunks of at
// most ch.  Up to `direct` segments need no chunk: the CTA that finishes the tile reads them.
struct RowChunks {
  int64_t ubeg, cf, cl;  // the row's first unit, and the ranges that hold units of it
  int cols, segs;        // chunks of column-partial rows and of segments
};
SK_FN RowChunks row_chunks(int64_t U, int P, int64_t ubeg, int64_t n_jt, int m, int64_t T, int64_t rows, int ch,
                           int direct) {
  RowChunks r;
  r.ubeg = ubeg + sym_rowstart(T, n_jt, m);
  r.cf = cta_of_unit(U, P, r.ubeg);
  r.cl = cta_of_unit(U, P, ubeg + sym_rowstart(T + 1, n_jt, m) - 1);
  r.cols = (int)((rows + ch - 1) / ch);
  r.segs = r.cl - r.cf < direct ? 0 : (int)((r.cl - r.cf + ch) / ch);
  return r;
}

// The largest number of chunks over a system's tiles, which sizes the finish grid.  A sum of two
// rounded-up quotients, one rising and one falling with T: its maximum can be anywhere.
static inline int most_chunks(int64_t U, int P, int64_t ubeg, int64_t n_it, int m, bool diag, int ch,
                              int direct) {
  int most = 1;
  for (int64_t T = 0; T < n_it; T++) {
    const RowChunks r = row_chunks(U, P, ubeg, m * n_it, m, T, T + (diag ? 1 : 0), ch, direct);
    most = r.cols + r.segs > most ? r.cols + r.segs : most;
  }
  return most;
}
