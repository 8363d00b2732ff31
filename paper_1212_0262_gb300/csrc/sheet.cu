// Unsoftened 1D sheets (eps = 0): the force by counting ranks.
//
// f_i = -(1/N) sum_j sign(x_i - x_j) = -(1/N) (#{x_j < x_i} - #{x_j > x_i}): the counts are
// whole numbers, so any way of finding them gives the pair sums' result bit for bit.  Two
// kernels per stage instead of N^2 comparisons:
//   1. tiles of TS positions, as order-preserving integer keys, are sorted, one tile per CTA
//      (bitonic network: strides below 8 in registers, below 256 by shuffles, the rest
//      through shared memory);
//   2. every particle finds its place in every sorted tile by a search in shared memory
//      (log2 TS steps), which gives both counts, and runs the stage's epilogue.  The tile
//      is stored as an implicit search tree (level by level): in sorted order the probes of
//      the early steps would all fall on one bank.
// FP32 mode counts on the FP32 positions, as the pair kernels decide their signs; equal
// keys count neither way.  A NaN position counts for nobody and feels nothing in FP32
// (both comparisons false); in FP64 the pair kernels compare integer keys, where it has a
// place like any other value.
//
// N^2 / TS log2 TS shared-memory probes replace N^2 / 2 pair terms.  Microseconds per stage,
// pair kernel -> ranks: FP32 N = 256: 15.9 -> 10.3, 4,096: 58.7 -> 11.8, 100,003: 933 -> 34.8
// (sort 12.9, searches 25.3 under ncu), 262,144: 5636 -> 75.7, 10^6: 73.5 -> 0.60 ms; FP64
// N = 256: 14.8 -> 14.3, 100,003: 2024 -> 53.6, 262,144: 13258 -> 156.  The sort is bound by its
// shuffles and by one CTA per tile, the searches by shared-memory bank conflicts (46% of the
// L1 throughput); sorted order instead of the tree: 68.7 us at N = 100,003.
#include "pairs_impl.cuh"

namespace {

constexpr int kSortKeys = 8;  // keys per thread of the sort
constexpr int kRankThreads = 512;

// Place in the search tree of the element with sorted index s of a tile of TS: node 1 is
// the root, node k has the children 2k and 2k + 1; the last element goes to slot 0.
template <int TS>
__device__ __forceinline__ int tree_slot(int s) {
  constexpr int L = TS == 2048 ? 11 : TS == 4096 ? 12 : 13;
  static_assert(TS == 1 << L, "tile size");
  const int r = s + 1, tz = __ffs(r) - 1;
  return r == TS ? 0 : (1 << (L - 1 - tz)) + (r >> (tz + 1));
}

template <bool MIXED>
struct SheetKey;
template <>
struct SheetKey<true> {
  using T = unsigned;
  static constexpr T kPad = 0xffffffffu;
  // key of record i (the mirror holds -(float)x): increasing with x, NaN the largest
  __device__ static T of(const void *mirror, int64_t i) {
    const float x = -((const float *)mirror)[i] + 0.f;  // -0 as +0
    const unsigned b = __float_as_uint(x);
    return x != x ? kPad : b ^ ((unsigned)((int)b >> 31) | 0x80000000u);
  }
};
template <>
struct SheetKey<false> {
  using T = unsigned long long;
  static constexpr T kPad = 0xffffffffffffffffull;
  __device__ static T of(const void *mirror, int64_t i) {
    return ((const unsigned long long *)mirror)[i] ^ 0x8000000000000000ull;
  }
};

template <class T>
__device__ __forceinline__ void order(T &a, T &b, bool up) {
  const T lo = a < b ? a : b, hi = a < b ? b : a;
  a = up ? lo : hi;
  b = up ? hi : lo;
}

// Sorts tile blockIdx.x of the keys of mirror[0 .. N) into sorted; valid[tile] = its keys
// that are counted (FP32: not NaN).  E keys per thread, in blocks.
template <bool MIXED, int TS>
__global__ void __launch_bounds__(TS / kSortKeys) sheet_sort_kernel(const void *__restrict__ mirror, int64_t N,
                                                                  typename SheetKey<MIXED>::T *__restrict__ sorted,
                                                                  int *__restrict__ valid) {
  using K = SheetKey<MIXED>;
  using T = typename K::T;
  constexpr int E = kSortKeys, THR = TS / E;
  extern __shared__ __align__(16) unsigned char smraw[];
  T *sm = (T *)smraw;
  const int64_t base = (int64_t)blockIdx.x * TS;
  const int t = threadIdx.x;
  T v[E];
#pragma unroll
  for (int e = 0; e < E; e++) {  // coalesced; any order will do
    const int64_t i = base + e * THR + t;
    v[e] = i < N ? K::of(mirror, i) : K::kPad;
  }
  for (int k = 2; k <= TS; k <<= 1) {
    // strides of at least 32 E: partners in other warps
    for (int j = k >> 1; j >= 32 * E; j >>= 1) {
      __syncthreads();
#pragma unroll
      for (int e = 0; e < E; e++) sm[e * THR + t] = v[e];
      __syncthreads();
      const int pt = t ^ (j / E);
      const bool up = ((t * E) & k) == 0, low = (t & (j / E)) == 0;
#pragma unroll
      for (int e = 0; e < E; e++) {
        const T o = sm[e * THR + pt];
        v[e] = (v[e] < o) == (low == up) ? v[e] : o;
      }
    }
    const bool up_t = ((t * E) & k) == 0;
    for (int j = min(k >> 1, 16 * E); j >= E; j >>= 1) {  // partners in the warp
      const bool low = (t & (j / E)) == 0;
#pragma unroll
      for (int e = 0; e < E; e++) {
        const T o = __shfl_xor_sync(0xffffffffu, v[e], j / E);
        v[e] = (v[e] < o) == (low == up_t) ? v[e] : o;
      }
    }
#pragma unroll
    for (int j = E / 2; j >= 1; j >>= 1) {  // in the thread
      if (j < k) {
#pragma unroll
        for (int e = 0; e < E; e++)
          if ((e & j) == 0) order(v[e], v[e ^ j], ((t * E + e) & k) == 0);
      }
    }
  }
  T *out = sorted + base;
#pragma unroll
  for (int e = 0; e < E; e++) out[tree_slot<TS>(t * E + e)] = v[e];
  int n = 0;
#pragma unroll
  for (int e = 0; e < E; e++) n += base + t * E + e < N && (!MIXED || v[e] != K::kPad);
  // FP32: the keys that are not NaN come first; FP64: all particles of the tile
  __shared__ int total;
  if (t == 0) total = 0;
  __syncthreads();
  n = __reduce_add_sync(0xffffffffu, n);
  if ((t & 31) == 0) atomicAdd(&total, n);
  __syncthreads();
  if (t == 0) valid[blockIdx.x] = MIXED ? total : (int)min((int64_t)TS, N - base);
}

// The counts of every particle over all sorted tiles and the stage's epilogue.
template <bool MIXED, int TS, int MODE, int Q>
__global__ void __launch_bounds__(kRankThreads) sheet_rank_kernel(PairArgs a,
                                                                  const typename SheetKey<MIXED>::T *__restrict__ sorted,
                                                                  const int *__restrict__ valid, int ntiles) {
  using K = SheetKey<MIXED>;
  using T = typename K::T;
  constexpr int CHUNKS = TS * (int)sizeof(T) / 16;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int64_t i0 = (int64_t)blockIdx.x * (kRankThreads * Q) + threadIdx.x;
  auto prefetch = [&](int tile) {
    unsigned char *dst = smraw + (tile & 1) * (TS * (int)sizeof(T));
    const unsigned char *src = (const unsigned char *)(sorted + (int64_t)tile * TS);
    for (int ch = threadIdx.x; ch < CHUNKS; ch += kRankThreads) cp_async16(dst + ch * 16, src + ch * 16);
    cp_async_commit();
  };
  prefetch(0);
  T key[Q];
  long long less[Q], more[Q];
#pragma unroll
  for (int u = 0; u < Q; u++) {
    const int64_t i = i0 + u * kRankThreads;
    key[u] = i < a.N ? K::of(a.mirror_in, i) : K::kPad;
    less[u] = more[u] = 0;
  }
  for (int tile = 0; tile < ntiles; tile++) {
    if (tile + 1 < ntiles) {
      prefetch(tile + 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();
    const T *sm = (const T *)(smraw + (tile & 1) * (TS * (int)sizeof(T)));
    const int nv = valid[tile];
    const T last = sm[0];
    int k[Q];
    T at[Q];  // the smallest key not below, on the path
#pragma unroll
    for (int u = 0; u < Q; u++) {
      k[u] = 1;
      at[u] = last;
    }
#pragma unroll
    for (int h = TS; h > 1; h >>= 1)
#pragma unroll
      for (int u = 0; u < Q; u++) {
        const T n = sm[k[u]];
        const bool below = n < key[u];
        at[u] = below ? at[u] : n;
        k[u] = 2 * k[u] + below;
      }
#pragma unroll
    for (int u = 0; u < Q; u++) {
      int lt = k[u] - TS;                                    // keys below key
      if (lt == TS - 1 && last < key[u]) lt = TS;
      int le = lt;                                           // keys up to and with key
      if (at[u] == key[u]) {                                 // equal keys: search for their end
        int j = 1;
#pragma unroll 1
        for (int h = TS; h > 1; h >>= 1) j = 2 * j + (sm[j] <= key[u]);
        le = j - TS;
        if (le == TS - 1 && last <= key[u]) le = TS;
      }
      less[u] += lt < nv ? lt : nv;
      more[u] += nv - (le < nv ? le : nv);
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < Q; u++) {
    const double acc = MIXED && key[u] == K::kPad ? 0.0 : (double)(less[u] - more[u]);
    finish_forward<MD_SHEET1D, MIXED, MODE, 0>(a, i0 + u * kRankThreads, &acc);
  }
}

template <bool MIXED, int TS, int MODE, int Q>
int launch_search(md_ctx *c, const PairArgs &a, const void *sorted, const int *valid, int ntiles) {
  using T = typename SheetKey<MIXED>::T;
  constexpr int kTwo = 2 * TS * (int)sizeof(T);  // two tiles
  auto kern = sheet_rank_kernel<MIXED, TS, MODE, Q>;
  if (kTwo > 48 * 1024) MD_CUDA(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTwo));
  const int64_t g = (c->N + kRankThreads * Q - 1) / (kRankThreads * Q);
  kern<<<(unsigned)g, kRankThreads, kTwo, c->stream>>>(a, (const T *)sorted, valid, ntiles);
  MD_LAUNCHED(c);
  return MD_OK;
}

template <bool MIXED, int TS, int MODE>
int launch_rank(md_ctx *c, PairArgs a) {
  using T = typename SheetKey<MIXED>::T;
  const int ntiles = (int)((c->N + TS - 1) / TS);
  const size_t keys = (size_t)ntiles * TS * sizeof(T), need = keys + (size_t)ntiles * sizeof(int);
  if (need > c->sym_colslot_bytes) {
    dev_free(c->sym_colslot);
    c->sym_colslot = dev_alloc(need);
    c->sym_colslot_bytes = c->sym_colslot ? need : 0;
    if (!c->sym_colslot) return set_err(c, MD_ENOMEM, "sheets: sorted keys: %zu bytes", need);
  }
  T *sorted = (T *)c->sym_colslot;
  int *valid = (int *)((char *)c->sym_colslot + keys);
  a.N = c->N;
  a.mirror_in = c->mirror[c->mirror_cur];
  a.mirror_out = c->mirror[1 - c->mirror_cur];
  a.q = c->q;
  a.p = c->p;
  a.epsd = 0.0;
  auto sort = sheet_sort_kernel<MIXED, TS>;
  constexpr int kOne = TS * (int)sizeof(T);
  if (kOne > 48 * 1024) MD_CUDA(c, cudaFuncSetAttribute(sort, cudaFuncAttributeMaxDynamicSharedMemorySize, kOne));
  sort<<<ntiles, TS / kSortKeys, kOne, c->stream>>>(a.mirror_in, c->N, sorted, valid);
  MD_LAUNCHED(c);
  // particles per thread: one while the CTAs fill the SMs at most twice, then two and four
  // (every CTA reads every tile once)
  const int64_t fill = 2 * (int64_t)c->nsm * kRankThreads;
  const int rc = c->N <= fill       ? launch_search<MIXED, TS, MODE, 1>(c, a, sorted, valid, ntiles)
                 : c->N <= 2 * fill ? launch_search<MIXED, TS, MODE, 2>(c, a, sorted, valid, ntiles)
                                    : launch_search<MIXED, TS, MODE, 4>(c, a, sorted, valid, ntiles);
  if (rc) return rc;
  if (MODE == STAGE_KICK_DRIFT) c->mirror_cur = 1 - c->mirror_cur;
  return MD_OK;
}

// Tile size: the sort's time grows with the tile (one CTA each; 25 us for 8192 keys with
// 1024 threads), the searches' falls: N = 100,003 sorts 25 tiles of 4096 in 13 us.
constexpr int64_t kRank2048 = 32768, kRank4096 = 131072;
template <bool MIXED, int MODE>
int rank_tiles(md_ctx *c, const PairArgs &a) {
  if (c->N <= kRank2048) return launch_rank<MIXED, 2048, MODE>(c, a);
  if (!MIXED || c->N <= kRank4096) return launch_rank<MIXED, 4096, MODE>(c, a);
  return launch_rank<MIXED, 8192, MODE>(c, a);
}

template <bool MIXED>
int rank_mode(md_ctx *c, int mode, PairArgs a) {
  switch (mode) {
  case STAGE_KICK_DRIFT: return rank_tiles<MIXED, STAGE_KICK_DRIFT>(c, a);
  case STAGE_KICK_ONLY: return rank_tiles<MIXED, STAGE_KICK_ONLY>(c, a);
  default: return rank_tiles<MIXED, STAGE_FORCE_ONLY>(c, a);
  }
}

}  // namespace

bool sheet_rank_applies(const md_ctx *c) { return c->model == MD_SHEET1D && c->eps == 0.0; }

int sheet_rank_stage(md_ctx *c, int mode, double kick, double drift, double *fout) {
  PairArgs a{};
  a.kick = kick;
  a.drift = drift;
  a.fout = fout;
  return c->prec == MD_MIXED ? rank_mode<true>(c, mode, a) : rank_mode<false>(c, mode, a);
}
