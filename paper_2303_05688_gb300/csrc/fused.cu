// Constraint-tile search: the batched hot loop of Algorithm 2 with on-chip
// sort-and-accumulate (Sec. 2.2) and the score of Eq. 1.
//
// Work is partitioned by target alpha string A' (the finest constraint class:
// all occupied alpha orbitals fixed).  Items sorted by A' (see excite.cu) make
// each class a contiguous range; a batch of classes is generated into a
// staging buffer as records (beta', v = H_ij c_j, a lower bound of |E0 - H_ii|)
// and then reduced tile by tile on chip:
//   small classes (<= kCap/2 pairs)   packed, several per tile, in item order
//   medium classes (<= kCap pairs)    one tile each, in item order
//   big classes                       split into hash buckets of beta' (each a
//                                     tile); all contributions to one target
//                                     land in the same bucket
// A tile groups its records by target in a shared-memory hash table, drops
// targets in psi, and appends the targets whose |score| can reach the running
// top-N threshold.  A target's values are summed by a rule that does not depend
// on the order of the contributions (long lists after the launch), so that the
// sum equals the sort-and-accumulate result bit for bit, and scored in FP64.
//
// The diagonal H_ii is exact in 64-bit fixed point: the integral terms are
// rounded once to multiples of 2^-s, and integer sums do not depend on their
// order.  Where a score or a decision needs it, it is summed from chunk tables;
// the bound that a record carries is the parent's H_jj plus the excitation's
// change, from the parent's Fock-like diagonals F_s(p) = h_pp + sum_{q in s}
// (J-K)_pq + sum_{q in s'} J_pq, in 32 bits.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "asci_internal.cuh"
#include "fixed192.cuh"
#include "fused.cuh"

namespace asci {

// ----------------------------------------------------------- fixed point ---


namespace {

// out[0] = max |h_pp|, out[1] = max_{p!=q} |J-K|, out[2] = max_{p,q} |J|, and
// out[3] = the largest single-excitation bound over (i, a): |h_ia| + sum_k
// (|(ia|kk) - (ik|ka)| + |(ia|kk)|), as bit patterns (ordered like the values,
// which are not negative).  A warp per pair (p, q); out is zero before.  (One CTA
// whose first thread compared all 256 partial maxima took 45 and 20 us.)
__global__ void __launch_bounds__(256) k_fx_bounds(const double *h1, const double *eri, int n,
                                                   unsigned long long *out) {
  const int lane = threadIdx.x & 31, t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  double m[4] = {0, 0, 0, 0};
  if (t < n * n) {
    const int p = t / n, q = t - p * n;
    const double J = eri[(((size_t)p * n + p) * n + q) * n + q];
    const double K = eri[(((size_t)p * n + q) * n + q) * n + p];
    if (p == q) m[0] = fabs(h1[t]);
    if (p != q) m[1] = fabs(J - K);
    m[2] = fabs(J);
    double b = 0.0;
    if (lane < n) {
      const double ijkk = eri[(((size_t)p * n + q) * n + lane) * n + lane];
      const double ikkj = eri[(((size_t)p * n + lane) * n + lane) * n + q];
      b = fabs(ijkk - ikkj) + fabs(ijkk);
    }
    for (int o = 16; o; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
    m[3] = fabs(h1[t]) + b;
  }
  __shared__ unsigned long long best[4];
  if (threadIdx.x < 4) best[threadIdx.x] = 0;
  __syncthreads();
  if (lane == 0)
    for (int k = 0; k < 4; ++k)
      atomicMax(&best[k], (unsigned long long)__double_as_longlong(m[k]));
  __syncthreads();
  if (threadIdx.x < 4 && best[threadIdx.x]) atomicMax(&out[threadIdx.x], best[threadIdx.x]);
}

__global__ void k_fx_tables(const double *h1, const double *eri, int n, int s, int64_t *hh,
                            int64_t *jk, int64_t *jj) {
  const double sc = ldexp(1.0, s);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * n; t += gridDim.x * blockDim.x) {
    int p = t / n, q = t % n;
    double J = eri[(((size_t)p * n + p) * n + q) * n + q];
    double K = eri[(((size_t)p * n + q) * n + q) * n + p];
    jk[t] = (p == q) ? 0 : __double2ll_rn((J - K) * sc);
    jj[t] = __double2ll_rn(J * sc);
    if (p == q) hh[p] = __double2ll_rn(h1[p * n + p] * sc);
  }
}

__global__ void k_fx_single_tables(const double *h1, const double *eri, int n, int s1,
                                   int64_t *h1x, int64_t *ssx, int64_t *sox) {
  const double sc = ldexp(1.0, s1);
  const size_t n3 = (size_t)n * n * n;
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < n3;
       t += (size_t)gridDim.x * blockDim.x) {
    const int k = (int)(t % n), ia = (int)(t / n), i = ia / n, a = ia % n;
    const double iakk = eri[(((size_t)i * n + a) * n + k) * n + k];
    const double ikka = eri[(((size_t)i * n + k) * n + k) * n + a];
    ssx[t] = __double2ll_rn((iakk - ikka) * sc);
    sox[t] = __double2ll_rn(iakk * sc);
    if (k == 0) h1x[ia] = __double2ll_rn(h1[ia] * sc);
  }
}

// Same-spin terms within the orbitals of m (with h_pp) and between m and r.
__device__ int64_t chunk_within(const int64_t *hh, const int64_t *jk, int n, uint32_t m) {
  int64_t v = 0;
  for (; m; m &= m - 1) {
    const int p = __ffs(m) - 1;
    v += hh[p];
    for (uint32_t r = m & (m - 1); r; r &= r - 1) v += jk[p * n + __ffs(r) - 1];
  }
  return v;
}
__device__ int64_t chunk_between(const int64_t *t, int n, uint32_t m, uint32_t r0) {
  int64_t v = 0;
  for (; m; m &= m - 1)
    for (uint32_t r = r0; r; r &= r - 1) v += t[(__ffs(m) - 1) * n + __ffs(r) - 1];
  return v;
}

// One table per blockIdx.y: the chunk pairs of xs, then the nc x nc tables of xo.
__global__ void k_fx_chunks(const int64_t *hh, const int64_t *jk, const int64_t *jj, int n, int nc,
                            int cb, int64_t *xs, int64_t *xo) {
  const int npair = nc * (nc - 1) / 2;
  const uint32_t mask = (1u << cb) - 1u, full = n >= 32 ? 0xffffffffu : ((1u << n) - 1u);
  const int t = (int)blockIdx.y;
  int k = 0, l = 1;
  if (t < npair) {
    for (int i = 0; i < t; ++i)
      if (++l == nc) l = ++k + 1;
  } else {
    k = (t - npair) / nc;
    l = (t - npair) % nc;
  }
  int64_t *out = t < npair ? xs + ((size_t)t << (2 * cb)) : xo + ((size_t)(t - npair) << (2 * cb));
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < 1u << (2 * cb);
       i += gridDim.x * blockDim.x) {
    // bits at or above n (in the last chunk) belong to no orbital
    const uint32_t x = ((i >> cb) << (k * cb)) & full;
    const uint32_t y = (uint32_t)((uint64_t)(i & mask) << (l * cb)) & full;
    int64_t v;
    if (t >= npair) {
      v = chunk_between(jj, n, x, y);
    } else {
      v = chunk_between(jk, n, x, y);
      if (k == 0) v += chunk_within(hh, jk, n, y);
      if (k == 0 && l == 1) v += chunk_within(hh, jk, n, x);
    }
    out[i] = v;
  }
}

}  // namespace

// x * 2^-s rounded to the nearest double (ties to even), by integer
// operations only; x * 2^-s must lie in the normal range.
__device__ __forceinline__ double fx64_to_double(int64_t x, int s) {
  if (x == 0) return 0.0;
  const uint64_t sign = x < 0 ? (1ull << 63) : 0ull;
  const uint64_t u = x < 0 ? 0ull - (uint64_t)x : (uint64_t)x;
  int P = 63 - __clzll((long long)u);  // leading bit
  uint64_t mant;
  if (P <= 52) {
    mant = u << (52 - P);
  } else {
    const int sh = P - 52;
    mant = u >> sh;
    const uint64_t rem = u & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (mant & 1ull))) {
      ++mant;
      if (mant == (1ull << 53)) {
        mant >>= 1;
        ++P;
      }
    }
  }
  return __longlong_as_double(
      (long long)(sign | ((uint64_t)(P - s + 1023) << 52) | (mant & ((1ull << 52) - 1ull))));
}

__device__ __forceinline__ int64_t fx_diag(const FxInts &X, uint32_t A, uint32_t B) {
  const int n = X.n;
  int64_t s = X.ecore_x;
  for (uint32_t m = A; m; m &= m - 1) {
    const int p = __ffs(m) - 1;
    s += X.hh[p];
    for (uint32_t r = m & (m - 1); r; r &= r - 1) s += X.jk[p * n + __ffs(r) - 1];
    for (uint32_t r = B; r; r &= r - 1) s += X.jj[p * n + __ffs(r) - 1];
  }
  for (uint32_t m = B; m; m &= m - 1) {
    const int p = __ffs(m) - 1;
    s += X.hh[p];
    for (uint32_t r = m & (m - 1); r; r &= r - 1) s += X.jk[p * n + __ffs(r) - 1];
  }
  return s;
}

namespace {

// The staged denominator E0 - H_ii serves screens only, so it is summed in
// 32-bit fixed point: multiples of 2^ds units of the 64-bit grid (|E0 - H_ii| <
// 2^30 of those: build_fx), each term rounded to nearest; a sum of at most 15 such
// terms is within 8 units of the exact value, and what is stored is a lower bound
// of the magnitude.  A test that these 8 units could decide forms the exact value.
// Half the registers, shuffles, table bytes and additions of 64 bits.  (Unsigned:
// sums may wrap on the way.)
constexpr int32_t kDenSlack = 8;
__device__ __forceinline__ uint32_t den_round(int64_t x, int ds) {
  return (uint32_t)((x + (1ll << (ds - 1))) >> ds);
}

// A core determinant as the emission reads it: one 16-byte load.
struct __align__(16) CoreRec {
  uint32_t beta;
  uint32_t den;  // E0 - H_jj
  double c;
};

// Parent data of each core det (alpha-sorted order): H_jj and both Fock-like
// diagonals.  Fb is determinant-major (Fb[j n + p]: a warp's lanes read one
// determinant's row); Fa is orbital-major (Fa[p m + j]: the lanes of an
// alpha-double step read one orbital of consecutive determinants).
// A thread per (orbital, determinant), determinants fastest; the thread of
// orbital n forms H_jj and the determinant's record.
__global__ void k_core_fock(FxInts X, int64_t E0_x, const uint32_t *core_alpha,
                            const uint32_t *core_beta, const double *core_c, size_t m,
                            CoreRec *rec, uint32_t *Fa, uint32_t *Fb) {
  const int n = X.n, p = (int)blockIdx.y;
  for (size_t j = (size_t)blockIdx.x * blockDim.x + threadIdx.x; j < m;
       j += (size_t)gridDim.x * blockDim.x) {
    const uint32_t A = core_alpha[j], B = core_beta[j];
    if (p == n) {
      CoreRec r;
      r.beta = B;
      r.den = den_round(E0_x - fx_diag(X, A, B), X.ds);
      r.c = core_c[j];
      rec[j] = r;
      continue;
    }
    int64_t fa = X.hh[p], fb = X.hh[p];
    for (uint32_t r = A; r; r &= r - 1) {
      const int q = __ffs(r) - 1;
      fa += X.jk[p * n + q];
      fb += X.jj[p * n + q];
    }
    for (uint32_t r = B; r; r &= r - 1) {
      const int q = __ffs(r) - 1;
      fb += X.jk[p * n + q];
      fa += X.jj[p * n + q];
    }
    Fa[(size_t)p * m + j] = den_round(fa, X.ds);
    Fb[j * n + p] = den_round(fb, X.ds);
  }
}

__global__ void k_den_tables(FxInts X, uint32_t *jk, uint32_t *jj) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < X.n * X.n; t += gridDim.x * blockDim.x) {
    jk[t] = den_round(X.jk[t], X.ds);
    jj[t] = den_round(X.jj[t], X.ds);
  }
}


// ------------------------------------------------------ groups of items ---

// gid holds the exclusive scan of the head flags; it becomes each item's group
// (heads up to and including it, less one), and each head fills its group's
// row.  Row G (one past the last group) gets the totals: T items, P pairs.
__global__ void k_group_tab(const uint64_t *items, uint32_t *gid, const uint64_t *Wexcl, uint64_t T,
                            uint32_t *g_alpha, uint64_t *g_P0, uint64_t *g_item0) {
  for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < T;
       t += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t hi = (uint32_t)(items[t] >> 32);
    const bool head = t == 0 || hi != (uint32_t)(items[t - 1] >> 32);
    const uint32_t g = gid[t] + (head ? 1u : 0u) - 1u;
    gid[t] = g;
    if (head) {
      g_alpha[g] = hi;
      g_P0[g] = Wexcl[t];
      g_item0[g] = t;
    }
    if (t == T - 1) {
      g_alpha[g + 1] = 0;
      g_P0[g + 1] = Wexcl[T];
      g_item0[g + 1] = T;
    }
  }
}

// ------------------------------------------------------- tile planning ---

enum : uint32_t { kTilePacked = 0, kTileMedium = 1, kTileBucket = 2 };

// bits of the device error word of the constraint-tile kernels
constexpr unsigned kErrProbe = 1u;      // exclusion probe ran past the table
constexpr unsigned kErrTile = 2u;       // a tile descriptor outside its limits
constexpr unsigned kErrStage = 4u;      // a record position outside the staging buffer
constexpr unsigned kErrCore = 8u;       // a core index outside the core
constexpr unsigned kErrAccum = 16u;     // a value outside the exact accumulator's range

struct TileDesc {  // 32 bytes; npairs at byte offset 4 (read by the host)
  uint32_t start;   // first record in the batch staging buffer
  uint32_t npairs;  // records in the tile
  uint32_t g0;      // first group (global id)
  uint32_t ng;      // groups (packed tiles)
  uint32_t kind;
  uint32_t alpha;   // target alpha string (medium / bucket tiles)
  uint32_t psi_lo;  // psi determinants that fall in the tile: [psi_lo, psi_hi) of
  uint32_t psi_hi;  // the batch's tile-ordered psi list
};

static_assert(sizeof(TileDesc) == 32, "tile descriptor layout");

// A screened-out record (Alg. 2's eps test) keeps its slot with a NaN value.
// (Tested on the bits: NaN compares cost FP64 instructions, which are scarce.)
__device__ __forceinline__ bool is_dropped(double v) {
  return ((uint64_t)__double_as_longlong(v) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}
__device__ __forceinline__ double drop_marker() {
  return __longlong_as_double(0x7ff8000000000000ll);
}
// Sum of four values that depends only on their multiset: they are ordered by
// magnitude (then sign) with a sorting network on the bits and added from the
// smallest.  Pad with +0.0 for fewer values.
__device__ __forceinline__ uint64_t mag_order(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  return (b << 1) | (b >> 63);
}
__device__ __forceinline__ void order2(double &x, double &y) {
  if (mag_order(y) < mag_order(x)) {
    const double t = x;
    x = y;
    y = t;
  }
}
__device__ __forceinline__ double sum4_ordered(double a, double b, double c, double d) {
  order2(a, b);
  order2(c, d);
  order2(a, c);
  order2(b, d);
  order2(b, c);
  return ((a + b) + c) + d;
}

// x with its sign flipped when flip is 1 (an integer operation on the bits).
__device__ __forceinline__ double flip_sign(double x, uint32_t flip) {
  return __longlong_as_double(__double_as_longlong(x) ^ ((long long)(flip & 1u) << 63));
}

}  // namespace

constexpr int kCellThreads = 128;
constexpr int kCellCtas = 8;                        // per SM
constexpr int kCap = 1024;                          // records per tile
constexpr uint32_t kSmallMax = kCap / 2;            // packable class size
constexpr uint32_t kBucketTarget = kCap * 13 / 16;  // expected records per hash bucket

namespace {

// Tile kind of each class and its staging slots: its pairs in place, or kCap
// slots for each hash bucket of a big class.
__global__ void k_group_class(const uint64_t *g_P0, uint32_t gb0, uint32_t gb1, uint64_t Pend,
                              uint32_t *kind, uint32_t *nb, uint64_t *small_pairs,
                              uint64_t *slots) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < gb1 - gb0;
       i += gridDim.x * blockDim.x) {
    const uint32_t g = gb0 + i;
    const uint64_t P = ((g + 1 < gb1) ? g_P0[g + 1] : Pend) - g_P0[g];
    uint32_t k = P <= kSmallMax ? kTilePacked : (P <= kCap ? kTileMedium : kTileBucket);
    kind[i] = k;
    nb[i] = k == kTileBucket ? (uint32_t)((P + kBucketTarget - 1) / kBucketTarget) : 0u;
    small_pairs[i] = k == kTilePacked ? P : 0;
    slots[i] = k == kTileBucket ? (uint64_t)nb[i] * kCap : P;
  }
}

__device__ __forceinline__ bool packed_start(uint32_t i, const uint32_t *kind,
                                             const uint64_t *Ws) {
  if (kind[i] != kTilePacked) return false;
  if (i == 0 || kind[i - 1] != kTilePacked) return true;
  return (Ws[i] / kSmallMax) != (Ws[i - 1] / kSmallMax);
}

__global__ void k_tile_count(uint32_t ng, const uint32_t *kind, const uint32_t *nb,
                             const uint64_t *Ws, uint32_t *ntile) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ng; i += gridDim.x * blockDim.x)
    ntile[i] = kind[i] == kTilePacked ? (packed_start(i, kind, Ws) ? 1u : 0u)
                                      : (kind[i] == kTileMedium ? 1u : nb[i]);
}

__global__ void k_tile_write(uint32_t gb0, uint32_t ng, const uint64_t *soff, uint64_t Pend,
                             const uint64_t *g_P0, const uint32_t *g_alpha,
                             const uint32_t *kind, const uint32_t *nb, const uint64_t *Ws,
                             const uint32_t *tile_base, TileDesc *tiles) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < ng; i += gridDim.x * blockDim.x) {
    const uint32_t g = gb0 + i;
    const uint64_t P = ((i + 1 < ng) ? g_P0[g + 1] : Pend) - g_P0[g];
    const uint32_t start = (uint32_t)soff[i];
    const uint32_t k = kind[i];
    if (k == kTilePacked) {
      const bool st = packed_start(i, kind, Ws);
      const uint32_t t = st ? tile_base[i] : tile_base[i] - 1;
      if (st) {
        tiles[t].start = start;
        tiles[t].g0 = g;
        tiles[t].kind = kTilePacked;
        tiles[t].alpha = g_alpha[g];
      }
      atomicAdd(&tiles[t].npairs, (uint32_t)P);
      atomicAdd(&tiles[t].ng, 1u);
    } else if (k == kTileMedium) {
      TileDesc d;
      d.start = start;
      d.npairs = (uint32_t)P;
      d.g0 = g;
      d.ng = 1;
      d.kind = kTileMedium;
      d.alpha = g_alpha[g];
      d.psi_lo = d.psi_hi = 0;
      tiles[tile_base[i]] = d;
    }
  }
}

// Bucket tiles of big classes, one thread per cell: the class holding cell c
// is the last one whose first cell is at or before c.  Bucket b of a class
// owns kCap staging slots; its record count is known after emission.
__global__ void k_cell_write(uint32_t gb0, uint32_t ng, uint32_t ncells, const uint64_t *soff,
                             const uint32_t *g_alpha, const uint32_t *tile_base,
                             const uint32_t *cellbase, TileDesc *tiles, uint32_t *cell_tile) {
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells;
       c += gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = ng - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (cellbase[mid] <= c) lo = mid; else hi = mid - 1;
    }
    const uint32_t g = gb0 + lo, b = c - cellbase[lo];
    TileDesc d;
    d.start = (uint32_t)(soff[lo] + (uint64_t)b * kCap);
    d.npairs = 0;
    d.g0 = g;
    d.ng = 1;
    d.kind = kTileBucket;
    d.alpha = g_alpha[g];
    d.psi_lo = d.psi_hi = 0;
    tiles[tile_base[lo] + b] = d;
    cell_tile[c] = tile_base[lo] + b;
  }
}

// Sort keys of the spilled records: tile << 32 | spill index.
__global__ void k_spill_keys(const uint32_t *spill_cell, const uint32_t *cell_tile, uint32_t n,
                             uint64_t *keys) {
  for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    keys[j] = ((uint64_t)cell_tile[spill_cell[j]] << 32) | j;
}

// Record counts of the bucket tiles after emission; a bucket that received
// more than kCap records (its surplus is in the spill list) is reduced by the
// global path.
__global__ void k_cell_finish(uint32_t ncells, const uint32_t *fill, const uint32_t *cell_tile,
                              TileDesc *tiles, unsigned *n_over, uint32_t *over_list,
                              uint32_t over_cap) {
  for (uint32_t c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells;
       c += gridDim.x * blockDim.x) {
    const uint32_t f = fill[c], t = cell_tile[c];
    tiles[t].npairs = f;
    if (f > (uint32_t)kCap) {
      const unsigned slot = atomicAdd(n_over, 1u);
      if (slot < over_cap) over_list[slot] = t;
    }
  }
}

// ------------------------------------------------------------ emission ---

__device__ __forceinline__ uint32_t bucket_of(uint32_t beta, uint32_t nb) {
  return (uint32_t)(((uint64_t)(beta * 0x9E3779B1u) * nb) >> 32);
}

// ----------------------------------------------------------- emission ---
// The pairs of a batch are emitted in two kinds of work units.
//  * Determinant runs: an item (core alpha group k, alpha operation o) whose
//    o is the identity or an alpha single, applied to one core determinant of
//    the group.  For o = 0 the run holds the determinant's beta singles and
//    beta doubles (sb + dbb pairs); for an alpha single, that single alone
//    and combined with each beta single (1 + sb pairs).  One warp walks a
//    run: lane L holds the L-th occupied and the L-th virtual beta orbital of
//    the determinant and the diagonal terms that depend on them, and each
//    pair fetches its orbitals and terms with shuffles.
//  * Alpha doubles: one pair per core determinant of the group.  These items
//    are laid out flat and each lane takes one pair; the operation, its
//    matrix element and the determinant-independent part of the diagonal
//    change are computed once per item.
// A pair keeps the position p = Wexcl[t] + m * npd + e of the item order
// (t: item, m: determinant in the group, e: pair in the run), so classes that
// fit a tile are staged in place and big classes go through bucket counters.

constexpr int kRunThreads = 256;
constexpr int kRunClaim = 4;   // runs a warp claims at a time, at most
// A determinant's o = 0 run (its beta singles and doubles, 10,314 pairs at
// (24e,30o)) is emitted in pieces, so that the last runs of a launch are short
// and its warps finish together: at most kPiecePairs pairs, fewer when the batch
// would give each of the kEmitWarps warps that the GPU holds less than four.
// (The small first batch of a search is nearly all o = 0 runs: 3.9 M pairs of
// (16e,16o) in 261 us with pieces of 1024 pairs claimed four at a time, which left
// half of the warps without work, and with the atomics waited for at once; 115 now.)
constexpr uint32_t kPiecePairs = 1024, kMinPiece = 128;
constexpr uint32_t kEmitWarps = 152 * 32;
constexpr int kPairTab = 496;  // C(32, 2): unranked index pairs
constexpr int kAdThreads = 256;
constexpr int kAdTile = 512;   // alpha-double pairs per CTA step

struct EmitArgs {
  DevInts I;
  FxInts X;
  ExcCounts E;
  FastDiv dv_vb, dv_pb_p, dv_pieces;
  uint32_t npd0, npd1;        // pairs per determinant for o = 0 and for an alpha single
  uint32_t piece, run_claim;  // pairs of a piece; runs a warp claims at a time
  uint32_t npieces;           // pieces of `piece` pairs a determinant's o = 0 run is cut into
  const uint64_t *items, *Wexcl;
  const uint32_t *item_group;
  uint64_t t0;
  int opbits;
  const uint32_t *grp_alpha, *grp_start, *grp_count;
  // the core's records, its Fock-like diagonals and jk, jj in units of the
  // 32-bit denominator
  const CoreRec *core;
  const uint32_t *Fa, *Fb, *jk, *jj;
  uint32_t gb0;
  const uint32_t *kind, *nb, *cellbase;
  const uint64_t *soff;       // first staging slot of each class of the batch
  const uint64_t *g_P0;       // first pair of each class
  uint32_t *fill;             // records placed in each bucket cell
  StageRec *spill_rec;        // records beyond a cell's kCap slots
  uint32_t *spill_cell;
  unsigned *n_spill;
  uint32_t spill_cap;
  const uint64_t *runs;       // (item - t0) << 32 | determinant in the group
  uint64_t nruns;
  unsigned long long *run_next;  // next unclaimed run (zeroed before each launch)
  const uint32_t *adl;        // alpha-double items (item - t0)
  const uint32_t *ad_off;     // first flat pair of each (exclusive prefix)
  uint32_t nad, ad_total;
  const uint32_t *ad_tile_item;  // first alpha-double item of each CTA step
  uint32_t ad_tiles;
  Stage st;
  uint32_t st_cap;            // st.cap (below 2^32)
  double eps;                 // Alg. 2 screen; 0 keeps every pair
  float eps_f;                // eps 2^eps_shift as a float (the screen's float pre-test)
  int eps_shift;
  int64_t E0_x;
  double inv_scale;
  float scale32;              // a unit of the 32-bit denominator
  unsigned long long *survivors;
  uint32_t ncore;
  unsigned *err;
};

// An excitation from the two strings: its holes and particles are the bits in
// which they differ.  Parities: with n(x) the occupied orbitals of s below x, a
// single i -> a crosses n(a) + n(i) + [a > i] (mod 2) of them, and a double i <
// j -> a < b, taken as i -> a then j -> b, n(a) + n(b) + n(i) + n(j) + 1 plus the
// particles between i and j.
__device__ __forceinline__ uint32_t below(int x) { return (1u << x) - 1u; }

__device__ __forceinline__ uint32_t single_orbitals(uint32_t s, uint32_t t, int *i, int *a) {
  *i = __ffs(s & ~t) - 1;
  *a = __ffs(t & ~s) - 1;
  return (uint32_t)__popc(s & (below(*i) ^ below(*a))) + (*a > *i ? 1u : 0u);
}

// Parity (bit 0) of the double from the holes i < j and the particle mask pm.
__device__ __forceinline__ uint32_t double_sign(uint32_t s, int i, int j, int a, int b) {
  const uint32_t m = below(i) ^ below(j) ^ below(a) ^ below(b);
  const uint32_t between = below(j) & ~((2u << i) - 1u);
  return (uint32_t)__popc(s & m) + (uint32_t)__popc(((1u << a) | (1u << b)) & between) + 1u;
}

// Single excitation i -> a of the string s (the other spin's string o) in
// fixed point (multiples of 2^-s1): h_ia plus, over the occupied orbitals k,
// (ia|kk) - (ik|ka) for k of the same spin and (ia|kk) for k of the other.
__device__ __forceinline__ int64_t fx_single(const FxInts &X, uint32_t s, uint32_t o, int i,
                                             int a) {
  const int n = X.n;
  const int64_t *ss = X.ssx + ((size_t)i * n + a) * n;
  const int64_t *so = X.sox + ((size_t)i * n + a) * n;
  int64_t v = X.h1x[i * n + a];
  for (uint32_t m = s; m; m &= m - 1) v += ss[__ffs(m) - 1];
  for (uint32_t m = o; m; m &= m - 1) v += so[__ffs(m) - 1];
  return v;
}

// A float widened to a double exactly, by operations on the bits (a widening
// conversion would take the FP64 pipe, which is scarce).
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  const uint32_t e = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  const uint64_t sign = (uint64_t)(u >> 31) << 63;
  if (e == 0xffu)  // inf or nan
    return __longlong_as_double((long long)(sign | 0x7ff0000000000000ull | ((uint64_t)m << 29)));
  if (e == 0) {    // zero or subnormal: normalise the mantissa
    if (!m) return __longlong_as_double((long long)sign);
    const int lz = __clz(m) - 8;  // leading zeros within the 23-bit field, plus one
    const uint64_t mm = ((uint64_t)m << lz) & 0x7fffffu;
    return __longlong_as_double(
        (long long)(sign | ((uint64_t)(1023 - 126 - lz) << 52) | (mm << 29)));
  }
  return __longlong_as_double(
      (long long)(sign | ((uint64_t)(e + 1023 - 127) << 52) | ((uint64_t)m << 29)));
}

// Precision of the pair values (the a8 variant): 0 = FP64 integrals and
// product; 1 = two-electron elements gathered from FP32 tables, FP64 product;
// 2 = FP32 tables and an FP32 product H_ij c_j.  Sums and diagonals are the
// same in all three.
template <int PREC>
__device__ __forceinline__ double pair_value(double h, double c, float cf) {
  if (PREC == 2) return widen((float)h * cf);
  return h * c;
}

// |x| as a float built from the bits, truncated (relative error below 2^-23);
// *ok is false when |x| lies outside the normal float range.
__device__ __forceinline__ float abs_as_float(double x, bool *ok) {
  const uint64_t b = (uint64_t)__double_as_longlong(x) & 0x7fffffffffffffffull;
  int e = (int)(b >> 52) - 1023 + 127;
  *ok = e >= 1 && e <= 254;
  e = e < 1 ? 1 : (e > 254 ? 254 : e);
  return __uint_as_float(((uint32_t)e << 23) | (uint32_t)((b >> 29) & 0x7fffffu));
}

template <bool EPS>
__device__ __forceinline__ void write_record(const EmitArgs &A, uint32_t pos, bool spill,
                                             uint32_t cell, uint32_t talpha, uint32_t tb,
                                             bool packed, double v, uint32_t den, bool *kept) {
  const int32_t mag = abs((int32_t)den);  // |den| < 2^30
  const float df = (float)max(mag - kDenSlack, 0) * A.scale32;
  if (EPS) {
    // Alg. 2's screen |v / (E0 - H_ii)| > eps, without a division.  A float
    // test settles every pair whose |v| is not within 4e-6 relative of eps
    // times the bounds of |E0 - H_ii| (|v| truncated to a float lies within
    // 2^-23 below its value, eps_f and the bounds within 2^-24 of theirs, the
    // product within 2^-24); the rest take the FP64 test on the exact
    // denominator, so every decision is that test's.  (FP64 instructions are
    // scarce on this GPU.)  Both sides are scaled by the power of two that
    // brings eps to eps_f in [0.5, 1]: eps_f times a bound is then in
    // [2^-32, 2^51] or zero, and a scaled |v| beyond the float range on either
    // side is replaced by a float that is beyond that interval too.  A pair of
    // value zero is never kept; with symmetry most pairs are such: summing their
    // exact denominators made a (24e,30o) search with seven eighths of the
    // integrals zero, C = 1e4, take 127 ms, against 18.3 (19.7 without a screen).
    const uint64_t b = (uint64_t)__double_as_longlong(v) & 0x7fffffffffffffffull;
    const int be = (int)(b >> 52), e = min(max(be - 896 + A.eps_shift, 1), 254);
    const float vf = __uint_as_float(((uint32_t)e << 23) | (uint32_t)((b >> 29) & 0x7fffffu));
    const bool normal = be > 0 && be < 0x7ff;  // neither zero, subnormal, infinite nor NaN
    const float lo = A.eps_f * df, hi = A.eps_f * ((float)(mag + kDenSlack) * A.scale32);
    bool keep;
    if (normal && vf > hi * 1.000004f) {
      keep = true;
    } else if ((normal && vf < lo * 0.999996f) || b == 0) {
      keep = false;
    } else {
      const double d = __ll2double_rn(A.E0_x - fx_diag(A.X, talpha, tb)) * A.inv_scale;
      keep = fabs(v) > A.eps * fabs(d);
    }
    if (!keep) v = drop_marker();
    *kept = keep;
  }
  const uint64_t vb = (uint64_t)__double_as_longlong(v);
  const uint4 r = make_uint4((uint32_t)vb, (uint32_t)(vb >> 32), tb, __float_as_uint(df));
  if (spill) {
    if (pos < A.spill_cap) {  // beyond: counted only, the host reports it
      reinterpret_cast<uint4 *>(A.spill_rec)[pos] = r;
      A.spill_cell[pos] = cell;
    }
  } else if (pos < A.st_cap) {
    reinterpret_cast<uint4 *>(A.st.rec)[pos] = r;
    if (packed) A.st.alpha[pos] = talpha;
  } else {
    atomicOr(A.err, kErrStage);
  }
}

// Next free slot of the lane's bucket cell (lanes with `big`), in two steps so
// that the atomic's latency can pass while other pairs are worked on: claim_slot
// issues the atomic, claimed_slot gives the slot number within the cell.  Lanes of
// one cell share an atomic when the class has few buckets (peers: the lanes of
// this lane's cell); with many, two lanes seldom meet and each takes its own.
__device__ __forceinline__ uint32_t claim_slot(uint32_t *fill, uint32_t cell, bool big, bool few,
                                               uint32_t *peers) {
  if (!few) return big ? atomicAdd(&fill[cell], 1u) : 0u;
  *peers = __match_any_sync(0xffffffffu, big ? cell : 0xffffffffu);
  if (!big || (int)(threadIdx.x & 31) != __ffs(*peers) - 1) return 0u;
  return atomicAdd(&fill[cell], (uint32_t)__popc(*peers));
}
__device__ __forceinline__ uint32_t claimed_slot(uint32_t raw, bool few, uint32_t peers) {
  if (!few) return raw;
  return __shfl_sync(0xffffffffu, raw, __ffs(peers) - 1) +
         __popc(peers & ((1u << (threadIdx.x & 31)) - 1u));
}

// The pairs an emission thread kept under the eps screen, added to the
// search's counter once per warp when the kernel ends (one counter for the
// whole grid: an atomic per chunk would serialise on it).
__device__ __forceinline__ void add_survivors(const EmitArgs &A, unsigned long long kept) {
  for (int d = 16; d; d >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, d);
  if ((threadIdx.x & 31) == 0 && kept) atomicAdd(A.survivors, kept);
}

// What a warp needs of one run, set up by one lane for each run of a claim (so
// that the chain of loads, run -> item -> group -> determinant, is walked once
// for all of them) and read back by the warp in a few wide loads.
struct __align__(16) RunInfo {
  uint32_t B, talpha, Ak, off0;       // off0: in-place slot of the run's first pair
  uint32_t cls0, cell0, nbk, jdx;     // bucket b's slots start at cls0 + b kCap
  uint32_t ebeg, eend, orb, flags;    // orb: i | a << 8 of the alpha single
  double c;
  uint32_t base, pad;                 // E0 - H_jj, less the alpha single's change
};
enum : uint32_t { kRunZero = 1u, kRunBig = 2u, kRunPacked = 4u, kRunFew = 8u, kRunOdd = 16u };
constexpr uint32_t kFewBuckets = 32;

// EPS compiles Alg. 2's screen in (eps > 0); PREC selects the pair-value
// precision (pair_value).
//
// Bound: instruction issue and the latency of the bucket atomics.  Seven pairs
// in ten combine an alpha single with a beta single; such a pair takes its
// ranks from a table, its orbitals and their diagonal terms from the
// determinant's lists in shared memory (one 8-byte load each), and its sign
// from the ranks: the occupied orbitals below the h-th occupied one are h, those
// below the p-th virtual orbital x are x - p.  Two chunks are in flight, in turn
// (a copy of one into the other costs 20 moves per pair), and a determinant's
// beta string, coefficient and denominator arrive in one load: with the 32-bit
// screen of write_record 3482 -> 3319 us for a (13e,19o) search with eps (64-bit
// denominators spilled registers there), 181.9 -> 178.6 ms at (24e,30o).
template <bool EPS, int PREC>
__global__ void __launch_bounds__(kRunThreads, 4) k_emit_runs(EmitArgs A) {
  using D = uint32_t;
  struct __align__(8) Orb {
    D z;          // diagonal term of removing or adding the orbital
    int32_t x;    // the orbital
  };
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint16_t s_pair[kPairTab];
  __shared__ uint16_t s_sp[256];  // beta single f: hole rank | particle rank << 8
  __shared__ RunInfo s_run[kRunThreads / 32][kRunClaim];
  __shared__ Orb s_occ[kRunThreads / 32][32], s_vir[kRunThreads / 32][32];
  const int n = A.I.n;
  // jk with the hole as the row (the lanes' particles are then on distinct banks)
  D *s_jk = reinterpret_cast<D *>(smem_raw), *s_jj = s_jk + n * n;
  for (int t = threadIdx.x; t < n * n; t += kRunThreads) {
    s_jk[(t % n) * n + t / n] = A.jk[t];
    s_jj[t] = A.jj[t];
  }
  for (int r = threadIdx.x; r < kPairTab; r += kRunThreads) {
    int x, y;
    unrank_pair((uint32_t)r, &x, &y);
    s_pair[r] = (uint16_t)(x | (y << 8));
  }
  const uint32_t sb = A.E.sb, vb = A.E.vb;
  for (uint32_t f = threadIdx.x; f < sb; f += kRunThreads) {
    const uint32_t h = A.dv_vb.div(f);
    s_sp[f] = (uint16_t)(h | ((f - h * vb) << 8));
  }
  __syncthreads();
  const uint32_t omask = (1u << A.opbits) - 1u;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Orb *occ = s_occ[warp], *vir = s_vir[warp];
  unsigned long long my_kept = 0;  // pairs kept by the eps screen (EPS)
  // runs are claimed kRunClaim at a time from a shared counter (their lengths
  // differ by a factor of about five); the next claim is issued before the
  // claimed runs are emitted
  unsigned long long claim = 0;
  if (lane == 0) claim = atomicAdd(A.run_next, (unsigned long long)A.run_claim);
  uint64_t r0 = (uint64_t)__shfl_sync(0xffffffffu, claim, 0);
#pragma unroll 1
  for (; r0 < A.nruns; r0 = (uint64_t)__shfl_sync(0xffffffffu, claim, 0)) {
    if (lane == 0) claim = atomicAdd(A.run_next, (unsigned long long)A.run_claim);
    const int nr = (int)(A.nruns - r0 < (uint64_t)A.run_claim ? A.nruns - r0 : (uint64_t)A.run_claim);
    __syncwarp();  // the previous claim's runs have been read
    if (lane < nr) {
      const uint64_t run = A.runs[r0 + lane];
      const uint64_t t = A.t0 + (run >> 32);
      const uint64_t it = A.items[t];
      const uint32_t k = (uint32_t)it >> A.opbits, o = (uint32_t)it & omask;
      // determinant m of the group; for o = 0, piece number mr % npieces of its run
      const uint32_t mr = (uint32_t)run;
      const uint32_t m = o == 0 ? A.dv_pieces.div(mr) : mr;
      const uint32_t gi = A.item_group[t] - A.gb0, kd = A.kind[gi];
      const uint32_t npd = o == 0 ? A.npd0 : A.npd1;
      RunInfo R;
      R.jdx = A.grp_start[k] + m;
      R.flags = (o == 0 ? kRunZero : 0u) | (kd == kTileBucket ? kRunBig : 0u) |
                (kd == kTilePacked ? kRunPacked : 0u);
      R.ebeg = o == 0 ? (mr - m * A.npieces) * A.piece : 0u;
      R.eend = o == 0 && R.ebeg + A.piece < npd ? R.ebeg + A.piece : npd;
      R.cls0 = (uint32_t)A.soff[gi];
      R.off0 = (uint32_t)(A.soff[gi] + (A.Wexcl[t] + (uint64_t)m * npd - A.g_P0[A.gb0 + gi]));
      R.cell0 = kd == kTileBucket ? A.cellbase[gi] : 0u;
      R.nbk = kd == kTileBucket ? A.nb[gi] : 1u;
      if (R.nbk < kFewBuckets) R.flags |= kRunFew;
      R.talpha = (uint32_t)(it >> 32);
      R.Ak = A.grp_alpha[k];
      R.orb = 0;
      if (R.jdx >= A.ncore) {
        atomicOr(A.err, kErrCore);
        R.eend = R.ebeg;
        R.jdx = 0;
      }
      const CoreRec cr = A.core[R.jdx];
      R.B = cr.beta;
      R.c = cr.c;
      R.base = cr.den;
      R.pad = 0;
      if (o != 0) {
        int i, a;
        const uint32_t odd = single_orbitals(R.Ak, R.talpha, &i, &a);
        R.orb = (uint32_t)i | ((uint32_t)a << 8);
        if (odd & 1u) R.flags |= kRunOdd;
        R.base -= A.Fa[(size_t)a * A.ncore + R.jdx] - A.Fa[(size_t)i * A.ncore + R.jdx] -
                  s_jk[i * n + a];
      }
      s_run[warp][lane] = R;
    }
#pragma unroll 1
    for (int r = 0; r < nr; ++r) {
      __syncwarp();  // the runs are set up; the previous run's lists have been read
      const RunInfo &R = s_run[warp][r];
      const uint32_t B = R.B, talpha = R.talpha, flags = R.flags, ebeg = R.ebeg, eend = R.eend;
      const uint32_t cls0 = R.cls0, off0 = R.off0, cell0 = R.cell0, nbk = R.nbk;
      const bool zero = (flags & kRunZero) != 0u, big = (flags & kRunBig) != 0u;
      const bool packed = (flags & kRunPacked) != 0u, few = (flags & kRunFew) != 0u;
      const uint32_t pa = (flags & kRunOdd) ? 1u : 0u;
      const double c = R.c;
      const float cf = (float)c;
      const D Bz = R.base;
      const int ia = (int)(R.orb & 0xffu), aa = (int)(R.orb >> 8);
      // the determinant's occupied and virtual beta orbitals by rank, with the
      // Fock-like diagonal (and, for an alpha single, its Coulomb change)
      if (lane < n) {
        Orb q;
        q.x = lane;
        q.z = A.Fb[(size_t)R.jdx * n + lane];
        if (!zero) q.z += s_jj[aa * n + lane] - s_jj[ia * n + lane];
        const uint32_t nb = (uint32_t)__popc(B & below(lane));
        if ((B >> lane) & 1u) occ[nb] = q;
        else vir[lane - nb] = q;
      }
      double h0 = 0.0;  // the alpha single alone
      const double *erow = A.I.eri;
      const float *erow32 = A.I.eri32;
      if (!zero) {
        // its matrix element, summed across the warp: lane p adds the terms of
        // orbital p where alpha and beta occupy it
        const size_t row = ((size_t)ia * n + aa) * n;
        int64_t part = 0;
        if (lane < n) {
          if ((R.Ak >> lane) & 1u) part = A.X.ssx[row + lane];
          if ((B >> lane) & 1u) part += A.X.sox[row + lane];
        }
#pragma unroll
        for (int d = 16; d; d >>= 1) part += (int64_t)__shfl_xor_sync(0xffffffffu, (long long)part, d);
        h0 = flip_sign(fx64_to_double(part + A.X.h1x[ia * n + aa], A.X.s1), pa);
        erow = A.I.eri + ((size_t)ia * n + aa) * n * n;
        if (PREC != 0) erow32 = A.I.eri32 + ((size_t)ia * n + aa) * n * n;
      }
      __syncwarp();
      // one chunk of 32 pairs: target, place, denominator and matrix element
      struct Chunk {
        uint32_t tb, pos, sign, peers;
        D den;
        bool valid;
        double g;   // the gathered integral, requested a chunk ahead
        float gf;   // the same from the FP32 tables
      };
      auto place = [&](Chunk &q, uint32_t e) {
        // big: the next free slot of the lane's bucket cell (warp-uniform)
        q.pos = big ? claim_slot(A.fill, cell0 + bucket_of(q.tb, nbk), q.valid, few, &q.peers)
                    : off0 + e;
      };
      auto emit = [&](const Chunk &q, double h, bool is_double) {
        // is_double: h holds the value; else the gathered integral is it
        double v;
        if (PREC == 2) {
          const float hf = is_double ? (float)h : __uint_as_float(__float_as_uint(q.gf) ^ (q.sign << 31));
          v = widen(hf * cf);
        } else {
          const double hh = is_double ? h : flip_sign(PREC == 1 ? widen(q.gf) : q.g, q.sign);
          v = hh * c;
        }
        uint32_t pos = q.pos, cell = cell0;
        bool spill = false, kept = false;
        if (big) {  // warp-uniform
          const uint32_t slot = claimed_slot(q.pos, few, q.peers), bkt = bucket_of(q.tb, nbk);
          cell += bkt;
          pos = cls0 + bkt * (uint32_t)kCap + slot;
          if (q.valid && slot >= (uint32_t)kCap) {  // the cell is full: the spill list
            spill = true;
            pos = atomicAdd(A.n_spill, 1u);
          }
        }
        if (q.valid) write_record<EPS>(A, pos, spill, cell, talpha, q.tb, packed, v, q.den, &kept);
        if (EPS) my_kept += kept ? 1u : 0u;
      };
      if (!zero) {
        auto decode = [&](uint32_t e0, Chunk &q) {
          const uint32_t e = e0 + lane;
          q.valid = e < eend;
          q.tb = B;
          q.den = Bz;
          q.sign = 0;
          q.g = 0.0;
          q.gf = 0.0f;
          if (q.valid && e > 0) {
            const uint32_t sp = s_sp[e - 1], h = sp & 0xffu, p = sp >> 8;
            const Orb i = occ[h], a = vir[p];
            const int ix = i.x * n + a.x;
            q.tb = B ^ (1u << i.x) ^ (1u << a.x);
            q.den = Bz - (a.z - i.z - s_jk[ix]);
            q.sign = (pa + h + (uint32_t)a.x - p + (a.x > i.x ? 1u : 0u)) & 1u;
            if (PREC != 0) q.gf = erow32[ix];
            else q.g = erow[ix];
          }
          place(q, e);
        };
        // software-pipelined: the next chunk's slots (an atomic for big
        // classes) and integrals are requested before this chunk is written
        Chunk x, y;
        decode(0, x);
#pragma unroll 1
        for (uint32_t e0 = 0; e0 < eend; e0 += 64) {  // warp-uniform
          if (e0 + 32 < eend) decode(e0 + 32, y);
          emit(x, h0, e0 + lane == 0);
          if (e0 + 32 >= eend) break;
          if (e0 + 64 < eend) decode(e0 + 64, x);
          emit(y, h0, false);
        }
      } else {
        auto decode = [&](uint32_t e0, Chunk &q) {
          const uint32_t e = e0 + lane;
          q.valid = e < eend;
          q.tb = B;
          q.den = Bz;
          q.sign = 0;
          q.g = 0.0;
          q.gf = 0.0f;
          if (q.valid && e >= sb) {
            const uint32_t f = e - sb, qq = A.dv_pb_p.div(f);
            const uint32_t hp = s_pair[qq], pp = s_pair[f - qq * A.dv_pb_p.d];
            const uint32_t h1 = hp & 0xffu, h2 = hp >> 8, p1 = pp & 0xffu, p2 = pp >> 8;
            const Orb i = occ[h1], j = occ[h2], a = vir[p1], b = vir[p2];
            const uint32_t pm = (1u << a.x) | (1u << b.x);
            q.tb = B ^ ((1u << i.x) | (1u << j.x)) ^ pm;
            q.den = Bz - (a.z + b.z - i.z - j.z + s_jk[j.x * n + i.x] + s_jk[b.x * n + a.x] -
                          s_jk[i.x * n + a.x] - s_jk[j.x * n + a.x] - s_jk[i.x * n + b.x] -
                          s_jk[j.x * n + b.x]);
            const uint32_t between = below(j.x) & ~((2u << i.x) - 1u);
            q.sign = (h1 + h2 + (uint32_t)a.x - p1 + (uint32_t)b.x - p2 + 1u +
                      (uint32_t)__popc(pm & between)) & 1u;
            const size_t ix = (((size_t)j.x * n + b.x) * n + i.x) * n + a.x;
            if (PREC != 0) q.gf = A.I.asymT32[ix];
            else q.g = A.I.asymT[ix];
          } else if (q.valid) {  // beta single
            const uint32_t sp = s_sp[e], h = sp & 0xffu, p = sp >> 8;
            const Orb i = occ[h], a = vir[p];
            q.tb = B ^ (1u << i.x) ^ (1u << a.x);
            q.den = Bz - (a.z - i.z - s_jk[i.x * n + a.x]);
            q.sign = (h + (uint32_t)a.x - p + (a.x > i.x ? 1u : 0u)) & 1u;
            q.g = flip_sign(fx64_to_double(fx_single(A.X, B, R.Ak, i.x, a.x), A.X.s1), q.sign);
          }
          place(q, e);
        };
        Chunk x, y;
        decode(ebeg, x);
#pragma unroll 1
        for (uint32_t e0 = ebeg; e0 < eend; e0 += 64) {
          if (e0 + 32 < eend) decode(e0 + 32, y);
          emit(x, x.g, e0 + lane < sb);
          if (e0 + 32 >= eend) break;
          if (e0 + 64 < eend) decode(e0 + 64, x);
          emit(y, y.g, e0 + 32 + lane < sb);
        }
      }
    }
  }
  if (EPS) add_survivors(A, my_kept);
}

// Alpha-double pairs, flat: CTA step s covers flat pairs [s * kAdTile, ...).
// An item's orbitals are the bits in which its target differs from its group's
// alpha string (unranking the operation's number took some 300 instructions an
// item, of 2.2 pairs at (24e,30o)).
template <bool EPS, int PREC>
__global__ void __launch_bounds__(kAdThreads) k_emit_ad(EmitArgs A) {
  using D = uint32_t;
  __shared__ uint32_t sF[kAdTile + 1];    // first flat pair of each item in the step
  __shared__ uint32_t sPos[kAdTile + 1];  // in-place staging slot of the item's first pair
  __shared__ uint32_t sG[kAdTile + 1];    // first core determinant of the item's group
  __shared__ uint32_t sOrb[kAdTile + 1];  // i | a << 5 | j << 10 | b << 15 | kind << 20
  __shared__ uint32_t sTA[kAdTile + 1];   // target alpha string
  __shared__ uint32_t sNb[kAdTile + 1];   // buckets and first cell of the item's class
  __shared__ uint32_t sCell[kAdTile + 1];
  __shared__ uint32_t sBase[kAdTile + 1]; // first staging slot of the class
  __shared__ double sH[kAdTile + 1];      // signed matrix element
  __shared__ D sD[kAdTile + 1];           // determinant-independent diagonal change
  __shared__ uint16_t sItem[kAdTile];     // item of each pair of the step
  const int n = A.I.n;
  const uint32_t omask = (1u << A.opbits) - 1u;
  const int lane = threadIdx.x & 31;
  const D *jk = A.jk;
  unsigned long long my_kept = 0;  // pairs kept by the eps screen (EPS)
#pragma unroll 1
  for (uint32_t step = blockIdx.x; step < A.ad_tiles; step += gridDim.x) {
    const uint32_t fb = step * kAdTile;
    const uint32_t fe = fb + kAdTile < A.ad_total ? fb + kAdTile : A.ad_total;
    const uint32_t ja = A.ad_tile_item[step];
    uint32_t jl = A.ad_tile_item[step + 1];
    if (jl >= A.nad) jl = A.nad - 1;
    const int nspan = (int)(jl - ja + 1);  // <= kAdTile + 1: every item has >= 1 pair
    for (int i = threadIdx.x; i < nspan; i += kAdThreads) {
      const uint64_t t = A.t0 + A.adl[ja + i];
      const uint64_t it = A.items[t];
      const uint32_t k = (uint32_t)it >> A.opbits;
      const uint32_t gi = A.item_group[t] - A.gb0;
      const uint32_t kd = A.kind[gi], Ak = A.grp_alpha[k], At = (uint32_t)(it >> 32);
      const uint64_t so = A.soff[gi];
      sF[i] = A.ad_off[ja + i];
      sPos[i] = (uint32_t)(so + (A.Wexcl[t] - A.g_P0[A.gb0 + gi]));
      sBase[i] = (uint32_t)so;
      sG[i] = A.grp_start[k];
      sTA[i] = At;
      sNb[i] = kd == kTileBucket ? A.nb[gi] : 0u;
      sCell[i] = kd == kTileBucket ? A.cellbase[gi] : 0u;
      const uint32_t hm = Ak & ~At, pm = At & ~Ak;
      const int ia = __ffs(hm) - 1, ja2 = 31 - __clz(hm), aa = __ffs(pm) - 1, ba = 31 - __clz(pm);
      sOrb[i] = (uint32_t)ia | ((uint32_t)aa << 5) | ((uint32_t)ja2 << 10) | ((uint32_t)ba << 15) |
                (kd << 20);
      const size_t ix = (((size_t)ia * n + aa) * n + ja2) * n + ba;
      sH[i] = flip_sign(PREC != 0 ? widen(A.I.asym32[ix]) : A.I.asym[ix],
                        double_sign(Ak, ia, ja2, aa, ba));
      sD[i] = jk[ia * n + ja2] + jk[aa * n + ba] - jk[aa * n + ia] - jk[aa * n + ja2] -
              jk[ba * n + ia] - jk[ba * n + ja2];
    }
    __syncthreads();
    // pair -> item map of the step: each item marks its pairs
    for (int i = threadIdx.x; i < nspan; i += kAdThreads) {
      const uint32_t a0 = sF[i] > fb ? sF[i] : fb;
      const uint32_t e1 = i + 1 < nspan ? sF[i + 1] : fe;
      const uint32_t a1 = e1 < fe ? e1 : fe;
      for (uint32_t f = a0; f < a1; ++f) sItem[f - fb] = (uint16_t)i;
    }
    __syncthreads();
#pragma unroll 1
    for (uint32_t f0 = fb + (threadIdx.x & ~31u); f0 < fe; f0 += kAdThreads) {
      const uint32_t f = f0 + lane;
      const bool valid = f < fe;
      const int lo = valid ? (int)sItem[f - fb] : 0;
      const uint32_t q = valid ? f - sF[lo] : 0u;
      uint32_t jdx = sG[lo] + q;
      const uint32_t ob = sOrb[lo], kd = ob >> 20;
      const bool bigl = valid && kd == kTileBucket;
      if (valid && jdx >= A.ncore) {
        atomicOr(A.err, kErrCore);
        jdx = 0;
      }
      CoreRec cr = {0u, 0u, 0.0};
      if (valid) cr = A.core[jdx];
      const uint32_t B = cr.beta;
      // lanes of one warp may straddle classes of both kinds: position per lane
      uint32_t pos = sPos[lo] + q, cell = 0;
      bool spill = false;
      if (__any_sync(0xffffffffu, bigl)) {
        const uint32_t bkt = bigl ? bucket_of(B, sNb[lo]) : 0u;
        cell = sCell[lo] + bkt;
        const bool few = __any_sync(0xffffffffu, bigl && sNb[lo] < kFewBuckets);
        uint32_t peers = 0;
        const uint32_t raw = claim_slot(A.fill, cell, bigl, few, &peers);
        const uint32_t slot = claimed_slot(raw, few, peers);
        if (bigl) {
          if (slot < (uint32_t)kCap) {
            pos = sBase[lo] + bkt * (uint32_t)kCap + slot;
          } else {
            spill = true;
            pos = atomicAdd(A.n_spill, 1u);
          }
        }
      }
      bool kept = false;
      if (valid) {
        const D *Fa = A.Fa + jdx;  // orbital p at Fa[p * ncore]
        const size_t m = A.ncore;
        const D dh = sD[lo] + Fa[((ob >> 5) & 31u) * m] + Fa[((ob >> 15) & 31u) * m] -
                     Fa[(ob & 31u) * m] - Fa[((ob >> 10) & 31u) * m];
        write_record<EPS>(A, pos, spill, cell, sTA[lo], B, kd == kTilePacked,
                          pair_value<PREC>(sH[lo], cr.c, (float)cr.c), cr.den - dh, &kept);
      }
      if (EPS) my_kept += kept ? 1u : 0u;
    }
    __syncthreads();  // the next step overwrites the item arrays
  }
  if (EPS) add_survivors(A, my_kept);
}

// Per item of the batch: determinant runs (o = 0 or an alpha single) and the
// alpha-double flag.
__global__ void k_batch_counts(const uint64_t *items, uint64_t t0, uint64_t nt, int opbits,
                               uint32_t sa, uint32_t npieces, const uint32_t *grp_count,
                               uint32_t *rcnt, uint32_t *adf, uint32_t *adw) {
  const uint32_t omask = (1u << opbits) - 1u;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nt;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t lo = (uint32_t)items[t0 + i];
    const uint32_t k = lo >> opbits, o = lo & omask;
    rcnt[i] = o == 0 ? grp_count[k] * npieces : (o <= sa ? grp_count[k] : 0u);
    adf[i] = o > sa ? 1u : 0u;
    adw[i] = o > sa ? grp_count[k] : 0u;
  }
}

// Totals of the batch plan's scans, for one copy to the host: staging slots,
// bucket cells, tiles, runs, alpha-double items and their pairs.
struct PlanTotals {
  uint64_t slots, cells, tiles, runs, ad, ad_pairs;
};
__global__ void k_plan_totals(uint32_t ng, const uint64_t *soff, const uint64_t *slots,
                              const uint32_t *cellbase, const uint32_t *nb,
                              const uint32_t *tile_base, const uint32_t *ntile, uint64_t nt,
                              const uint32_t *roff, const uint32_t *rcnt, const uint32_t *adpos,
                              const uint32_t *adf, const uint32_t *adsum, const uint32_t *adw,
                              PlanTotals *out) {
  const uint32_t g = ng - 1;
  const uint64_t i = nt - 1;
  out->slots = soff[g] + slots[g];
  out->cells = (uint64_t)cellbase[g] + nb[g];
  out->tiles = (uint64_t)tile_base[g] + ntile[g];
  out->runs = (uint64_t)roff[i] + rcnt[i];
  out->ad = (uint64_t)adpos[i] + adf[i];
  out->ad_pairs = (uint64_t)adsum[i] + adw[i];
}

__global__ void k_batch_lists(const uint64_t *items, uint64_t t0, uint64_t nt, int opbits,
                              uint32_t sa, const uint32_t *rcnt, const uint32_t *roff,
                              const uint32_t *adpos, const uint32_t *adsum,
                              uint64_t *runs, uint32_t *adl, uint32_t *ad_off) {
  const uint32_t omask = (1u << opbits) - 1u;
  const int lane = (int)(threadIdx.x & 31u);
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  // warps take 32 items at a time (warp-uniform loop); the runs of the 32
  // items are then written by the whole warp, item by item, so that an item
  // with many runs (a big group's o = 0 item, in pieces) is not one thread's
  for (uint64_t base = (((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 32; base < nt;
       base += nwarps * 32) {
    const uint64_t i = base + (uint64_t)lane;
    uint32_t cnt = 0, start = 0;
    if (i < nt) {
      const uint32_t lo = (uint32_t)items[t0 + i];
      const uint32_t o = lo & omask;
      if (o <= sa) {
        cnt = rcnt[i];
        start = roff[i];
      } else {
        adl[adpos[i]] = (uint32_t)i;
        ad_off[adpos[i]] = adsum[i];
      }
    }
    for (uint32_t have = __ballot_sync(0xffffffffu, cnt != 0); have; have &= have - 1) {
      const int j = __ffs(have) - 1;
      const uint32_t c = __shfl_sync(0xffffffffu, cnt, j);
      const uint32_t st = __shfl_sync(0xffffffffu, start, j);
      const uint64_t ii = base + (uint64_t)j;
      for (uint32_t m = (uint32_t)lane; m < c; m += 32) runs[(uint64_t)st + m] = (ii << 32) | m;
    }
  }
}

// The psi determinants of each tile (as a set: their order within a tile does
// not matter), by counting instead of sorting: k_psi_route finds each one's
// tile and its number in it (counted in psi_hi), k_psi_base gives every tile met
// a range of the list, k_psi_place fills it.  A sort of the (tile, index) words
// took some 25 launches a batch, 0.4 of the 7.6 ms of a (16e,16o) search.
__global__ void k_psi_route(const uint64_t *psi_keys, size_t npsi, const uint32_t *g_alpha,
                            uint32_t gb0, uint32_t ng, const uint32_t *kind, const uint32_t *nb,
                            const uint64_t *Ws, const uint32_t *tile_base, TileDesc *tiles,
                            uint64_t *out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npsi;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t key = psi_keys[i];
    const uint32_t a = key_alpha(key), b = (uint32_t)(key >> 32);
    uint32_t lo = 0, hi = ng;  // first class with alpha >= a
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if (g_alpha[gb0 + mid] < a) lo = mid + 1; else hi = mid;
    }
    uint64_t r = ~0ull;  // its alpha string is no class of the batch
    if (lo < ng && g_alpha[gb0 + lo] == a) {
      const uint32_t k = kind[lo];
      uint32_t t;
      if (k == kTilePacked) t = packed_start(lo, kind, Ws) ? tile_base[lo] : tile_base[lo] - 1;
      else if (k == kTileMedium) t = tile_base[lo];
      else t = tile_base[lo] + bucket_of(b, nb[lo]);
      r = ((uint64_t)t << 32) | atomicAdd(&tiles[t].psi_hi, 1u);
    }
    out[i] = r;
  }
}

__global__ void k_psi_base(const uint64_t *route, size_t npsi, TileDesc *tiles, unsigned *total) {
  const uint32_t lane = threadIdx.x & 31u;
  // warp-uniform loop: one atomic per warp
  for (size_t i0 = (size_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); i0 < npsi;
       i0 += (size_t)gridDim.x * blockDim.x) {
    const uint64_t r = i0 + lane < npsi ? route[i0 + lane] : ~0ull;
    const bool first = (uint32_t)r == 0u;  // number 0 of its tile
    const uint32_t t = (uint32_t)(r >> 32), c = first ? tiles[t].psi_hi : 0u;
    uint32_t sum = c;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, sum, o);
      if ((int)lane >= o) sum += y;
    }
    uint32_t base = 0;
    if (lane == 31 && sum) base = atomicAdd(total, sum);
    base = __shfl_sync(0xffffffffu, base, 31) + sum - c;
    if (first) {
      tiles[t].psi_lo = base;
      tiles[t].psi_hi = base + c;
    }
  }
}

__global__ void k_psi_place(const uint64_t *route, const uint64_t *psi_keys, size_t npsi,
                            const TileDesc *tiles, uint64_t *psi_list) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < npsi;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t r = route[i];
    if (r != ~0ull) psi_list[tiles[(uint32_t)(r >> 32)].psi_lo + (uint32_t)r] = psi_keys[i];
  }
}

// First alpha-double item of each CTA step: the last item starting at or
// before the step's first flat pair.
__global__ void k_ad_tile_items(const uint32_t *ad_off, uint32_t nad, uint32_t total,
                                uint32_t nsteps, uint32_t *tile_item) {
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s <= nsteps;
       s += gridDim.x * blockDim.x) {
    uint32_t f = s * (uint32_t)kAdTile;
    if (f >= total) f = total - 1;
    uint32_t lo = 0, hi = nad - 1;
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (ad_off[mid] <= f) lo = mid; else hi = mid - 1;
    }
    tile_item[s] = lo;
  }
}

// ---------------------------------------------------------- tile kernel ---

struct CellArgs {
  const TileDesc *tiles;
  uint32_t ntiles;     // tiles [tile0, ntiles) are visited
  uint32_t tile0;
  Stage st;
  double tau;
  float tau_f;
  const uint64_t *psi_ht;
  uint64_t psi_mask;
  const uint64_t *psi_list;  // psi keys of the batch in tile order
  uint64_t *cand_key;
  double *cand_score;
  unsigned long long *cand_count;
  unsigned long long cand_cap;
  unsigned long long *n_unique, *n_excluded;
  unsigned *err;
  int screened;  // records may carry the eps screen's drop marker
  // targets of several records that can reach the threshold, summed by
  // k_long_sums: the values of each, and (candidate slot, offset << 16 | length)
  double *lv;
  unsigned long long *lv_count;
  unsigned long long lv_cap;
  ulonglong2 *fix;
  unsigned long long *nfix;
  unsigned long long fix_cap;
};

__device__ __forceinline__ uint64_t mix_key(uint64_t z) {
  z ^= z >> 33;
  z *= 0xff51afd7ed558ccdull;
  z ^= z >> 33;
  z *= 0xc4ceb9fe1a85ec53ull;
  z ^= z >> 33;
  return z;
}

// Hash of a target key within a tile: a product per word and the multiply of
// a finalizer, whose high half picks the slot (the top bits of a product
// depend on every bit below them).  Bucket tiles hold one alpha string and the
// betas of one bucket, which another multiplier picked.  The two rounds more
// of the full MurmurHash3 finalizer (Appleby) spread no better and cost 0.5%
// of a (24e,30o) search.
__device__ __forceinline__ uint32_t tile_mix(uint64_t key) {
  uint32_t h = (uint32_t)key * 0x9E3779B1u + (uint32_t)(key >> 32) * 0x85EBCA6Bu;
  h ^= h >> 16;
  h *= 0xC2B2AE35u;
  return h >> 16;
}

// Open addressing with linear probing; the table is at most 1/4 full, and the
// probe count is bounded by the table size (exceeding it sets *err).
__device__ __forceinline__ bool psi_contains(const uint64_t *ht, uint64_t mask, uint64_t key,
                                             unsigned *err) {
  uint64_t h = mix_key(key) & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    uint64_t s = ht[h];
    if (s == key) return true;
    if (s == ~0ull) return false;
    h = (h + 1) & mask;
  }
  atomicOr(err, kErrProbe);
  return false;
}

// A tile's records are grouped by target in a shared-memory hash table whose
// slots are single words: the first record of the target (the one that claimed
// the slot), how many more records it has, and the sum over those of a
// quantised bound of |v| / (tau |E0 - H_ii|).  Integer atomics build the word,
// so nothing is walked: after one pass over the records the claiming thread
// knows whether its target has one record (it is scored by its own value),
// cannot reach the threshold (it is only counted), or can (its values are
// copied out and summed after the launch by k_long_sums).  The psi
// determinants that fall in the tile are entered as markers, so a target in
// psi is recognised without a global lookup.  The numerator is formed by a
// rule that depends only on the multiset of a target's values, so grouping by
// hashing gives the result of sorting the records and summing the runs.
//
// Word of a slot, B = log2 of the tile's record capacity:
//   bits 0 .. B-1        the claiming record, or the index of a psi marker
//   bit  B               the target is in psi
//   bit  B+1             psi marker; empty slot (index all ones); or, once the
//                        target was found to reach the threshold, the index
//                        (below CAP / 2) of its cursor in S.cur
//   bits B+2 .. 2B+1     further records of the target
//   bits 2B+2 .. 31      sum of their quantised bounds
// A quantised bound is at most kThr, and a target of kLong or more records
// reaches the threshold whatever its sum, so the sum of a target that is
// tested, of at most kLong - 2 further records, cannot overflow its field;
// the sum of a longer one may, off the top of the word.  A target's records
// all count before any is tested, and their order does not matter.
constexpr int kPsiCap = 64;  // psi markers per tile; more: global lookups

// The tile kernel comes in three sizes: tiles of kCap records (every packed,
// medium and bucket tile) and tiles of kMidCap and kBigCap records for the
// hash buckets that hot targets overfilled (bucket tiles only).  Eight records
// per thread (a warp's overhead per tile and the longest of its lanes' probe
// sequences are shared by more of them) and four hash slots per record (with
// two, an eighth of the records meet another target on their first probe).
constexpr int kMidCap = 2048;
constexpr int kMidThreads = 256;
constexpr int kBigCap = 4096;
constexpr int kBigThreads = 512;
constexpr int kRPT = 8;  // records per thread

template <int CAP>
constexpr int log2_of() {
  int b = 0;
  while ((1 << b) < CAP) ++b;
  return b;
}

template <int CAP>
struct SlotWord {
  static constexpr int B = log2_of<CAP>();
  static constexpr uint32_t kIndex = (uint32_t)CAP - 1u;
  static constexpr uint32_t kPsi = 1u << B;
  static constexpr uint32_t kMark = 2u << B;
  static constexpr uint32_t kEmpty = kMark | kIndex;
  static constexpr int kCountShift = B + 2;
  static constexpr uint32_t kOne = 1u << kCountShift;
  static constexpr int kSumShift = 2 * B + 2;
  static constexpr uint32_t kLong = CAP <= 1024 ? 32u : 8u;
  static constexpr uint32_t kThr = (1u << (32 - kSumShift)) / kLong;
  static_assert((1 << B) == CAP, "capacity must be a power of two");
  static_assert((kLong - 2) * kThr < (1u << (32 - kSumShift)), "the sum must fit its field");
  static_assert(kPsiCap < CAP / 2, "markers and cursors differ from the empty word");
};

template <int CAP>
struct CellSmem {
  static constexpr int kTab = 4 * CAP;  // hash slots (load <= 1/4)
  uint64_t key[CAP];            // target keys of the tile's records
  uint64_t psik[kPsiCap];       // psi keys of the tile
  uint32_t slot[kTab];
  uint32_t cur[CAP / 2];        // next value position of each target that reaches the threshold
  uint32_t ncur;                // their number
};

// A tile that the kernel reduces on chip; oversized hash buckets go to the
// global path, anything else outside the limits is a planning bug.
template <int CAP>
__device__ __forceinline__ bool tile_on_chip(const TileDesc &d, uint64_t stage_cap,
                                             unsigned *err) {
  const bool fits = d.npairs <= (uint32_t)CAP && (uint64_t)d.start + d.npairs <= stage_cap;
  if (!fits && threadIdx.x == 0 &&
      !(d.kind == kTileBucket && d.npairs > (uint32_t)kCap &&
        (uint64_t)d.start + kCap <= stage_cap))
    atomicOr(err, kErrTile);
  return fits;
}

// |v| / (tau |den|) in units of 1 / kThr, rounded up, at most kThr.  inv_tau is
// kThr / tau_f, or infinity without a threshold.  An upper bound: |v| is
// truncated to a float from its bits (no FP64 instruction; within 2^-23),
// |den| was staged as a lower bound, rounded to a float, and tau_f rounded down,
// and the factor 1.00001 covers those and the float operations.  A value above the normal
// float range, a zero denominator and anything that is not a number count as
// reaching the threshold; a |v| below the range counts as its smallest value.
template <uint32_t kThr>
__device__ __forceinline__ uint32_t quantised_bound(uint32_t v_lo, uint32_t v_hi, float den,
                                                    float inv_tau) {
  const uint32_t hi = v_hi & 0x7fffffffu;
  float vf = __uint_as_float(__funnelshift_l(v_lo, hi - 0x38000000u, 3));
  if (hi < 0x38100000u) vf = 1.17549435e-38f;
  const float r = __fdividef(vf * 1.00001f, fabsf(den)) * inv_tau;
  const bool big = !(r < (float)kThr) || hi >= 0x47f00000u || den == 0.0f;
  return big ? kThr : __float2uint_ru(r);
}

// One CTA reduces tiles blockIdx.x, + gridDim.x, ...  Thread t holds records t,
// t + THREADS, ... of a tile in registers.  Three barriers per tile, a fourth
// when a target of several records reaches the threshold.
//
// Bound: instruction issue (the records are read once, at 1.7 TB/s): about 200
// warp instructions per 32 records at (24e,30o), 58% of issue slots.  The
// linked lists this replaces (a filter of singletons, then a list per target,
// walked by one thread) issued about 340 and waited at the barriers for the
// warps that walked: 116.8 ms per (24e,30o) search, C = 1e5, against 71.  Four
// records in 256 threads take 95 ms; twice the CTAs on half the slots 12 ms
// more; keys in place before the claims without the first barrier (fences
// instead) 8 ms more.
template <int CAP, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS) k_cells(CellArgs C) {
  using Smem = CellSmem<CAP>;
  using W = SlotWord<CAP>;
  constexpr uint32_t kTabMask = (uint32_t)Smem::kTab - 1u;
  static_assert(CAP == kRPT * THREADS && THREADS >= kPsiCap, "records per thread");
  static_assert(kRPT == 8 && W::kThr < 256 && Smem::kTab <= 65536, "packed bounds and slots");
  // a warp's candidates, lists and values in one word
  constexpr int kListShift = 9, kValueShift = 18;
  constexpr uint32_t kWarpMask = (1u << kListShift) - 1u;
  static_assert(32 * kRPT <= (int)kWarpMask && kValueShift == 2 * kListShift &&
                    (uint32_t)CAP <= (0xffffffffu >> kValueShift),
                "a warp's counts must fit their fields");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem &S = *reinterpret_cast<Smem *>(smem_raw);
  const int lane = threadIdx.x & 31;
  uint32_t my_unique = 0, my_excl = 0;
  for (int i = threadIdx.x; i < Smem::kTab; i += THREADS) S.slot[i] = W::kEmpty;
  if (threadIdx.x == 0) S.ncur = 0;
  const float inv_tau = C.tau_f > 0.0f ? (float)W::kThr / C.tau_f : __int_as_float(0x7f800000);
  uint32_t tile = C.tile0 + blockIdx.x;
  TileDesc d = {0, 0, 0, 0, 0, 0, 0, 0};
  if (tile < C.ntiles) d = C.tiles[tile];
#pragma unroll 1
  for (; tile < C.ntiles; tile += gridDim.x) {
    const bool on = tile_on_chip<CAP>(d, C.st.cap, C.err);
    const uint32_t nrec = on ? d.npairs : 0u;
    const uint32_t npsi = on ? d.psi_hi - d.psi_lo : 0u;
    const bool psi_local = npsi <= (uint32_t)kPsiCap;
    // record k of this thread: its value, and by 8 and 16 bits its quantised
    // bound and its slot
    double v[kRPT];
    uint64_t q = 0, slot_lo = 0, slot_hi = 0;
    uint32_t live = 0;
    auto bound_of = [&](int k) { return (uint32_t)(q >> (8 * k)) & 0xffu; };
    auto slot_of = [&](int k) {
      return (uint32_t)((k < 4 ? slot_lo : slot_hi) >> (16 * (k & 3))) & 0xffffu;
    };
    const StageRec *src = C.st.rec + d.start + threadIdx.x;
    uint64_t pkey = 0;
    const bool has_marker = psi_local && threadIdx.x < npsi;
    if (has_marker) pkey = C.psi_list[d.psi_lo + threadIdx.x];
#pragma unroll
    for (int k0 = 0; k0 < kRPT; k0 += 4) {
      if ((uint32_t)(k0 * THREADS) >= nrec) {  // uniform
#pragma unroll
        for (int k = k0; k < k0 + 4; ++k) v[k] = 0.0;
        continue;
      }
      uint4 raw[4];
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (threadIdx.x + (uint32_t)((k0 + k) * THREADS) < nrec)
          raw[k] = __ldcs(reinterpret_cast<const uint4 *>(src + (k0 + k) * THREADS));
        else
          raw[k] = make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t e = threadIdx.x + (uint32_t)((k0 + k) * THREADS);
        v[k0 + k] = __hiloint2double((int)raw[k].y, (int)raw[k].x);
        if (e < nrec) {
          const uint32_t alpha = d.kind == kTilePacked ? __ldcs(C.st.alpha + d.start + e) : d.alpha;
          const uint64_t key = pack_key(alpha, raw[k].z);
          S.key[e] = key;
          const uint64_t h = tile_mix(key) & kTabMask;
          if (k0 == 0) slot_lo |= h << (16 * k);
          else slot_hi |= h << (16 * k);
          if (!(C.screened && is_dropped(v[k0 + k]))) live |= 1u << (k0 + k);
          q |= (uint64_t)quantised_bound<W::kThr>(raw[k].x, raw[k].y, __uint_as_float(raw[k].w),
                                                  inv_tau)
               << (8 * (k0 + k));
        }
      }
    }
    if (has_marker) S.psik[threadIdx.x] = pkey;
    TileDesc dn = {0, 0, 0, 0, 0, 0, 0, 0};
    if (tile + gridDim.x < C.ntiles) dn = C.tiles[tile + gridDim.x];
    __syncthreads();  // keys in place; the previous tile is done with the table
    if (threadIdx.x == 0) S.ncur = 0;
    // the next tile's records start towards L2
    if (threadIdx.x == 0 && dn.npairs - 1u < (uint32_t)CAP &&
        (uint64_t)dn.start + dn.npairs <= C.st.cap)
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(C.st.rec + dn.start),
                   "r"(dn.npairs * 16u)
                   : "memory");
    // psi markers: claim a slot, or flag the slot that a record holds
    uint32_t marker = 0xffffffffu;
    if (has_marker) {
      uint32_t h = tile_mix(pkey) & kTabMask;
      int probe = 0;
      for (; probe < Smem::kTab; ++probe) {
        const uint32_t w = atomicCAS(&S.slot[h], W::kEmpty, W::kMark | threadIdx.x);
        if (w == W::kEmpty) {
          marker = h;
          break;
        }
        if (!(w & W::kMark) && S.key[w & W::kIndex] == pkey) {
          atomicOr(&S.slot[h], W::kPsi);
          break;
        }
        h = (h + 1) & kTabMask;
      }
      if (probe == Smem::kTab) atomicOr(C.err, kErrTile);  // cannot happen at load < 1/2
    }
    // the records' first probes, issued before any result is used
    uint32_t claimed = live, rest = 0, met = 0;
#pragma unroll
    for (int k0 = 0; k0 < kRPT; k0 += 4) {
      if ((uint32_t)(k0 * THREADS) >= nrec) break;  // uniform
      uint32_t got[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        got[k] = W::kEmpty;
        if ((live >> (k0 + k)) & 1u)
          got[k] = atomicCAS(&S.slot[slot_of(k0 + k)], W::kEmpty,
                             threadIdx.x + (uint32_t)((k0 + k) * THREADS));
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (got[k] != W::kEmpty) {
          const uint64_t key = S.key[threadIdx.x + (uint32_t)((k0 + k) * THREADS)];
          claimed &= ~(1u << (k0 + k));
          const bool mark = (got[k] & W::kMark) != 0u;
          if (!mark && S.key[got[k] & W::kIndex] == key) {
            atomicAdd(&S.slot[slot_of(k0 + k)], W::kOne | (bound_of(k0 + k) << W::kSumShift));
          } else {
            rest |= 1u << (k0 + k);
            if (!mark) met |= 1u << (k0 + k);
          }
        }
      }
    }
    // the others probe on, a thread's one after another in one loop (so that
    // a warp loops for its busiest thread, not for its unluckiest record of
    // each round)
    if (rest) {
      int k = __ffs(rest) - 1, probe = 0;
      uint64_t key = S.key[threadIdx.x + (uint32_t)(k * THREADS)];
      // a first probe that met another target's record need not be repeated
      uint32_t h = (slot_of(k) + ((met >> k) & 1u)) & kTabMask;
      for (;;) {
        const uint32_t e = threadIdx.x + (uint32_t)(k * THREADS);
        const uint32_t w = atomicCAS(&S.slot[h], W::kEmpty, e);
        bool done = w == W::kEmpty, own = done;
        if (!done) {
          const bool mark = (w & W::kMark) != 0u;
          done = (mark ? S.psik[w & W::kIndex] : S.key[w & W::kIndex]) == key;
          // the first record of a psi marker's target takes the slot over
          if (done && mark) own = atomicCAS(&S.slot[h], w, e | W::kPsi) == w;
          if (done && !own) atomicAdd(&S.slot[h], W::kOne | (bound_of(k) << W::kSumShift));
        }
        if (!done && ++probe < Smem::kTab) {
          h = (h + 1) & kTabMask;
          continue;
        }
        if (!done) atomicOr(C.err, kErrTile);  // cannot happen at load < 1/2
        if (own) claimed |= 1u << k;
        const int sh = 16 * (k & 3);
        if (k < 4) slot_lo = (slot_lo & ~(0xffffull << sh)) | ((uint64_t)h << sh);
        else slot_hi = (slot_hi & ~(0xffffull << sh)) | ((uint64_t)h << sh);
        rest &= rest - 1u;
        if (!rest) break;
        k = __ffs(rest) - 1;
        probe = 0;
        h = (slot_of(k) + ((met >> k) & 1u)) & kTabMask;
        key = S.key[threadIdx.x + (uint32_t)(k * THREADS)];
      }
    }
    __syncthreads();  // every slot word is complete
    // the claiming thread decides on its target and empties the slot, unless
    // the target's values are to be copied out
    uint32_t pass = 0, multi = 0, own = 0;  // own: candidates, lists, values (packed)
    my_unique += (uint32_t)__popc(claimed);
#pragma unroll
    for (int k = 0; k < kRPT; ++k) {
      if (!((claimed >> k) & 1u)) continue;
      const uint32_t h = slot_of(k), w = S.slot[h];
      const uint32_t more = (w >> W::kCountShift) & (uint32_t)(CAP - 1);
      bool in_psi = (w & W::kPsi) != 0u;
      if (!psi_local)
        in_psi = psi_contains(C.psi_ht, C.psi_mask,
                              S.key[threadIdx.x + (uint32_t)(k * THREADS)], C.err);
      if (in_psi) {
        ++my_excl;
      } else if ((w >> W::kSumShift) + bound_of(k) >= W::kThr || more + 1u >= W::kLong) {
        pass |= 1u << k;
        if (more) {
          multi |= 1u << k;
          own += (1u << kListShift) + ((more + 1u) << kValueShift);
          continue;
        }
      }
      S.slot[h] = W::kEmpty;
    }
    // a marker that no record's target took over (in_psi targets are never
    // copied out, so no cursor takes its place either)
    if (marker != 0xffffffffu && S.slot[marker] == (W::kMark | threadIdx.x))
      S.slot[marker] = W::kEmpty;
    if (__any_sync(0xffffffffu, pass != 0u)) {
      // candidates, targets to be summed and their values: one scan over the
      // warp (at most a candidate and a list for each of its records, whose
      // targets' other records may all be other warps', and CAP values)
      own += (uint32_t)__popc(pass);
      uint32_t sum = own;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, sum, o);
        if (lane >= o) sum += y;
      }
      const uint32_t all = __shfl_sync(0xffffffffu, sum, 31);
      const uint32_t nf = (all >> kListShift) & kWarpMask;
      unsigned long long b0 = 0, f0 = 0, l0 = 0;
      uint32_t c0 = 0;
      if (lane == 0) {
        b0 = atomicAdd(C.cand_count, (unsigned long long)(all & kWarpMask));
        if (nf) {
          f0 = atomicAdd(C.nfix, (unsigned long long)nf);
          l0 = atomicAdd(C.lv_count, (unsigned long long)(all >> kValueShift));
          c0 = atomicAdd(&S.ncur, nf);
        }
      }
      b0 = __shfl_sync(0xffffffffu, b0, 0);
      if (nf) {  // warp-uniform
        f0 = __shfl_sync(0xffffffffu, f0, 0);
        l0 = __shfl_sync(0xffffffffu, l0, 0);
        c0 = __shfl_sync(0xffffffffu, c0, 0);
      }
      const uint32_t before = sum - own;
      b0 += before & kWarpMask;
      f0 += (before >> kListShift) & kWarpMask;
      c0 += (before >> kListShift) & kWarpMask;
      l0 += before >> kValueShift;
#pragma unroll
      for (int k = 0; k < kRPT; ++k) {
        if (!((pass >> k) & 1u)) continue;
        const unsigned long long at = b0++;
        if (at < C.cand_cap) {
          C.cand_key[at] = S.key[threadIdx.x + (uint32_t)(k * THREADS)];
          C.cand_score[at] = v[k];  // the numerator; the exact score is formed after the launch
        }
        if ((multi >> k) & 1u) {
          uint32_t *sl = &S.slot[slot_of(k)];
          const uint32_t len = ((*sl >> W::kCountShift) & (uint32_t)(CAP - 1)) + 1u;
          if (f0 < C.fix_cap && l0 + len <= C.lv_cap && at < C.cand_cap) {
            C.lv[l0] = v[k];
            C.fix[f0] = make_ulonglong2(at, (l0 << 16) | len);
            S.cur[c0] = (uint32_t)l0 + 1u;
            *sl = W::kMark | c0;
          } else {
            atomicOr(C.err, kErrValues);  // the host runs the launch again with more room
            if (f0 < C.fix_cap) C.fix[f0].y = ~0ull;
            *sl = W::kEmpty;
            multi &= ~(1u << k);
          }
          ++f0;
          ++c0;
          l0 += len;
        }
      }
    }
    if (__syncthreads_or(multi != 0u)) {
      // the other records of the targets to be summed
#pragma unroll
      for (int k = 0; k < kRPT; ++k) {
        if (!(((live & ~claimed) >> k) & 1u)) continue;
        const uint32_t w = S.slot[slot_of(k)];
        if (w != W::kEmpty) C.lv[atomicAdd(&S.cur[w & W::kIndex], 1u)] = v[k];
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kRPT; ++k)
        if ((multi >> k) & 1u) S.slot[slot_of(k)] = W::kEmpty;
    }
    d = dn;
  }
  unsigned long long u = my_unique, x = my_excl;
  for (int dl = 16; dl; dl >>= 1) {
    u += __shfl_xor_sync(0xffffffffu, u, dl);
    x += __shfl_xor_sync(0xffffffffu, x, dl);
  }
  if (lane == 0) {
    if (u) atomicAdd(C.n_unique, u);
    if (x) atomicAdd(C.n_excluded, x);
  }
}

// The numerators of the targets with several records that can reach the
// threshold, from the values the tile kernel copied out: two by IEEE addition
// (the correctly rounded exact sum), three or four by the ordered FP64 sum,
// more by the 128-bit fixed-point accumulator anchored to the largest
// exponent.  Each depends only on the multiset of values, so not on the order
// in which they were copied.  Lists of two to four values take one thread, those
// of up to 64 eight lanes, longer ones the warp (integer additions: the same
// bits); a thread that walked lists of up to 32 values alone, load after load,
// made the launch wait 50 us for the longest ones.
constexpr unsigned kLaneList = 64;

// The rule for five or more values, by the LANES lanes of a group (a power of
// two); every lane of the warp takes part, len = 0 for an idle group.  The
// first HELD values of each lane stay in registers, loaded together.
template <unsigned LANES>
__device__ __forceinline__ double group_list_sum(const double *x, unsigned len, unsigned *ovf) {
  constexpr unsigned kHeld = kLaneList / 8;
  const unsigned lane = threadIdx.x & (LANES - 1u);
  double v[kHeld];
#pragma unroll
  for (unsigned k = 0; k < kHeld; ++k) v[k] = lane + k * LANES < len ? x[lane + k * LANES] : 0.0;
  int emax = 1;
#pragma unroll
  for (unsigned k = 0; k < kHeld; ++k) emax = max(emax, fx_exponent(v[k]));
  for (unsigned j = lane + kHeld * LANES; j < len; j += LANES) emax = max(emax, fx_exponent(x[j]));
#pragma unroll
  for (unsigned o = LANES / 2; o; o >>= 1)
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  const int frac = fx128_frac_for(emax);
  Fx128 acc = {0, 0};
#pragma unroll
  for (unsigned k = 0; k < kHeld; ++k)
    if (lane + k * LANES < len) {
      Fx128 t = fx128_from_double(v[k], frac, ovf);
      fx128_add(acc, t);
    }
  for (unsigned j = lane + kHeld * LANES; j < len; j += LANES) {
    Fx128 t = fx128_from_double(x[j], frac, ovf);
    fx128_add(acc, t);
  }
#pragma unroll
  for (unsigned o = LANES / 2; o; o >>= 1) {
    Fx128 t;
    t.lo = __shfl_xor_sync(0xffffffffu, acc.lo, o);
    t.hi = __shfl_xor_sync(0xffffffffu, acc.hi, o);
    fx128_add(acc, t);
  }
  return fx128_to_double(acc, frac);
}

__global__ void __launch_bounds__(256) k_long_sums(const ulonglong2 *fix,
                                                   const unsigned long long *nfix,
                                                   unsigned long long fix_cap, const double *lv,
                                                   double *cand_score, unsigned *err) {
  const unsigned long long n = *nfix < fix_cap ? *nfix : fix_cap;
  const unsigned lane = threadIdx.x & 31u;
  unsigned ovf = 0;
  // warp-uniform loop: the longer lists are shared by the warp's lanes
  for (unsigned long long base = (unsigned long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31u);
       base < n; base += (unsigned long long)gridDim.x * blockDim.x) {
    ulonglong2 f = make_ulonglong2(0, ~0ull);
    if (base + lane < n) f = fix[base + lane];
    const bool used = f.y != ~0ull;
    const unsigned len = (unsigned)(f.y & 0xffffull);
    const double *x = lv + (f.y >> 16);
    if (used && len == 2) cand_score[f.x] = x[0] + x[1];
    if (used && len == 3) cand_score[f.x] = sum4_ordered(0.0, x[0], x[1], x[2]);
    if (used && len == 4) cand_score[f.x] = sum4_ordered(x[0], x[1], x[2], x[3]);
    for (unsigned m = __ballot_sync(0xffffffffu, used && len > 4u && len <= kLaneList); m;) {
      // the next four lists, one per group of eight lanes
      int src = -1;
      for (unsigned g = 0; g < 4 && m; ++g, m &= m - 1)
        if (g == lane >> 3) src = __ffs(m) - 1;
      const unsigned long long y = __shfl_sync(0xffffffffu, f.y, src < 0 ? 0 : src);
      const unsigned long long at = __shfl_sync(0xffffffffu, f.x, src < 0 ? 0 : src);
      const double s = group_list_sum<8>(lv + (src < 0 ? 0ull : y >> 16),
                                         src < 0 ? 0u : (unsigned)(y & 0xffffull), &ovf);
      if (src >= 0 && (lane & 7u) == 0u) cand_score[at] = s;
    }
    for (unsigned m = __ballot_sync(0xffffffffu, used && len > kLaneList); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const unsigned long long y = __shfl_sync(0xffffffffu, f.y, src);
      const double s = group_list_sum<32>(lv + (y >> 16), (unsigned)(y & 0xffffull), &ovf);
      if ((int)lane == src) cand_score[f.x] = s;
    }
  }
  if (ovf) atomicOr(err, kErrAccum);
}

// ---------------------------------------------- oversized hash buckets ---
// A bucket holding more records than one tile is sorted in global memory on
// beta' and its runs are reduced one target per thread.

// Per listed oversized tile: first in-place record, in-place count, target
// alpha string, and its range of the tile-ordered spill list.
__global__ void k_tile_gather(const TileDesc *tiles, const uint32_t *list, uint32_t n,
                              const uint64_t *spill_keys, uint32_t nspill, uint32_t *info) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t t = list[i];
    const TileDesc d = tiles[t];
    uint32_t lo = 0, hi = nspill;  // first spill key of tile t
    while (lo < hi) {
      const uint32_t mid = (lo + hi) >> 1;
      if ((uint32_t)(spill_keys[mid] >> 32) < t) lo = mid + 1; else hi = mid;
    }
    // its end by another search (a hot tile spills thousands of records)
    uint32_t e = lo;
    hi = nspill;
    while (e < hi) {
      const uint32_t mid = (e + hi) >> 1;
      if ((uint32_t)(spill_keys[mid] >> 32) <= t) e = mid + 1; else hi = mid;
    }
    info[5 * i] = d.start;
    info[5 * i + 1] = d.npairs < (uint32_t)kCap ? d.npairs : (uint32_t)kCap;
    info[5 * i + 2] = d.alpha;
    info[5 * i + 3] = lo;
    info[5 * i + 4] = e - lo;
  }
}

// Records of every oversized tile, concatenated (in-place records, then the
// tile's spilled ones): key = (tile position << 32 | beta'), payload =
// position in the concatenation; src = staging index, or spill index with the
// top bit set.
__device__ __forceinline__ const StageRec &big_rec(const StageRec *rec, const StageRec *spill,
                                                   uint64_t src) {
  return (src >> 63) ? spill[(uint32_t)src] : rec[src];
}

__global__ void k_big_gather(const StageRec *rec, const StageRec *spill,
                             const uint64_t *spill_keys, const uint32_t *start,
                             const uint32_t *nin, const uint32_t *slo, const uint32_t *off,
                             uint32_t nt, uint64_t total, uint64_t *keys, uint32_t *idx,
                             uint64_t *src) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = nt - 1;  // tile holding record i
    while (lo < hi) {
      const uint32_t mid = (lo + hi + 1) >> 1;
      if (off[mid] <= i) lo = mid; else hi = mid - 1;
    }
    const uint32_t o = (uint32_t)(i - off[lo]);
    const uint64_t sr = o < nin[lo]
                            ? (uint64_t)start[lo] + o
                            : ((1ull << 63) | (uint32_t)spill_keys[slo[lo] + (o - nin[lo])]);
    keys[i] = ((uint64_t)lo << 32) | big_rec(rec, spill, sr).beta;
    idx[i] = (uint32_t)i;
    src[i] = sr;
  }
}

// One CTA per oversized bucket tile of at most kBigCap records: its in-place
// records and its spilled ones (info row: start, in-place count, alpha, first
// entry of the tile-ordered spill list, spilled count) are copied into one
// range of a scratch staging buffer, and its descriptor is rewritten to point
// there (kind, alpha and psi range unchanged).
__global__ void k_big_tile_gather(const TileDesc *tiles, const uint32_t *list,
                                  const uint32_t *info, const uint32_t *off,
                                  const StageRec *rec, const StageRec *spill_rec,
                                  const uint64_t *spill_keys, StageRec *out, TileDesc *out_desc) {
  const uint32_t i = blockIdx.x;
  const uint32_t *r = info + 5 * (size_t)i;
  const uint32_t start = r[0], nin = r[1], slo = r[3], nsp = r[4], o = off[i];
  for (uint32_t e = threadIdx.x; e < nin; e += blockDim.x) out[o + e] = rec[start + e];
  for (uint32_t e = threadIdx.x; e < nsp; e += blockDim.x)
    out[o + nin + e] = spill_rec[(uint32_t)spill_keys[slo + e]];
  if (threadIdx.x == 0) {
    TileDesc d = tiles[list[i]];
    d.start = o;
    d.npairs = nin + nsp;
    out_desc[i] = d;
  }
}

// A target whose numerator is formed: its psi test, the float screen against
// tau and the append, as on chip; counts unique and excluded targets.
__device__ __forceinline__ void big_emit(double num, uint64_t full, float den, const CellArgs &C,
                                         unsigned long long *my_unique,
                                         unsigned long long *my_excl) {
  ++*my_unique;
  if (psi_contains(C.psi_ht, C.psi_mask, full, C.err)) {
    ++*my_excl;
    return;
  }
  bool pass = true;
  if (C.tau > 0.0) {  // float screen first, as on chip
    bool okn;
    const float nf = abs_as_float(num, &okn);
    const float df = fabsf(den);
    if (okn && df != 0.0f) pass = nf >= C.tau_f * df * 0.99999f;
  }
  if (pass) {  // the exact score is formed after the launch (k_exact_scores)
    const unsigned long long slot = atomicAdd(C.cand_count, 1ull);
    if (slot < C.cand_cap) {
      C.cand_key[slot] = full;
      C.cand_score[slot] = num;
    }
  }
}

// Runs (targets) longer than this go to k_big_reduce_long: a CTA per run.
constexpr uint64_t kLongRun = 64;

__global__ void k_big_reduce(const uint64_t *keys, const uint32_t *idx, const uint64_t *src,
                             uint64_t n, const uint32_t *alpha, const StageRec *spill,
                             CellArgs C, uint64_t *long_runs, unsigned *n_long) {
  unsigned long long my_unique = 0, my_excl = 0;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t sk = keys[i];
    if (i > 0 && keys[i - 1] == sk) continue;
    if (i + kLongRun < n && keys[i + kLongRun] == sk) {  // sorted: the run is long
      long_runs[atomicAdd(n_long, 1u)] = i;
      continue;
    }
    // the same rule as on chip: one or two values by IEEE addition, three or
    // four by the ordered FP64 sum, more by the 128-bit accumulator
    int emax = 1, live = 0;
    double w[4] = {0.0, 0.0, 0.0, 0.0};
    for (uint64_t e = i; e < n && keys[e] == sk; ++e) {
      const double v = big_rec(C.st.rec, spill, src[idx[e]]).v;
      if (is_dropped(v)) continue;
      const int ex = fx_exponent(v);
      emax = ex > emax ? ex : emax;
      if (live < 4) w[live] = v;
      ++live;
    }
    if (!live) continue;
    double num;
    if (live == 1) {
      num = w[0];
    } else if (live == 2) {
      num = w[0] + w[1];
    } else if (live <= 4) {
      num = sum4_ordered(w[0], w[1], w[2], w[3]);
    } else {
      const int frac = fx128_frac_for(emax);
      Fx128 acc = {0, 0};
      unsigned ovf = 0;
      for (uint64_t e = i; e < n && keys[e] == sk; ++e) {
        const double v = big_rec(C.st.rec, spill, src[idx[e]]).v;
        if (is_dropped(v)) continue;
        Fx128 x = fx128_from_double(v, frac, &ovf);
        fx128_add(acc, x);
      }
      if (ovf) atomicOr(C.err, kErrAccum);
      num = fx128_to_double(acc, frac);
    }
    const uint64_t full = pack_key(alpha[sk >> 32], (uint32_t)sk);
    big_emit(num, full, big_rec(C.st.rec, spill, src[idx[i]]).den, C, &my_unique, &my_excl);
  }
  for (int dl = 16; dl; dl >>= 1) {
    my_unique += __shfl_xor_sync(0xffffffffu, my_unique, dl);
    my_excl += __shfl_xor_sync(0xffffffffu, my_excl, dl);
  }
  if ((threadIdx.x & 31) == 0) {
    if (my_unique) atomicAdd(C.n_unique, my_unique);
    if (my_excl) atomicAdd(C.n_excluded, my_excl);
  }
}

// Long runs (hot targets with more than kLongRun records), one CTA per run:
// the run's largest exponent and live count by block reductions, then each
// thread's share in the 128-bit fixed-point accumulator anchored to that
// exponent, added exactly across the block: the same value as one thread
// walking the run (the sum is a function of the multiset).  A run with at
// most four live values (the rest dropped by the screen) takes the ordered
// FP64 rule on thread 0.
__global__ void __launch_bounds__(256) k_big_reduce_long(const uint64_t *keys, const uint32_t *idx,
                                                         const uint64_t *src, uint64_t n,
                                                         const uint32_t *alpha,
                                                         const StageRec *spill, CellArgs C,
                                                         const uint64_t *long_runs,
                                                         const unsigned *n_long) {
  __shared__ int s_emax, s_live;
  __shared__ Fx128 part[256];
  unsigned long long my_unique = 0, my_excl = 0;
  const unsigned nl = *n_long;
  for (unsigned r = blockIdx.x; r < nl; r += gridDim.x) {
    const uint64_t i = long_runs[r];
    const uint64_t sk = keys[i];
    if (threadIdx.x == 0) {
      s_emax = 1;
      s_live = 0;
    }
    __syncthreads();
    int emax = 1, live = 0;
    for (uint64_t e = i + threadIdx.x; e < n && keys[e] == sk; e += blockDim.x) {
      const double v = big_rec(C.st.rec, spill, src[idx[e]]).v;
      if (is_dropped(v)) continue;
      const int ex = fx_exponent(v);
      emax = ex > emax ? ex : emax;
      ++live;
    }
    atomicMax(&s_emax, emax);
    atomicAdd(&s_live, live);
    __syncthreads();
    const int frac = fx128_frac_for(s_emax);
    const int nlive = s_live;
    Fx128 acc = {0, 0};
    unsigned ovf = 0;
    if (nlive > 4)
      for (uint64_t e = i + threadIdx.x; e < n && keys[e] == sk; e += blockDim.x) {
        const double v = big_rec(C.st.rec, spill, src[idx[e]]).v;
        if (is_dropped(v)) continue;
        Fx128 x = fx128_from_double(v, frac, &ovf);
        fx128_add(acc, x);
      }
    if (ovf) atomicOr(C.err, kErrAccum);
    part[threadIdx.x] = acc;
    __syncthreads();
    for (int st = 128; st; st >>= 1) {
      if ((int)threadIdx.x < st) fx128_add(part[threadIdx.x], part[threadIdx.x + st]);
      __syncthreads();
    }
    if (threadIdx.x == 0 && nlive > 0) {
      double num;
      if (nlive > 4) {
        num = fx128_to_double(part[0], frac);
      } else {  // the rare run whose values the screen dropped: the on-chip rule
        double w[4] = {0.0, 0.0, 0.0, 0.0};
        int k = 0;
        for (uint64_t e = i; e < n && keys[e] == sk && k < 4; ++e) {
          const double v = big_rec(C.st.rec, spill, src[idx[e]]).v;
          if (!is_dropped(v)) w[k++] = v;
        }
        num = nlive == 1 ? w[0]
              : nlive == 2 ? w[0] + w[1]
                           : sum4_ordered(w[0], w[1], w[2], w[3]);
      }
      const uint64_t full = pack_key(alpha[sk >> 32], (uint32_t)sk);
      big_emit(num, full, big_rec(C.st.rec, spill, src[idx[i]]).den, C, &my_unique, &my_excl);
    }
    __syncthreads();  // part[] and the shared counters are reused by the next run
  }
  if (threadIdx.x == 0) {
    if (my_unique) atomicAdd(C.n_unique, my_unique);
    if (my_excl) atomicAdd(C.n_excluded, my_excl);
  }
}

// Linear-probing insert; the table is at most 1/4 full, so a free slot is
// always found, and the probe count is bounded by the table size regardless
// (exceeding it sets *err).
__global__ void k_psi_insert(const uint64_t *keys, size_t n, uint64_t *ht, uint64_t mask,
                             unsigned *err) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t k = keys[i];
    uint64_t h = mix_key(k) & mask;
    uint64_t probe = 0;
    for (; probe <= mask; ++probe) {
      unsigned long long prev =
          atomicCAS((unsigned long long *)&ht[h], ~0ull, (unsigned long long)k);
      if (prev == ~0ull || prev == k) break;
      h = (h + 1) & mask;
    }
    if (probe > mask) atomicOr(err, kErrProbe);
  }
}

__global__ void k_abs_min(const double *s, size_t n, unsigned long long *out) {
  // min |s| as ordered bits (non-negative doubles order like their bit patterns)
  unsigned long long m = ~0ull;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    unsigned long long b = (unsigned long long)__double_as_longlong(fabs(s[i]));
    m = b < m ? b : m;
  }
  for (int dl = 16; dl; dl >>= 1) {
    unsigned long long o = __shfl_xor_sync(0xffffffffu, m, dl);
    m = o < m ? o : m;
  }
  if ((threadIdx.x & 31) == 0) atomicMin(out, m);
}

inline unsigned grid_for(size_t n, unsigned cap = 152 * 16) {
  size_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  return (unsigned)(b < cap ? b : cap);
}

}  // namespace


// ------------------------------------------------------------ host side ---

int kept_count(const uint32_t *keep, const uint32_t *pos, size_t n, size_t *host_count,
               Arena &arena);

// The four maxima that size the fixed-point grids (k_fx_bounds), to `out`
// (zeroed by the caller).
int fx_bounds(const double *h1, const double *eri, int n, unsigned long long *out, cudaStream_t s) {
  k_fx_bounds<<<(unsigned)((n * n * 32 + 255) / 256), 256, 0, s>>>(h1, eri, n, out);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

int build_fx(const double *h1, const double *eri, int n, int na, int nb, double ecore, double E0,
             const double h3[4], Arena &arena, FxInts *out, int64_t *E0_x) {
  cudaStream_t s = arena.stream();
  // B bounds |E0|, every diagonal element and every Fock-like diagonal value:
  // (na+nb) one-body terms, C(na,2)+C(nb,2) same-spin and na*nb opposite-spin
  // pair terms.  With s = 58 - log2(B) a sum of up to 32 such values cannot
  // overflow 64 bits.
  const double nn = (double)(na + nb), pairs_same = 0.5 * (na * (na - 1) + nb * (nb - 1));
  const double terms = nn * h3[0] + (pairs_same + n) * h3[1] + ((double)na * nb + n) * h3[2] + 1.0;
  const double B = fabs(ecore) + fabs(E0) + terms;
  int e = 0;
  frexp(B, &e);  // B < 2^e
  int sc = 58 - e;
  if (sc > 60) sc = 60;
  if (sc < 8) {
    record_error("integrals too large for the fixed-point diagonal", __FILE__, __LINE__);
    return ASCI_EINVAL;
  }
  int64_t *hh, *jk, *jj;
  ASCI_TRY(arena.alloc(&hh, n));
  ASCI_TRY(arena.alloc(&jk, (size_t)n * n));
  ASCI_TRY(arena.alloc(&jj, (size_t)n * n));
  k_fx_tables<<<(n * n + 255) / 256, 256, 0, s>>>(h1, eri, n, sc, hh, jk, jj);
  ASCI_CHECK_LAUNCH();
  // single excitations: a sum of at most n + 1 table values stays below the
  // bound Bs, and s1 = 61 - log2(Bs) keeps it inside 64 bits
  const double bs = h3[3];
  int e1 = 0;
  frexp(bs + 1e-300, &e1);
  int s1 = 61 - e1;
  if (s1 > 1000) s1 = 1000;
  const size_t n3 = (size_t)n * n * n;
  int64_t *h1x, *ssx, *sox;
  ASCI_TRY(arena.alloc(&h1x, (size_t)n * n));
  ASCI_TRY(arena.alloc(&ssx, n3));
  ASCI_TRY(arena.alloc(&sox, n3));
  k_fx_single_tables<<<(unsigned)std::min<size_t>((n3 + 255) / 256, 4096), 256, 0, s>>>(
      h1, eri, n, s1, h1x, ssx, sox);
  ASCI_CHECK_LAUNCH();
  // the 32-bit denominators: |E0 - H_ii| is bounded without the core energy, which
  // E0 contains as well (with it, ecore = 1e9 left so few bits that a (24e,30o) search
  // with eps = 1e-6, C = 3000, took 43 ms instead of 7.2)
  int ed = 0;
  frexp(fabs(E0 - ecore) + terms, &ed);
  FxInts X;
  X.n = n;
  X.s = sc;
  X.ds = std::max(1, ed + sc - 30);
  X.s1 = s1;
  X.h1x = h1x;
  X.ssx = ssx;
  X.sox = sox;
  X.ecore_x = llrint(ldexp(ecore, sc));
  X.hh = hh;
  X.jk = jk;
  X.jj = jj;
  // chunk tables of the diagonal: at most 8 bits a chunk, at least two chunks
  X.nc = std::max(2, (n + 7) / 8);
  X.cb = (n + X.nc - 1) / X.nc;
  const int npair = X.nc * (X.nc - 1) / 2;
  const size_t tab = (size_t)1 << (2 * X.cb);
  int64_t *xs, *xo;
  ASCI_TRY(arena.alloc(&xs, npair * tab));
  ASCI_TRY(arena.alloc(&xo, X.nc * X.nc * tab));
  k_fx_chunks<<<dim3((unsigned)((tab + 255) / 256), npair + X.nc * X.nc), 256, 0, s>>>(
      hh, jk, jj, n, X.nc, X.cb, xs, xo);
  ASCI_CHECK_LAUNCH();
  X.xs = xs;
  X.xo = xo;
  *out = X;
  *E0_x = llrint(ldexp(E0, sc));
  return ASCI_OK;
}

// The core's records, its Fock-like diagonals and the pair tables in units of
// the emission's denominator.
int core_fock(const uint32_t *core_alpha, const uint32_t *core_beta, const double *core_c, size_t m,
              FusedCore *F, Arena &arena) {
  const int n = F->X.n;
  cudaStream_t s = arena.stream();
  CoreRec *rec;
  uint32_t *Fa, *Fb, *jk, *jj;
  ASCI_TRY(arena.alloc(&rec, m));
  ASCI_TRY(arena.alloc(&Fa, m * n));
  ASCI_TRY(arena.alloc(&Fb, m * n));
  ASCI_TRY(arena.alloc(&jk, (size_t)n * n));
  ASCI_TRY(arena.alloc(&jj, (size_t)n * n));
  k_core_fock<<<dim3(grid_for(m, 152 * 4), n + 1), 256, 0, s>>>(F->X, F->E0_x, core_alpha, core_beta,
                                                               core_c, m, rec, Fa, Fb);
  ASCI_CHECK_LAUNCH();
  k_den_tables<<<(n * n + 255) / 256, 256, 0, s>>>(F->X, jk, jj);
  ASCI_CHECK_LAUNCH();
  F->core = rec;
  F->Fa = Fa;
  F->Fb = Fb;
  F->ejk = jk;
  F->ejj = jj;
  return ASCI_OK;
}

namespace {
__global__ void k_item_totals(const uint32_t *item_group, const uint64_t *Wexcl, uint64_t T,
                              uint64_t *out) {
  out[0] = item_group[T];
  out[1] = Wexcl[T];
}
}  // namespace

// Groups (distinct target alpha strings) of the sorted item list.  item_group
// has T + 1 entries; the group tables have G + 1 rows (row G: T and P).
// *P receives the total weight, read with the group count.
int item_groups(const uint64_t *items, const uint64_t *Wexcl, uint64_t T, uint32_t *item_group,
                uint32_t **g_alpha, uint64_t **g_P0, uint64_t **g_item0, size_t *G, uint64_t *P,
                Arena &arena) {
  cudaStream_t s = arena.stream();
  ASCI_TRY(scan_item_heads(items, T, item_group, arena));
  uint64_t *d_tot, tot[2] = {0, 0};
  ASCI_TRY(arena.alloc(&d_tot, 2));
  k_item_totals<<<1, 1, 0, s>>>(item_group, Wexcl, T, d_tot);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaMemcpyAsync(tot, d_tot, sizeof(tot), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  const size_t ng = (size_t)tot[0];
  ASCI_TRY(arena.alloc(g_alpha, ng + 1));
  ASCI_TRY(arena.alloc(g_P0, ng + 1));
  ASCI_TRY(arena.alloc(g_item0, ng + 1));
  k_group_tab<<<grid_for(T), 256, 0, s>>>(items, item_group, Wexcl, T, *g_alpha, *g_P0, *g_item0);
  ASCI_CHECK_LAUNCH();
  *G = ng;
  *P = tot[1];
  return ASCI_OK;
}

int psi_hash_build(const uint64_t *psi_keys, size_t nd, uint64_t **ht, uint64_t *mask,
                   unsigned *err, Arena &arena) {
  uint64_t size = 1024;
  while (size < 4 * (uint64_t)nd) size <<= 1;
  ASCI_TRY(arena.alloc(ht, size));
  cudaStream_t s = arena.stream();
  ASCI_TRY_CUDA(cudaMemsetAsync(*ht, 0xff, size * sizeof(uint64_t), s));
  k_psi_insert<<<grid_for(nd), 256, 0, s>>>(psi_keys, nd, *ht, size - 1, err);
  ASCI_CHECK_LAUNCH();
  *mask = size - 1;
  return ASCI_OK;
}


// Stage one batch (items [t0, t1), pairs [P0, P1), groups [gb0, gb1)): plan
// its tiles, count the hash buckets of big classes and emit every record into
// the staging buffer.  The tile table is left in *tiles_out (arena memory).
// Launch of an emission kernel instantiated by (eps screen, precision).
using EmitKernel = void (*)(EmitArgs);
static unsigned emit_grid(EmitKernel k, int threads, size_t smem, size_t ntl, int cap);
static void launch_emit(EmitKernel e0, EmitKernel n0, EmitKernel e1, EmitKernel n1,
                        EmitKernel e2, EmitKernel n2, bool eps, int prec, size_t work,
                        int threads, size_t smem, int cap, cudaStream_t s, const EmitArgs &A) {
  EmitKernel k = prec == 2 ? (eps ? e2 : n2) : prec == 1 ? (eps ? e1 : n1) : (eps ? e0 : n0);
  k<<<emit_grid(k, threads, smem, work, cap), threads, smem, s>>>(A);
}

// Persistent emission grid: as many CTAs as the GPU holds at once (the
// kernel's occupancy at this block size and shared memory, at most `cap` per
// SM when cap > 0), at most `ntl`.
static unsigned emit_grid(EmitKernel k, int threads, size_t smem, size_t ntl, int cap) {
  int dev = 0, sms = 152, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    sms = 152;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k, threads, smem) != cudaSuccess ||
      per < 1) {
    cudaGetLastError();
    per = 1;
  }
  if (cap > 0 && cap < per) per = cap;
  return (unsigned)std::max<size_t>(1, std::min<size_t>(ntl, (size_t)sms * per));
}

int fused_stage(const FusedCore &F, uint64_t t0, uint64_t t1, uint64_t P0, uint64_t P1,
                uint32_t gb0, uint32_t gb1, const Stage &st, double eps,
                unsigned long long *survivors, unsigned *err,
                void **tiles_out, size_t *ntiles_out, const uint64_t **psi_list_out,
                Spill *spill_out, std::vector<uint32_t> *oversized, Arena &arena) {
  cudaStream_t s = arena.stream();
  const uint32_t ng = gb1 - gb0;
  *psi_list_out = nullptr;
  *spill_out = Spill{nullptr, nullptr, 0};
  *ntiles_out = 0;
  oversized->clear();
  if (P1 <= P0 || ng == 0) return ASCI_OK;
  uint32_t *kind, *nb, *cellbase, *ntile, *tile_base;
  uint64_t *small_pairs, *Ws, *slots, *soff;
  ASCI_TRY(arena.alloc(&slots, ng));
  ASCI_TRY(arena.alloc(&soff, ng));
  ASCI_TRY(arena.alloc(&kind, ng));
  ASCI_TRY(arena.alloc(&nb, ng));
  ASCI_TRY(arena.alloc(&cellbase, ng));
  ASCI_TRY(arena.alloc(&ntile, ng));
  ASCI_TRY(arena.alloc(&tile_base, ng));
  ASCI_TRY(arena.alloc(&small_pairs, ng));
  ASCI_TRY(arena.alloc(&Ws, ng));
  k_group_class<<<grid_for(ng), 256, 0, s>>>(F.g_P0, gb0, gb1, P1, kind, nb, small_pairs,
                                             slots);
  ASCI_CHECK_LAUNCH();
  ASCI_TRACE("stage: classified %u groups", ng);
  ASCI_TRY(scan_exclusive_u64(slots, soff, ng, arena));
  ASCI_TRY(scan_exclusive_u64(small_pairs, Ws, ng, arena));
  ASCI_TRY(scan_exclusive_u32(nb, cellbase, ng, arena));
  k_tile_count<<<grid_for(ng), 256, 0, s>>>(ng, kind, nb, Ws, ntile);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(scan_exclusive_u32(ntile, tile_base, ng, arena));

  // work lists of the batch: determinant runs and alpha-double items
  const uint64_t nt = t1 - t0;
  if (nt >= (1ull << 32)) return ASCI_EINVAL;
  uint32_t *rcnt, *roff, *adf, *adpos, *adw, *adsum;
  ASCI_TRY(arena.alloc(&rcnt, nt));
  ASCI_TRY(arena.alloc(&roff, nt));
  ASCI_TRY(arena.alloc(&adf, nt));
  ASCI_TRY(arena.alloc(&adpos, nt));
  ASCI_TRY(arena.alloc(&adw, nt));
  ASCI_TRY(arena.alloc(&adsum, nt));
  const uint32_t piece = (uint32_t)std::min<uint64_t>(
      kPiecePairs, std::max<uint64_t>(kMinPiece, (P1 - P0) / (4ull * kEmitWarps) / 32 * 32));
  const uint32_t npieces =
      (uint32_t)std::max<uint64_t>(1, ((uint64_t)F.E.sb + F.E.dbb + piece - 1) / piece);
  k_batch_counts<<<grid_for(nt), 256, 0, s>>>(F.items, t0, nt, F.opbits, F.E.sa, npieces,
                                              F.grp_count, rcnt, adf, adw);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(scan_exclusive_u32(rcnt, roff, nt, arena));
  ASCI_TRY(scan_exclusive_u32(adf, adpos, nt, arena));
  ASCI_TRY(scan_exclusive_u32(adw, adsum, nt, arena));
  // every total the host needs, in one copy (one round trip for the plan)
  PlanTotals *d_tot, tot{};
  ASCI_TRY(arena.alloc(&d_tot, 1));
  k_plan_totals<<<1, 1, 0, s>>>(ng, soff, slots, cellbase, nb, tile_base, ntile, nt, roff, rcnt,
                                adpos, adf, adsum, adw, d_tot);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaMemcpyAsync(&tot, d_tot, sizeof(tot), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  if (tot.slots > st.cap) {
    record_error("staging buffer too small for the batch's hash buckets (lower max_batch_pairs)",
                 __FILE__, __LINE__);
    return ASCI_ENOMEM;
  }
  const size_t ncells = tot.cells, ntiles = tot.tiles, nruns = tot.runs, nad = tot.ad,
               ad_total = tot.ad_pairs;
  ASCI_TRACE("stage: cells=%zu tiles=%zu", ncells, ntiles);
  if (ncells > P1 - P0 || ntiles > P1 - P0) {
    record_error("inconsistent tile plan", __FILE__, __LINE__);
    return ASCI_ECUDA;
  }
  if (ad_total > P1 - P0) {
    record_error("alpha-double pairs exceed the batch", __FILE__, __LINE__);
    return ASCI_ECUDA;
  }
  uint64_t *runs;
  uint32_t *adl, *ad_off;
  ASCI_TRY(arena.alloc(&runs, nruns + 1));
  ASCI_TRY(arena.alloc(&adl, nad + 1));
  ASCI_TRY(arena.alloc(&ad_off, nad + 1));
  k_batch_lists<<<grid_for(nt), 256, 0, s>>>(F.items, t0, nt, F.opbits, F.E.sa, rcnt, roff, adpos,
                                             adsum, runs, adl, ad_off);
  ASCI_CHECK_LAUNCH();
  uint32_t ad_tiles = 0;
  uint32_t *ad_tile_item = nullptr;
  if (nad) {
    ad_tiles = (uint32_t)((ad_total + kAdTile - 1) / kAdTile);
    ASCI_TRY(arena.alloc(&ad_tile_item, (size_t)ad_tiles + 1));
    k_ad_tile_items<<<grid_for((size_t)ad_tiles + 1), 256, 0, s>>>(
        ad_off, (uint32_t)nad, (uint32_t)ad_total, ad_tiles, ad_tile_item);
    ASCI_CHECK_LAUNCH();
  }
  ASCI_TRACE("stage: runs=%zu alpha-double items=%zu pairs=%zu", nruns, nad, ad_total);

  // tiles: packed and medium classes in place; each bucket of a big class owns
  // kCap slots from its class's first slot on
  TileDesc *tiles;
  unsigned *n_over, *n_spill;
  uint32_t *over_list, *cell_tile, *fill, *spill_cell;
  const uint32_t over_cap = (uint32_t)std::min<size_t>(ncells + 1, 1u << 20);
  uint32_t spill_cap = (uint32_t)std::min<uint64_t>(
      std::max<uint64_t>(1ull << 20, (P1 - P0) / 32), 1ull << 30);
  StageRec *spill_rec;
  ASCI_TRY(arena.alloc(&tiles, ntiles + 1));
  ASCI_TRY(arena.alloc(&n_over, 3));  // overfilled cells, spilled records, psi determinants routed
  n_spill = n_over + 1;
  ASCI_TRY(arena.alloc(&over_list, over_cap));
  ASCI_TRY(arena.alloc(&cell_tile, ncells + 1));
  ASCI_TRY(arena.alloc(&fill, ncells + 1));
  ASCI_TRY(arena.alloc(&spill_rec, spill_cap));
  ASCI_TRY(arena.alloc(&spill_cell, spill_cap));
  ASCI_TRY_CUDA(cudaMemsetAsync(tiles, 0, (ntiles + 1) * sizeof(TileDesc), s));
  ASCI_TRY_CUDA(cudaMemsetAsync(n_over, 0, 3 * sizeof(unsigned), s));
  ASCI_TRY_CUDA(cudaMemsetAsync(fill, 0, (ncells + 1) * sizeof(uint32_t), s));
  k_tile_write<<<grid_for(ng), 256, 0, s>>>(gb0, ng, soff, P1, F.g_P0, F.g_alpha, kind, nb, Ws,
                                            tile_base, tiles);
  ASCI_CHECK_LAUNCH();
  if (ncells) {
    k_cell_write<<<grid_for(ncells), 256, 0, s>>>(gb0, ng, (uint32_t)ncells, soff, F.g_alpha,
                                                  tile_base, cellbase, tiles, cell_tile);
    ASCI_CHECK_LAUNCH();
  }
  ASCI_TRACE("stage: tiles written");
  // psi determinants routed to their tiles (entered there as markers)
  uint64_t *psi_list = nullptr;
  if (F.npsi) {
    uint64_t *route;
    ASCI_TRY(arena.alloc(&route, F.npsi));
    ASCI_TRY(arena.alloc(&psi_list, F.npsi));
    k_psi_route<<<grid_for(F.npsi), 256, 0, s>>>(F.psi_keys, F.npsi, F.g_alpha, gb0, ng, kind, nb,
                                                 Ws, tile_base, tiles, route);
    ASCI_CHECK_LAUNCH();
    k_psi_base<<<grid_for(F.npsi), 256, 0, s>>>(route, F.npsi, tiles, n_over + 2);
    ASCI_CHECK_LAUNCH();
    k_psi_place<<<grid_for(F.npsi), 256, 0, s>>>(route, F.psi_keys, F.npsi, tiles, psi_list);
    ASCI_CHECK_LAUNCH();
  }
  *psi_list_out = psi_list;

  EmitArgs A{};
  A.I = F.I;
  A.X = F.X;
  A.E = F.E;
  A.dv_vb = FastDiv(F.E.vb ? F.E.vb : 1);
  A.dv_pb_p = FastDiv(F.E.pb_p ? F.E.pb_p : 1);
  A.dv_pieces = FastDiv(npieces);
  A.npd0 = (uint32_t)(F.E.sb + F.E.dbb);
  A.npd1 = 1u + F.E.sb;
  A.npieces = npieces;
  A.piece = piece;
  A.run_claim = (uint32_t)std::min<uint64_t>(kRunClaim, std::max<uint64_t>(1, nruns / kEmitWarps));
  A.items = F.items;
  A.Wexcl = F.Wexcl;
  A.item_group = F.item_group;
  A.t0 = t0;
  A.opbits = F.opbits;
  A.grp_alpha = F.grp_alpha;
  A.grp_start = F.grp_start;
  A.grp_count = F.grp_count;
  A.core = static_cast<const CoreRec *>(F.core);
  A.Fa = F.Fa;
  A.Fb = F.Fb;
  A.jk = F.ejk;
  A.jj = F.ejj;
  A.gb0 = gb0;
  A.kind = kind;
  A.nb = nb;
  A.cellbase = cellbase;
  A.soff = soff;
  A.g_P0 = F.g_P0;
  A.fill = fill;
  A.spill_rec = spill_rec;
  A.spill_cell = spill_cell;
  A.n_spill = n_spill;
  A.spill_cap = spill_cap;
  A.runs = runs;
  A.nruns = nruns;
  A.adl = adl;
  A.ad_off = ad_off;
  A.nad = (uint32_t)nad;
  A.ad_total = (uint32_t)ad_total;
  A.ad_tile_item = ad_tile_item;
  A.ad_tiles = ad_tiles;
  A.st = st;
  A.st_cap = (uint32_t)std::min<uint64_t>(st.cap, 0xffffffffull);
  A.eps = eps;
  int eps_exp = 0;
  A.eps_f = (float)frexp(eps, &eps_exp);
  A.eps_shift = -eps_exp;
  A.E0_x = F.E0_x;
  A.inv_scale = ldexp(1.0, -F.X.s);
  A.scale32 = (float)ldexp(1.0, F.X.ds - F.X.s);
  A.survivors = survivors;
  A.ncore = F.ncore;
  A.err = err;
  const size_t emit_smem = 2 * (size_t)F.X.n * F.X.n * sizeof(uint32_t);
  unsigned long long *run_next;
  ASCI_TRY(arena.alloc(&run_next, 1));
  A.run_next = run_next;
  unsigned long long surv0 = 0;
  if (eps > 0.0) {
    ASCI_TRY_CUDA(cudaMemcpyAsync(&surv0, survivors, sizeof(surv0), cudaMemcpyDefault, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  }
  unsigned hov = 0, hsp = 0;
  for (int attempt = 0;; ++attempt) {
    if (nruns) {
      ASCI_TRY_CUDA(cudaMemsetAsync(run_next, 0, sizeof(unsigned long long), s));
      launch_emit(k_emit_runs<true, 0>, k_emit_runs<false, 0>, k_emit_runs<true, 1>,
                  k_emit_runs<false, 1>, k_emit_runs<true, 2>, k_emit_runs<false, 2>, eps > 0.0,
                  F.prec, (nruns + 7) / 8, kRunThreads, emit_smem, F.ctas_per_sm, s, A);
      ASCI_CHECK_LAUNCH();
    }
    if (ad_tiles) {
      launch_emit(k_emit_ad<true, 0>, k_emit_ad<false, 0>, k_emit_ad<true, 1>,
                  k_emit_ad<false, 1>, k_emit_ad<true, 2>, k_emit_ad<false, 2>, eps > 0.0,
                  F.prec, ad_tiles, kAdThreads, 0, F.ctas_per_sm, s, A);
      ASCI_CHECK_LAUNCH();
    }
    ASCI_TRACE("stage: emission launched");
    if (ncells) {
      k_cell_finish<<<grid_for(ncells), 256, 0, s>>>((uint32_t)ncells, fill, cell_tile, tiles,
                                                     n_over, over_list, over_cap);
      ASCI_CHECK_LAUNCH();
    }
    unsigned hcnt[2] = {0, 0};
    ASCI_TRY_CUDA(cudaMemcpyAsync(hcnt, n_over, sizeof(hcnt), cudaMemcpyDefault, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    hov = hcnt[0];
    hsp = hcnt[1];
    if (hsp <= spill_cap) break;
    if (attempt > 0) {
      record_error("spill list inconsistent between emissions", __FILE__, __LINE__);
      return ASCI_ECUDA;
    }
    // Hot targets overfilled their buckets beyond the spill list.  Bucket fills
    // do not depend on the order of the atomics, so the spill count is exact:
    // size the list to it and emit the batch again.
    ASCI_TRACE("stage: %u spilled records exceed the list (%u); emitting again", hsp, spill_cap);
    spill_cap = hsp;
    ASCI_TRY(arena.alloc(&spill_rec, spill_cap));
    ASCI_TRY(arena.alloc(&spill_cell, spill_cap));
    A.spill_rec = spill_rec;
    A.spill_cell = spill_cell;
    A.spill_cap = spill_cap;
    ASCI_TRY_CUDA(cudaMemsetAsync(n_over, 0, 2 * sizeof(unsigned), s));
    ASCI_TRY_CUDA(cudaMemsetAsync(fill, 0, (ncells + 1) * sizeof(uint32_t), s));
    if (eps > 0.0)
      ASCI_TRY_CUDA(cudaMemcpyAsync(survivors, &surv0, sizeof(surv0), cudaMemcpyDefault, s));
  }
  if (hov > over_cap) {
    record_error("too many oversized hash buckets", __FILE__, __LINE__);
    return ASCI_ENOMEM;
  }
  if (hsp) {  // spilled records in tile order
    uint64_t *sk, *sk_alt;
    ASCI_TRY(arena.alloc(&sk, hsp));
    ASCI_TRY(arena.alloc(&sk_alt, hsp));
    k_spill_keys<<<grid_for(hsp), 256, 0, s>>>(spill_cell, cell_tile, hsp, sk);
    ASCI_CHECK_LAUNCH();
    int topbit = 1;
    while ((1ull << topbit) <= (uint64_t)ntiles) ++topbit;
    ASCI_TRY(radix_sort_u64(&sk, &sk_alt, hsp, 0, 32 + topbit, arena));
    *spill_out = Spill{spill_rec, sk, hsp};
  }
  ASCI_TRACE("stage: oversized buckets=%u spilled records=%u", hov, hsp);
  if (hov) {
    oversized->resize(hov);
    ASCI_TRY_CUDA(cudaMemcpyAsync(oversized->data(), over_list, hov * sizeof(uint32_t),
                                  cudaMemcpyDefault, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    std::sort(oversized->begin(), oversized->end());
  }
  *tiles_out = tiles;
  *ntiles_out = ntiles;
  return ASCI_OK;
}

size_t tile_capacity() { return (size_t)kCap; }
size_t big_tile_capacity() { return (size_t)kBigCap; }

static CellArgs cell_args(const FusedCore &F, const Stage &st,
                          double tau, uint64_t *cand_key, double *cand_score,
                          unsigned long long *cand_count, unsigned long long cand_cap,
                          unsigned long long *n_unique, unsigned long long *n_excluded,
                          unsigned *err) {
  CellArgs CA;
  memset(&CA, 0, sizeof(CA));
  CA.st = st;
  CA.tau = tau;
  CA.tau_f = (float)tau;
  if ((double)CA.tau_f > tau) CA.tau_f = nextafterf(CA.tau_f, 0.0f);
  CA.psi_ht = F.psi_ht;
  CA.psi_mask = F.psi_mask;
  CA.cand_key = cand_key;
  CA.cand_score = cand_score;
  CA.cand_count = cand_count;
  CA.cand_cap = cand_cap;
  CA.n_unique = n_unique;
  CA.n_excluded = n_excluded;
  CA.err = err;
  CA.screened = F.screened;
  return CA;
}

// Buffers of the targets that the tile kernels leave to k_long_sums, in a
// scratch arena that outlives the launch and the fix-up that follows it.  With
// a threshold few targets of several records can reach it, most where targets
// collect many records (at most 6 a tile with 75 values at (24e,30o), C = 1e5;
// 25 with 300 at (16e,16o), C = 1e4): the buffers hold 48 and 512 per kCap
// records of capacity, 4.9 KB against the 16 KB of the records.  (16 and 80
// made those two searches run their first launches twice: 209 ms against 199,
// 6.3 against 5.6.)  `full` gives room for every record (no threshold, as in
// ASCI-PT2 and the first batch, where every such target is summed); a launch
// whose buffers were too small sets kErrValues and is run again so.
static int enable_long_sums(CellArgs &CA, size_t tiles, bool full, Arena &la) {
  const unsigned long long t = tiles, all_fix = t * (kCap / 2), all_lv = t * kCap;
  const unsigned long long fix_cap =
      full ? all_fix : std::max(t * 48, std::min(all_fix, 1ull << 16));
  const unsigned long long lv_cap = std::min<unsigned long long>(
      full ? all_lv : std::max(t * 512, std::min(all_lv, 1ull << 18)), 0xffffffffull);
  unsigned long long *cnt;
  ASCI_TRY(la.alloc(&CA.lv, (size_t)lv_cap));
  ASCI_TRY(la.alloc(&CA.fix, (size_t)fix_cap));
  ASCI_TRY(la.alloc(&cnt, 2));
  ASCI_TRY_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), la.stream()));
  CA.lv_count = cnt;
  CA.nfix = cnt + 1;
  CA.lv_cap = lv_cap;
  CA.fix_cap = fix_cap;
  return ASCI_OK;
}

static int run_long_sums(const CellArgs &CA, int sms, cudaStream_t s) {
  k_long_sums<<<(unsigned)sms * 8, 256, 0, s>>>(CA.fix, CA.nfix, CA.fix_cap, CA.lv, CA.cand_score,
                                                 CA.err);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

// Tiles per launch when every record has room in the buffers of k_long_sums
// (16 KB a tile): a quarter of the batch, between 128 MB and 2 GB of buffers.
size_t full_tiles(size_t ntiles) {
  return std::min<size_t>(std::max<size_t>(ntiles / 4, 8192), 131072);
}

// Reduce tiles [tile_begin, tile_end) of a staged batch on chip and append the
// targets with |S| >= tau to the candidate buffer (at most kCap per tile).
int fused_cells(const FusedCore &F, const void *tiles, const uint64_t *psi_list,
                uint32_t tile_begin, uint32_t tile_end, const Stage &st, double tau,
                uint64_t *cand_key, double *cand_score,
                unsigned long long *cand_count, unsigned long long cand_cap,
                unsigned long long *n_unique, unsigned long long *n_excluded, unsigned *err,
                bool full, Arena &arena) {
  if (tile_end <= tile_begin) return ASCI_OK;
  cudaStream_t s = arena.stream();
  CellArgs CA = cell_args(F, st, tau, cand_key, cand_score, cand_count, cand_cap, n_unique,
                          n_excluded, err);
  CA.tiles = static_cast<const TileDesc *>(tiles);
  CA.psi_list = psi_list;
  CA.tile0 = tile_begin;
  CA.ntiles = tile_end;
  const size_t cell_smem = sizeof(CellSmem<kCap>);
  // once (thread-safe static initialisation): attribute and occupancy
  static const int per_sm = [cell_smem]() {
    int p = 0;
    if (cudaFuncSetAttribute(k_cells<kCap, kCellThreads, kCellCtas>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)cell_smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &p, k_cells<kCap, kCellThreads, kCellCtas>, kCellThreads, cell_smem) !=
            cudaSuccess)
      return 0;
    return p < 1 ? 1 : p;
  }();
  if (!per_sm) {
    record_error("tile kernel: cannot set its shared memory size", __FILE__, __LINE__);
    return ASCI_ECUDA;
  }
  int dev = 0, sms = 152;
  ASCI_TRY_CUDA(cudaGetDevice(&dev));
  ASCI_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int per = (F.ctas_per_sm > 0 && F.ctas_per_sm < per_sm) ? F.ctas_per_sm : per_sm;
  const unsigned grid = (unsigned)std::min<size_t>((size_t)sms * per, tile_end - tile_begin);
  ASCI_TRACE("cells: launch grid=%u smem=%zu per_sm=%d", grid, cell_smem, per_sm);
  Arena la(s);
  ASCI_TRY(enable_long_sums(CA, tile_end - tile_begin, full, la));
  k_cells<kCap, kCellThreads, kCellCtas><<<grid, kCellThreads, cell_smem, s>>>(CA);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(run_long_sums(CA, sms, s));
  return ASCI_OK;
}

// Per listed tile (start, in-place records, target alpha, first spill entry,
// spilled records): one gather kernel and one copy back.
int tile_info(const void *tiles, const std::vector<uint32_t> &list, const Spill &spill,
              std::vector<uint32_t> *info, cudaStream_t s) {
  const size_t n = list.size();
  info->assign(5 * n, 0u);
  if (!n) return ASCI_OK;
  Arena ta(s);
  uint32_t *d_list, *d_info;
  ASCI_TRY(ta.alloc(&d_list, n));
  ASCI_TRY(ta.alloc(&d_info, 5 * n));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_list, list.data(), n * 4, cudaMemcpyDefault, s));
  k_tile_gather<<<grid_for(n), 256, 0, s>>>(static_cast<const TileDesc *>(tiles), d_list,
                                            (uint32_t)n, spill.keys, spill.n, d_info);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaMemcpyAsync(info->data(), d_info, 5 * n * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  return ASCI_OK;
}

// Launch the tile kernel of one size over tiles [t0, t1) of CA.tiles.
template <int CAP, int THREADS, int CTAS>
static int launch_big_cells(CellArgs CA, uint32_t t0, uint32_t t1, int sms, cudaStream_t s) {
  if (t1 <= t0) return ASCI_OK;
  const size_t smem = sizeof(CellSmem<CAP>);
  static const int per_sm = [smem]() {
    int p = 0;
    if (cudaFuncSetAttribute(k_cells<CAP, THREADS, CTAS>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, k_cells<CAP, THREADS, CTAS>, THREADS,
                                                      smem) != cudaSuccess)
      return 0;
    return p < 1 ? 1 : p;
  }();
  if (!per_sm) {
    record_error("large tile kernel: cannot set its shared memory size", __FILE__, __LINE__);
    return ASCI_ECUDA;
  }
  CA.tile0 = t0;
  CA.ntiles = t1;
  const unsigned grid = (unsigned)std::min<size_t>((size_t)sms * per_sm, t1 - t0);
  k_cells<CAP, THREADS, CTAS><<<grid, THREADS, smem, s>>>(CA);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

// Reduce oversized bucket tiles of at most kBigCap records on chip: list[i]
// is a tile of the batch and info[5i..5i+4] its row from tile_info.  Tiles of
// at most kMidCap records go to the middle-size kernel, the rest to the
// kBigCap one.  Appends at most as many candidates as there are records
// (*nrec_out).
int fused_big_cells(const FusedCore &F, const void *tiles, const uint64_t *psi_list,
                    const uint32_t *list_in, const uint32_t *info_in, size_t nt,
                    const Stage &st, const Spill &spill, double tau, uint64_t *cand_key,
                    double *cand_score, unsigned long long *cand_count,
                    unsigned long long cand_cap, unsigned long long *n_unique,
                    unsigned long long *n_excluded, unsigned *err, bool full, uint64_t *nrec_out,
                    Arena &arena) {
  cudaStream_t s = arena.stream();
  *nrec_out = 0;
  if (!nt) return ASCI_OK;
  // middle-size tiles first
  std::vector<uint32_t> list(nt), info(5 * nt), off(nt);
  size_t nmid = 0;
  for (size_t i = 0; i < nt; ++i) {
    const uint32_t *r = info_in + 5 * i;
    if ((uint64_t)r[1] + r[4] <= (uint64_t)kMidCap) ++nmid;
  }
  {
    size_t a = 0, b = nmid;
    for (size_t i = 0; i < nt; ++i) {
      const uint32_t *r = info_in + 5 * i;
      const size_t j = ((uint64_t)r[1] + r[4] <= (uint64_t)kMidCap) ? a++ : b++;
      list[j] = list_in[i];
      for (int w = 0; w < 5; ++w) info[5 * j + w] = r[w];
    }
  }
  uint64_t total = 0;
  for (size_t i = 0; i < nt; ++i) {
    const uint32_t *r = info.data() + 5 * i;
    const uint64_t nrec = (uint64_t)r[1] + r[4];
    if (nrec > (uint64_t)kBigCap || (uint64_t)r[0] + r[1] > st.cap ||
        (uint64_t)r[3] + r[4] > spill.n)
      return ASCI_ECUDA;
    off[i] = (uint32_t)total;
    total += nrec;
  }
  if (total >= (1ull << 32)) return ASCI_ENOMEM;
  *nrec_out = total;
  Arena ta(s);
  uint32_t *d_list, *d_info, *d_off;
  StageRec *big;
  TileDesc *desc;
  ASCI_TRY(ta.alloc(&d_list, nt));
  ASCI_TRY(ta.alloc(&d_info, 5 * nt));
  ASCI_TRY(ta.alloc(&d_off, nt));
  ASCI_TRY(ta.alloc(&big, total));
  ASCI_TRY(ta.alloc(&desc, nt));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_list, list.data(), nt * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_info, info.data(), 5 * nt * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_off, off.data(), nt * 4, cudaMemcpyDefault, s));
  k_big_tile_gather<<<(unsigned)nt, 256, 0, s>>>(static_cast<const TileDesc *>(tiles), d_list,
                                                 d_info, d_off, st.rec, spill.rec, spill.keys,
                                                 big, desc);
  ASCI_CHECK_LAUNCH();
  CellArgs CA = cell_args(F, Stage{big, nullptr, total}, tau, cand_key, cand_score, cand_count,
                          cand_cap, n_unique, n_excluded, err);
  CA.tiles = desc;
  CA.psi_list = psi_list;
  int dev = 0, sms = 152;
  ASCI_TRY_CUDA(cudaGetDevice(&dev));
  ASCI_TRY_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  ASCI_TRY(enable_long_sums(CA, nt * (kBigCap / kCap), full, ta));
  ASCI_TRY((launch_big_cells<kMidCap, kMidThreads, 4>(CA, 0, (uint32_t)nmid, sms, s)));
  ASCI_TRY((launch_big_cells<kBigCap, kBigThreads, 2>(CA, (uint32_t)nmid, (uint32_t)nt, sms, s)));
  ASCI_TRY(run_long_sums(CA, sms, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));  // the host vectors above are read by copies
  return ASCI_OK;
}

// Reduce the oversized bucket tiles described by info[5i..5i+4], i in
// [0, nt), at once: their records are gathered under keys (position << 32 |
// beta'), radix-sorted in global memory and reduced one target per thread.
// Appends at most as many candidates as there are records.
int fused_big_tiles(const FusedCore &F, const uint32_t *info, size_t nt, const Stage &st,
                    const Spill &spill, double tau, uint64_t *cand_key, double *cand_score,
                    unsigned long long *cand_count, unsigned long long cand_cap,
                    unsigned long long *n_unique, unsigned long long *n_excluded, unsigned *err,
                    uint64_t *nrec_out, Arena &arena) {
  cudaStream_t s = arena.stream();
  *nrec_out = 0;
  if (!nt) return ASCI_OK;
  std::vector<uint32_t> start(nt), nin(nt), slo(nt), off(nt + 1), alpha(nt);
  uint64_t total = 0;
  for (size_t i = 0; i < nt; ++i) {
    const uint32_t *r = info + 5 * i;
    if ((uint64_t)r[0] + r[1] > st.cap || (uint64_t)r[3] + r[4] > spill.n) return ASCI_ECUDA;
    start[i] = r[0];
    nin[i] = r[1];
    alpha[i] = r[2];
    slo[i] = r[3];
    off[i] = (uint32_t)total;
    total += (uint64_t)r[1] + r[4];
  }
  if (total >= (1ull << 32)) return ASCI_ENOMEM;
  off[nt] = (uint32_t)total;
  *nrec_out = total;
  Arena ta(s);
  uint32_t *d_start, *d_nin, *d_slo, *d_off, *d_alpha, *i0, *i1;
  uint64_t *k0, *k1, *src;
  ASCI_TRY(ta.alloc(&d_start, nt));
  ASCI_TRY(ta.alloc(&d_nin, nt));
  ASCI_TRY(ta.alloc(&d_slo, nt));
  ASCI_TRY(ta.alloc(&d_off, nt + 1));
  ASCI_TRY(ta.alloc(&d_alpha, nt));
  ASCI_TRY(ta.alloc(&k0, total));
  ASCI_TRY(ta.alloc(&k1, total));
  ASCI_TRY(ta.alloc(&i0, total));
  ASCI_TRY(ta.alloc(&i1, total));
  ASCI_TRY(ta.alloc(&src, total));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_start, start.data(), nt * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_nin, nin.data(), nt * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_slo, slo.data(), nt * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_off, off.data(), (nt + 1) * 4, cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(d_alpha, alpha.data(), nt * 4, cudaMemcpyDefault, s));
  k_big_gather<<<grid_for(total), 256, 0, s>>>(st.rec, spill.rec, spill.keys, d_start, d_nin,
                                               d_slo, d_off, (uint32_t)nt, total, k0, i0, src);
  ASCI_CHECK_LAUNCH();
  int topbit = 0;
  while ((1ull << topbit) < (uint64_t)nt) ++topbit;
  ASCI_TRY(radix_sort_u64_u32(&k0, &k1, &i0, &i1, total, 0, 32 + topbit, ta));
  CellArgs CA = cell_args(F, st, tau, cand_key, cand_score, cand_count, cand_cap, n_unique,
                          n_excluded, err);
  uint64_t *long_runs;
  unsigned *n_long;
  ASCI_TRY(ta.alloc(&long_runs, total / kLongRun + 1));
  ASCI_TRY(ta.alloc(&n_long, 1));
  ASCI_TRY_CUDA(cudaMemsetAsync(n_long, 0, sizeof(unsigned), s));
  k_big_reduce<<<grid_for(total), 256, 0, s>>>(k0, i0, src, total, d_alpha, spill.rec, CA,
                                               long_runs, n_long);
  ASCI_CHECK_LAUNCH();
  k_big_reduce_long<<<152 * 2, 256, 0, s>>>(k0, i0, src, total, d_alpha, spill.rec, CA,
                                            long_runs, n_long);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));  // the host vectors above are read by the copies
  return ASCI_OK;
}

namespace {


// ASCI-PT2 terms num^2 / (E0 - H_ii) of appended candidates (Alg. 1, last
// step), summed without rounding in a fixed-point grid of 2^-216 held as eight
// signed 32-bit limbs in 64-bit counters (a term of magnitude below 2^40 spans
// at most three limbs; bits below the grid are truncated).  Integer addition
// is exact and associative, so the sum does not depend on the order of the
// terms, on the batches or on the tiles: the result is a function of the set
// of targets.  Per-thread limb sums in shared memory are reduced over the
// block, then added to the counters with one atomic per limb and block; a
// launch holds fewer than 2^31 terms, so no counter overflows.
constexpr int kPt2Limbs = 8;
constexpr int kPt2Grid = 216;  // the grid is 2^-216

__device__ __forceinline__ void pt2_add(double t, long long (*acc)[256], unsigned *bad) {
  if (t == 0.0) return;
  if (!(fabs(t) < 0x1p40)) {  // also catches NaN and infinities
    *bad = 1u;
    return;
  }
  const unsigned long long b = (unsigned long long)__double_as_longlong(t);
  const int e = (int)((b >> 52) & 0x7ffu);
  unsigned long long m = (b & 0xfffffffffffffull) | (e ? (1ull << 52) : 0ull);
  int p = (e ? e : 1) - 1075 + kPt2Grid;  // grid position of m's lowest bit
  if (p < 0) {
    if (p <= -64) return;
    m >>= -p;
    p = 0;
  }
  const int k0 = p >> 5, o = p & 31;
  const unsigned long long lo = m << o;
  const unsigned long long hi = o ? (m >> (64 - o)) : 0ull;
  const long long sg = t < 0.0 ? -1 : 1;
  // |t| < 2^40: k0 + 2 is at most the last limb, or hi is zero
  acc[k0][threadIdx.x] += sg * (long long)(lo & 0xffffffffull);
  if (k0 + 1 < kPt2Limbs) acc[k0 + 1][threadIdx.x] += sg * (long long)(lo >> 32);
  if (k0 + 2 < kPt2Limbs) acc[k0 + 2][threadIdx.x] += sg * (long long)hi;
}

// The exact fixed-point H_ii of a target from the chunk tables of FxInts
// (equal bit for bit to fx_diag: integer sums): 28 loads at 25 to 32 orbitals,
// 15 at 17 to 24 and 6 below, against some 300 terms at (24e,30o).  The
// tables (12 MB at 30 orbitals, built in a few microseconds) stay in L2, and
// the rows that the targets of one alpha string share in L1.  Before, the
// terms were added one by one, the alpha part once per alpha string of a warp:
// ASCI-PT2 of 4000 determinants at (24e,30o) took 47.0 ms against 21.0, a
// (24e,30o) search 223.4 against 214.8.
template <int NC>
__device__ __forceinline__ int64_t table_diag(const FxInts &X, uint32_t A, uint32_t B) {
  const int cb = X.cb;
  const uint32_t mask = (1u << cb) - 1u;
  uint32_t a[NC], b[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    a[k] = (A >> (k * cb)) & mask;
    b[k] = (B >> (k * cb)) & mask;
  }
  int64_t s = X.ecore_x;
  uint32_t t = 0;
#pragma unroll
  for (int k = 0; k < NC; ++k)
#pragma unroll
    for (int l = k + 1; l < NC; ++l, t += 1u << (2 * cb))
      s += __ldg(X.xs + (t | (a[k] << cb) | a[l])) + __ldg(X.xs + (t | (b[k] << cb) | b[l]));
  t = 0;
#pragma unroll
  for (int k = 0; k < NC; ++k)
#pragma unroll
    for (int l = 0; l < NC; ++l, t += 1u << (2 * cb)) s += __ldg(X.xo + (t | (a[k] << cb) | b[l]));
  return s;
}

// Exact scores of appended candidates, which hold their numerator:
// S = num / (E0 - H_ii), with H_ii summed in fixed point (exact) and E0 - H_ii
// rounded once to a double.
template <int NC>
__global__ void __launch_bounds__(256) k_exact_scores(const uint64_t *key, double *score, size_t n,
                                                      FxInts X, int64_t E0_x, double inv_scale) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t k = key[i];
    const int64_t dg = table_diag<NC>(X, key_alpha(k), (uint32_t)(k >> 32));
    score[i] = score[i] / (__ll2double_rn(E0_x - dg) * inv_scale);
  }
}

template <int NC>
__global__ void __launch_bounds__(256) k_pt2_terms(const uint64_t *key, const double *num,
                                                   size_t n, FxInts X, int64_t E0_x,
                                                   double inv_scale, long long *limbs,
                                                   unsigned long long *count,
                                                   unsigned long long left, unsigned *err) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *count = left;  // these candidates are dropped
  // limb sums of each thread, thread-contiguous so that any limbs are free of
  // bank conflicts
  __shared__ long long acc[kPt2Limbs][256];
  for (int k = 0; k < kPt2Limbs; ++k) acc[k][threadIdx.x] = 0;
  unsigned bad = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t k = key[i];
    const double v = num[i];
    const int64_t dg = table_diag<NC>(X, key_alpha(k), (uint32_t)(k >> 32));
    const double den = __ll2double_rn(E0_x - dg) * inv_scale;
    const double r = (fabs(den) >= 1e-30 && fabs(den) <= 1e30) ? recip_fast(den) : 1.0 / den;
    pt2_add(v * v * r, acc, &bad);
  }
  if (bad) atomicOr(err, kErrTerm);
  __syncthreads();
  const int k = threadIdx.x >> 5;  // a warp per limb
  long long t = 0;
  for (int j = threadIdx.x & 31; j < 256; j += 32) t += acc[k][j];
  for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0 && t)
    atomicAdd((unsigned long long *)&limbs[k], (unsigned long long)t);
}

// The counters as one double: the limbs in a fixed order, low to high.
__global__ void k_pt2_value(const long long *limbs, double *out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double x = 0.0;
  for (int k = 0; k < kPt2Limbs; ++k) x += ldexp((double)limbs[k], 32 * k - kPt2Grid);
  *out = x;
}

}  // namespace

// Adds the terms of n candidates and sets *count to the `left` that stay.
int pt2_terms(const FusedCore &F, const uint64_t *key, const double *num, size_t n,
              long long *limbs, unsigned long long *count, unsigned long long left, unsigned *err,
              cudaStream_t s) {
  if (!n) return ASCI_OK;
  auto *k = F.X.nc == 2 ? k_pt2_terms<2> : (F.X.nc == 3 ? k_pt2_terms<3> : k_pt2_terms<4>);
  k<<<grid_for(n, 152 * 8), 256, 0, s>>>(key, num, n, F.X, F.E0_x, ldexp(1.0, -F.X.s), limbs, count,
                                         left, err);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

int pt2_value(const long long *limbs, double *out, cudaStream_t s) {
  k_pt2_value<<<1, 32, 0, s>>>(limbs, out);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

int exact_scores(const FusedCore &F, const uint64_t *key, double *score, size_t n,
                 cudaStream_t s) {
  if (!n) return ASCI_OK;
  auto *k = F.X.nc == 2 ? k_exact_scores<2>
                        : (F.X.nc == 3 ? k_exact_scores<3> : k_exact_scores<4>);
  k<<<grid_for(n, 152 * 32), 256, 0, s>>>(key, score, n, F.X, F.E0_x, ldexp(1.0, -F.X.s));
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

// Smallest |score| among n candidates (host result), used as the threshold.
int abs_min(const double *s, size_t n, double *host_min, Arena &arena) {
  unsigned long long *d;
  ASCI_TRY(arena.alloc(&d, 1));
  cudaStream_t st = arena.stream();
  ASCI_TRY_CUDA(cudaMemsetAsync(d, 0xff, sizeof(unsigned long long), st));
  k_abs_min<<<grid_for(n), 256, 0, st>>>(s, n, d);
  ASCI_CHECK_LAUNCH();
  unsigned long long h = 0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDefault, st));
  ASCI_TRY_CUDA(cudaStreamSynchronize(st));
  double v;
  memcpy(&v, &h, sizeof(v));
  *host_min = v;
  return ASCI_OK;
}

}  // namespace asci
