// The variational step of the ASCI loop (Algorithm 1, "diagonalize the
// Hamiltonian in the selected determinant space"; Sec. 2.3).
//
//  * H over a determinant list (Sec. 2.3, CSR): the paper's double loop over
//    determinant pairs, pruned by the structure of the keys.  In key order
//    (beta word high) each beta string's determinants are one group; a row
//    visits the groups whose beta string is within one excitation (a group
//    graph built by a tiled double loop over the beta strings), where it tests
//    the alpha distance against 4 - popc(beta_i ^ beta_j), and, merged with
//    them, the determinants of its own alpha string a beta double away (listed, or
//    searched where they are fewer than the alpha string's).
//    Connected pairs get H_ij by the Slater-Condon rules, evaluated 32 at a
//    time from a per-warp queue; nonzero elements are stored, each row's
//    columns ascending.  A counting pass and a scan give the row pointers, the
//    filling pass the elements; rows in the caller's order come from one sort
//    of the key-ordered entries.
//  * y = H x (Algorithm 6 on one device): a warp per row, lanes strided over
//    the row, a fixed shuffle tree: the same bits on every call.
//  * Davidson (Algorithm 5): basis V and products W = H V resident on the
//    device, the subspace matrix V^T H V grown one column per product, its
//    lowest eigenpairs by FP32 Jacobi refined in FP64 in one CTA, the shifted
//    Jacobi preconditioner, two passes of classical Gram-Schmidt, a thick
//    restart (the four lowest Ritz vectors) at the subspace limit.  Every
//    reduction has a fixed order.
//  * The ASCI loop itself: search, merge, build, diagonalise, repeat.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "asci_internal.cuh"

namespace asci {
namespace {

constexpr int kRowThreads = 256;   // rows per CTA of the build
constexpr int kColStage = 2048;    // column keys staged in shared memory at a time
constexpr int kMaxSub = 32;        // largest Davidson subspace (shared-memory Jacobi)
constexpr int kDotBlocks = 296;    // fixed partial-sum grid of the dot products
constexpr int kKeep = 4;           // Ritz vectors kept by a Davidson restart
constexpr int kDotThreads = 256;

inline unsigned blocks_for(size_t n, unsigned threads, unsigned cap = 152 * 16) {
  size_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  return (unsigned)(b < cap ? b : cap);
}

// ------------------------------ validation ---------------------------------

enum : uint32_t { kBadRange = 1u, kBadCount = 2u, kDuplicate = 4u, kBadValue = 8u };

__global__ void k_det_keys(const asci_det *dets, size_t n, int norb, int na, int nb,
                           uint64_t *keys, unsigned *err) {
  const uint64_t hi = ~((1ull << norb) - 1ull);
  unsigned e = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const asci_det d = dets[i];
    if ((d.alpha & hi) || (d.beta & hi)) e |= kBadRange;
    if (__popcll(d.alpha) != na || __popcll(d.beta) != nb) e |= kBadCount;
    keys[i] = pack_key((uint32_t)d.alpha, (uint32_t)d.beta);
  }
  if (e) atomicOr(err, e);
}

__global__ void k_adjacent_equal(const uint64_t *sorted, size_t n, unsigned *err) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x + 1; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (sorted[i] == sorted[i - 1]) atomicOr(err, kDuplicate);
}

__global__ void k_finite(const double *x, size_t n, unsigned *err) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (!isfinite(x[i])) atomicOr(err, kBadValue);
}

__global__ void k_keys_to_dets(const uint64_t *keys, size_t n, asci_det *out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    asci_det d;
    d.alpha = key_alpha(keys[i]);
    d.beta = key_beta(keys[i]);
    out[i] = d;
  }
}

// ------------------------------ the build ----------------------------------

// <D_i|H|D_j> for distinct determinants within two excitations: the holes are
// the ket's orbitals missing from the bra, the particles the bra's orbitals
// missing from the ket, ascending.
__device__ double offdiag_element(const DevInts &I, uint32_t ai, uint32_t bi, uint32_t aj,
                                  uint32_t bj) {
  const uint32_t xa = ai ^ aj, xb = bi ^ bj;
  const int da = __popc(xa), db = __popc(xb);
  if (db == 0 && da == 2) {
    const int h = __ffs(aj & xa) - 1, p = __ffs(ai & xa) - 1;
    const double v = single_value(I, aj, bj, h, p);
    return single_parity(aj, h, p) ? -v : v;
  }
  if (da == 0 && db == 2) {
    const int h = __ffs(bj & xb) - 1, p = __ffs(bi & xb) - 1;
    const double v = single_value(I, bj, aj, h, p);
    return single_parity(bj, h, p) ? -v : v;
  }
  if (da == 2) {  // opposite-spin double
    const int ha = __ffs(aj & xa) - 1, pa = __ffs(ai & xa) - 1;
    const int hb = __ffs(bj & xb) - 1, pb = __ffs(bi & xb) - 1;
    const double v = eri4(I.eri, I.n, ha, pa, hb, pb);
    return (single_parity(aj, ha, pa) ^ single_parity(bj, hb, pb)) ? -v : v;
  }
  // same-spin double (da == 4 or db == 4)
  const uint32_t ket = da ? aj : bj, x = da ? xa : xb, bra = da ? ai : bi;
  uint32_t hm = ket & x, pm = bra & x;
  const int h1 = __ffs(hm) - 1;
  hm &= hm - 1;
  const int h2 = __ffs(hm) - 1;
  const int p1 = __ffs(pm) - 1;
  pm &= pm - 1;
  const int p2 = __ffs(pm) - 1;
  const double v = eri4(I.asym, I.n, h1, p1, h2, p2);
  return double_parity(ket, h1, h2, p1, p2) ? -v : v;
}

// The build works on determinants in key order (beta word high), so that
// every beta string's determinants form one contiguous group.  Two
// determinants are within two excitations iff
//   popc(alpha_i ^ alpha_j) + popc(beta_i ^ beta_j) <= 4,
// so a row has to visit the groups whose beta string is equal or a single
// excitation away (the group graph, built once per list by a tiled double loop
// over the G group strings), where only the alpha test remains, and the
// determinants of its own alpha string whose beta string is a double away: from
// the list in alpha order, or, where an alpha string has many determinants,
// searched in the groups a double away (mates_are_fewer).  A warp takes a row and
// walks both, merged in ascending order, 32 columns at a time; a ballot places the
// hits, so each row's columns come out ascending.  A counting pass gives the row lengths, a scan the row
// pointers, and the filling pass writes (never past a row's counted end).

// head[i] = 1 where a new beta string starts (keys sorted)
__global__ void k_beta_heads(const uint64_t *keys, uint32_t n, uint32_t *head) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    head[i] = (i == 0 || key_beta(keys[i]) != key_beta(keys[i - 1])) ? 1u : 0u;
}

// group of each row; start and beta string of each group (gid: exclusive scan of head)
__global__ void k_beta_groups(const uint64_t *keys, uint32_t n, const uint32_t *head,
                              const uint32_t *gid, uint32_t *of_row, uint32_t *gstart,
                              uint32_t *gbeta) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t g = gid[i] + head[i] - 1u;
    of_row[i] = g;
    if (head[i]) {
      gstart[g] = i;
      gbeta[g] = key_beta(keys[i]);
    }
    if (i == n - 1) gstart[g + 1] = n;  // end of the last group
  }
}

// Group graph: count (kFill false) or list (kFill true) the groups g2 with
// popc(beta_g1 ^ beta_g2) <= reach, for the groups g1 = [blockIdx.x * 256, +256)
// (one per thread) against the groups [blockIdx.y * chunk, +chunk) staged in
// shared memory.
template <bool kFill>
__global__ void __launch_bounds__(kRowThreads) k_beta_pairs(const uint32_t *gbeta, uint32_t G,
                                                            uint32_t chunk, uint32_t nchunks,
                                                            int reach, uint64_t *cnt_off,
                                                            uint32_t *nbr) {
  __shared__ uint32_t sb[kColStage];
  const uint32_t g1 = blockIdx.x * kRowThreads + threadIdx.x;
  const bool live = g1 < G;
  const uint32_t b1 = live ? gbeta[g1] : 0u;
  const uint32_t c0 = blockIdx.y * chunk;
  const uint32_t c1 = min(G, c0 + chunk);
  const size_t slot = (size_t)g1 * nchunks + blockIdx.y;
  uint64_t cnt = 0, pos = 0, end = 0;
  if (kFill && live) {
    pos = cnt_off[slot];
    end = cnt_off[slot + 1];
  }
  for (uint32_t s = c0; s < c1; s += kColStage) {
    const uint32_t m = min((uint32_t)kColStage, c1 - s);
    __syncthreads();
    for (uint32_t t = threadIdx.x; t < m; t += kRowThreads) sb[t] = gbeta[s + t];
    __syncthreads();
    if (!live) continue;
#pragma unroll 4
    for (uint32_t t = 0; t < m; ++t) {
      if (__popc(b1 ^ sb[t]) > reach) continue;
      if (kFill) {
        if (pos < end) nbr[pos] = s + t;
        ++pos;
      } else {
        ++cnt;
      }
    }
  }
  if (!kFill && live) cnt_off[slot] = cnt;
}

// Rows in alpha order: akey = alpha << 32 | row, to be sorted by alpha (stably,
// so rows of one alpha string stay in ascending order).
__global__ void k_alpha_keys(const uint64_t *keys, uint32_t n, uint64_t *akey) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    akey[i] = ((uint64_t)key_alpha(keys[i]) << 32) | i;
}
// mates[t] = (row, its beta string) in alpha order; span[row] = the row's
// [first, end) there, the rows of its own alpha string.  out (zero before): their
// number over all rows, and the groups.
__global__ void k_alpha_mates(const uint64_t *keys, const uint64_t *akey, uint32_t n,
                              const uint32_t *head, const uint32_t *gid, uint2 *mates, uint2 *span,
                              unsigned long long *out) {
  unsigned long long all = 0;
  for (uint32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const uint32_t r = (uint32_t)akey[t], a = (uint32_t)(akey[t] >> 32);
    mates[t] = make_uint2(r, key_beta(keys[r]));
    uint32_t lo = 0, hi = t;  // first position of alpha a
    while (lo < hi) {
      const uint32_t mid = lo + ((hi - lo) >> 1);
      if ((uint32_t)(akey[mid] >> 32) < a) lo = mid + 1;
      else hi = mid;
    }
    uint32_t lo2 = t, hi2 = n;  // first position past alpha a
    while (lo2 < hi2) {
      const uint32_t mid = lo2 + ((hi2 - lo2) >> 1);
      if ((uint32_t)(akey[mid] >> 32) <= a) lo2 = mid + 1;
      else hi2 = mid;
    }
    span[r] = make_uint2(lo, lo2);
    all += lo2 - lo;
    if (t == n - 1) out[1] = gid[t] + head[t];
  }
  for (int o = 16; o; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
  if ((threadIdx.x & 31u) == 0 && all) atomicAdd(out, all);
}

// Row lengths (kFill false: rp[r] = count) or elements (kFill true: rp holds
// the row pointers) of rows r = warp, warp + warps, ...  The diagonal is
// always stored; off-diagonal elements when nonzero.  The columns that pass
// the excitation test are queued in shared memory (in column order) and
// evaluated 32 at a time, one per lane, so that the Slater-Condon work runs
// on full warps rather than on the one or two lanes that hit in a step.
//
// Bound: latency of the gathers (integrals, columns' keys).  kMates: the doubles of
// the row's own alpha string from its mates, merged; else by searching that string
// in every group a beta double away.  A counting pass over 1e5 random-walk
// determinants (117 mates a row against some 700 searches) takes 1.34 ms by mates,
// 1.75 by searches; lists on either side of the choice are at mates_are_fewer.
// (32 registers a thread by mates: with 48, 8 x 12870 strings took 20.4 instead of
// 18.5 ms; the gathers want warps.)
constexpr int kRowWarps = 8;

template <bool kFill>
__device__ __forceinline__ void flush_queue(const DevInts &I, const uint64_t *keys, uint32_t r,
                                            uint32_t ai, uint32_t bi, const double *diag,
                                            uint32_t *q, int k, uint32_t lane, uint32_t below,
                                            int64_t &pos, int64_t end, int64_t &cnt, int32_t *col,
                                            double *val) {
  double v = 0.0;
  uint32_t j = 0;
  bool nz = false;
  if ((int)lane < k) {
    j = q[lane];
    if (j == r) {
      v = diag[r];
      nz = true;
    } else {
      const uint64_t kj = keys[j];
      v = offdiag_element(I, ai, bi, key_alpha(kj), key_beta(kj));
      nz = v != 0.0;
    }
  }
  const uint32_t bal = __ballot_sync(0xffffffffu, nz);
  if (kFill) {
    if (nz) {
      const int64_t p = pos + __popc(bal & below);
      if (p < end) {
        col[p] = (int32_t)j;
        val[p] = v;
      }
    }
    pos += __popc(bal);
  } else {
    cnt += __popc(bal);
  }
}

template <bool kFill, bool kMates>
__global__ void __launch_bounds__(kRowWarps * 32, kMates ? 8 : 6) k_ham_rows(
    DevInts I, const uint64_t *__restrict__ keys, uint32_t n, const uint32_t *__restrict__ of_row,
    const uint32_t *__restrict__ gstart, const uint32_t *__restrict__ gbeta,
    const int64_t *__restrict__ nbr_ptr, const uint32_t *__restrict__ nbr,
    const uint2 *__restrict__ mates, const uint2 *__restrict__ span,
    const double *__restrict__ diag, int64_t *rp, int32_t *col, double *val) {
  __shared__ uint32_t queue[kRowWarps][64];
  __shared__ uint2 place[kMates ? kRowWarps : 1][32];
  __shared__ uint32_t found[kMates ? kRowWarps : 1][64];
  uint2 *pl = place[kMates ? threadIdx.x >> 5 : 0];
  uint32_t *yq = found[kMates ? threadIdx.x >> 5 : 0];
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t below = (1u << lane) - 1u;
  uint32_t *q = queue[threadIdx.x >> 5];
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
    const uint64_t ki = keys[r];
    const uint32_t ai = key_alpha(ki), bi = key_beta(ki);
    const uint32_t g = of_row[r];
    int64_t pos = 0, end = 0, cnt = 0;
    if (kFill) {
      pos = rp[r];
      end = rp[r + 1];
    }
    int qn = 0;  // queued columns (warp-uniform, < 64)
    // two ascending lists, merged 32 entries at a time: the neighbour groups (x,
    // first column and length) and the row's alpha mates a beta double away (y,
    // one column each); lane k then holds entry k's first column, length and
    // alpha threshold, and the columns are walked as one concatenated range, 32
    // per step, each lane finding its entry by a binary search over the lanes'
    // offsets.  Without the mates, the groups a beta double away are among x, and
    // the row's alpha string is searched in each.
    int64_t x0 = nbr_ptr[g];
    const int64_t x1 = nbr_ptr[g + 1];
    const uint2 ys = kMates ? span[r] : make_uint2(0u, 0u);
    constexpr uint32_t kNone = 0xffffffffu;  // n < 2^31
    uint32_t y0 = ys.x;
    int yn = 0;  // mates in hand (warp-uniform, < 64)
    while (kMates || x0 < x1) {
      uint32_t gs = 0, len = 0;
      int thr = -1;
      if constexpr (!kMates) {
        if (x1 - x0 > (int64_t)lane) {
          const uint32_t g2 = nbr[x0 + lane];
          gs = gstart[g2];
          len = gstart[g2 + 1] - gs;
          thr = 4 - __popc(bi ^ gbeta[g2]);
          if (thr == 0) {  // the group (in alpha order) is that one column, or nothing
            uint32_t lo = gs, hi = gs + len;
            while (lo < hi) {
              const uint32_t mid = (lo + hi) >> 1;
              if (key_alpha(keys[mid]) < ai) lo = mid + 1;
              else hi = mid;
            }
            len = lo < gs + len && key_alpha(keys[lo]) == ai ? 1u : 0u;
            gs = lo;
          }
        }
        x0 += 32;
      } else {
        for (; yn < 32 && y0 < ys.y; y0 += 32) {
          uint2 m = make_uint2(0u, bi);
          if (ys.y - y0 > lane) m = mates[y0 + lane];
          const bool hit = __popc(bi ^ m.y) == 4;
          const uint32_t bal = __ballot_sync(0xffffffffu, hit);
          if (!bal) continue;
          if (hit) yq[yn + __popc(bal & below)] = m.x;
          yn += __popc(bal);
        }
        __syncwarp();
        if (x0 >= x1 && yn == 0) break;
        // groups that start past the mates seen so far wait for the next mates
        const uint32_t lim = y0 < ys.y ? mates[y0 - 1u].x : kNone;
        const uint32_t yj = (int)lane < yn ? yq[lane] : kNone;
        uint32_t xs = kNone, xl = 0, xt = 0;
        if (x1 - x0 > (int64_t)lane) {
          const uint32_t g2 = nbr[x0 + lane];
          xs = gstart[g2];
          xl = gstart[g2 + 1] - xs;
          xt = 4u - (uint32_t)__popc(bi ^ gbeta[g2]);  // 4 or 2
        }
        uint32_t nx = 0, ny = 0;  // groups up to this lane's mate, mates before its group
        for (int step = 16; step; step >>= 1) {
          const uint32_t a = __shfl_sync(0xffffffffu, xs, nx + step - 1);
          const uint32_t b = __shfl_sync(0xffffffffu, yj, ny + step - 1);
          if (a <= yj) nx += step;
          if (b < xs) ny += step;
        }
        const uint32_t xlast = __shfl_sync(0xffffffffu, xs, 31);
        if (nx == 31 && xlast <= yj) nx = 32;
        const uint32_t y32 = __shfl_sync(0xffffffffu, yj, 31);
        if (ny == 31 && y32 < xs) ny = 32;
        const uint32_t rx = lane + ny, ry = lane + nx;
        const bool take_x = xs != kNone && xs <= lim && rx < 32u, take_y = yj != kNone && ry < 32u;
        // the threshold's two bits (0, 2 or 4) above the column and the length
        if (take_x) pl[rx] = make_uint2(xs | ((xt & 2u) << 30), xl | ((xt & 4u) << 29));
        if (take_y) pl[ry] = make_uint2(yj, 1u);
        const uint32_t tx = __ballot_sync(0xffffffffu, take_x), ty = __ballot_sync(0xffffffffu, take_y);
        __syncwarp();
        if ((int)lane < __popc(tx) + __popc(ty)) {
          const uint2 e = pl[lane];
          gs = e.x & 0x7fffffffu;
          len = e.y & 0x7fffffffu;
          thr = (int)(((e.x >> 30) & 2u) | ((e.y >> 29) & 4u));
        }
        __syncwarp();
        x0 += __popc(tx);
        if (ty) {
          const int k = __popc(ty);
          const uint32_t a = (int)lane + k < yn ? yq[lane + k] : 0u;
          const uint32_t b = (int)lane + 32 + k < yn ? yq[lane + 32 + k] : 0u;
          __syncwarp();
          yn -= k;
          if ((int)lane < yn) yq[lane] = a;
          if ((int)lane + 32 < yn) yq[lane + 32] = b;
          __syncwarp();
        }
      }
      uint32_t off = len;  // inclusive scan of the lengths
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, off, o);
        if ((int)lane >= o) off += y;
      }
      const uint32_t total = __shfl_sync(0xffffffffu, off, 31);
      off -= len;  // exclusive
      for (uint32_t c = 0; c < total; c += 32) {
        const uint32_t idx = c + lane;
        int k = 0;  // the last lane whose offset is <= idx
        for (int step = 16; step; step >>= 1) {
          const uint32_t o2 = __shfl_sync(0xffffffffu, off, k + step);
          if (o2 <= idx) k += step;
        }
        const uint32_t j = __shfl_sync(0xffffffffu, gs, k) + (idx - __shfl_sync(0xffffffffu, off, k));
        const int t = __shfl_sync(0xffffffffu, thr, k);
        const bool hit = idx < total && __popc(ai ^ key_alpha(keys[idx < total ? j : r])) <= t;
        const uint32_t bal = __ballot_sync(0xffffffffu, hit);
        if (hit) q[qn + __popc(bal & below)] = j;
        qn += __popc(bal);
        __syncwarp();
        if (qn >= 32) {
          flush_queue<kFill>(I, keys, r, ai, bi, diag, q, 32, lane, below, pos, end, cnt, col,
                             val);
          const uint32_t rest = (lane + 32 < (uint32_t)qn) ? q[lane + 32] : 0u;
          __syncwarp();
          if (lane + 32 < (uint32_t)qn) q[lane] = rest;
          qn -= 32;
          __syncwarp();
        }
      }
    }
    if (qn > 0)
      flush_queue<kFill>(I, keys, r, ai, bi, diag, q, qn, lane, below, pos, end, cnt, col, val);
    __syncwarp();
    if (!kFill && lane == 0) rp[r] = cnt;
  }
}

__global__ void k_row_ptr(const uint64_t *off, uint32_t n, uint32_t nchunks, int64_t *row_ptr) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x)
    row_ptr[i] = (int64_t)off[(size_t)i * nchunks];
}

// Remapping a key-ordered CSR to the caller's order: perm[r] is the caller's
// index of key-ordered row r.
__global__ void k_user_counts(const int64_t *rp, const uint32_t *perm, uint32_t n,
                              int64_t *cnt_user) {
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x)
    cnt_user[perm[r]] = rp[r + 1] - rp[r];
}

__global__ void k_user_entries(const int64_t *rp, const int32_t *col, const uint32_t *perm,
                               uint32_t n, uint64_t *ekey) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
    const uint64_t u = (uint64_t)perm[r] << 32;
    for (int64_t k = rp[r] + lane; k < rp[r + 1]; k += 32) {
      const uint32_t c = (uint32_t)col[k];
      ekey[k] = u | (c < n ? perm[c] : 0xffffffffu);
    }
  }
}

__global__ void k_low_cols(const uint64_t *ekey, size_t nnz, int32_t *col) {
  for (size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x; k < nnz;
       k += (size_t)gridDim.x * blockDim.x)
    col[k] = (int32_t)(uint32_t)ekey[k];
}

__global__ void k_iota(uint32_t *v, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    v[i] = i;
}

__global__ void k_not_identity(const uint32_t *perm, uint32_t n, unsigned *flag) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (perm[i] != i) *flag = 1u;
}

struct HamGeom {
  uint32_t gx, gy, chunk;
};

// Rows in CTAs of 256; columns split so that the grid holds about 8 CTAs per
// SM (a slice never narrower than one shared-memory stage).
HamGeom ham_geom(uint32_t n) {
  HamGeom g;
  g.gx = (n + kRowThreads - 1) / kRowThreads;
  uint32_t want = (152u * 8u + g.gx - 1) / g.gx;
  const uint32_t most = (n + kColStage - 1) / kColStage;
  want = std::max(1u, std::min(want, most));
  g.chunk = (n + want - 1) / want;
  g.gy = (n + g.chunk - 1) / g.chunk;
  return g;
}

// ------------------------------ products -----------------------------------

__global__ void k_spmv(const int64_t *__restrict__ rp, const int32_t *__restrict__ col,
                       const double *__restrict__ val, uint32_t n, const double *__restrict__ x,
                       double *__restrict__ y, const int *stop) {
  if (stop && *stop) return;
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
    const int64_t b = rp[r], e = rp[r + 1];
    double s = 0.0;
#pragma unroll 4
    for (int64_t k = b + lane; k < e; k += 32) s = fma(__ldg(val + k), __ldg(x + __ldg(col + k)), s);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) y[r] = s;
  }
}

// out[k * s1] (and out2[k * s2] when given) = V_k . b for k = blockIdx.y
// (V_k = V + k * ld).  Each block writes the partial sum of its slice; the
// last block of a vector to finish (a ticket counter, reset by that block)
// adds the partials in block order, so the result does not depend on which
// block finishes last.
__global__ void __launch_bounds__(kDotThreads) k_dots(const double *V, size_t ld,
                                                      const double *b, size_t n, double *part,
                                                      unsigned *ticket, double *out, int s1,
                                                      double *out2, int s2) {
  __shared__ double red[kDotThreads / 32];
  __shared__ bool last;
  const size_t per = (n + gridDim.x - 1) / gridDim.x;
  const size_t lo = (size_t)blockIdx.x * per, hi = min(n, lo + per);
  const int k = blockIdx.y;
  const double *v = V + (size_t)k * ld;
  double s = 0.0;
  for (size_t i = lo + threadIdx.x; i < hi; i += kDotThreads) s = fma(v[i], b[i], s);
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31u) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kDotThreads / 32; ++w) t += red[w];
    part[(size_t)k * gridDim.x + blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(ticket + k, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x >= 32) return;
  __threadfence();
  const volatile double *pk = part + (size_t)k * gridDim.x;
  double t = 0.0;
  for (unsigned g = threadIdx.x; g < gridDim.x; g += 32) t += pk[g];
  for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (threadIdx.x == 0) {
    out[(size_t)k * s1] = t;
    if (out2) out2[(size_t)k * s2] = t;
    ticket[k] = 0u;
  }
}

// out = sum_k coef[k] scale[k] V_k
__global__ void k_combine(const double *V, size_t ld, int m, const double *coef,
                          const double *scale, size_t n, double *out) {
  __shared__ double cf[kMaxSub];
  for (int k = threadIdx.x; k < m; k += blockDim.x) cf[k] = coef[k] * scale[k];
  __syncthreads();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int k = 0; k < m; ++k) s = fma(cf[k], V[(size_t)k * ld + i], s);
    out[i] = s;
  }
}

// State of a Davidson solve on the device.  The host enqueues several
// iterations at a time; once `stop` is set, the kernels of the iterations
// behind it return at once, so the basis, its size and the coefficients stay
// those of the iteration that stopped.
//
// A basis vector is kept as the correction it was made from, with its factor:
// v_j = scale[j] T_j, W_j = H T_j, so no pass over the vectors normalises them.
enum : int { kStopConverged = 1, kStopSpent = 2, kStopBad = 3 };  // spent: nothing left to add
struct DavState {
  int stop;
  int iter;      // products performed when the last residual was formed
  double theta;  // lowest Ritz value
  double res2;   // |H x - theta x|^2
  double scale[kMaxSub + 1];
};

constexpr int kPassThreads = 128;
constexpr int kPassBlocks = 304;  // at most: two per SM

// One pass over the vectors, an element per thread and step.  Each mode forms
// per-element values and sums over the elements (in registers per thread, then
// over the block, then by the last block over the blocks: a fixed order, so the
// same bits on every call):
//   kProject  sums j < m: T_j . W_(m-1): the new column of v^T H v, written to
//             row and column m - 1 of Hs
//   kRitz     x = v c, H x = W c, r = H x - theta x, t = r / (theta - H_ii)
//             (the denominator kept at least 1e-8 in magnitude; t = r when
//             unpreconditioned); sums j < m: T_j . t, and r . r
//   kRestart  the same with T, W replaced in place by the `keep` lowest Ritz
//             vectors and their products; sums k < keep: T_k . t, and r . r
//   kOrth1    t -= v h; sums j < m: T_j . t (for the second pass)
//   kOrth2    t -= v h; sum t . t
// t is the next basis vector's place.  A pass reads its vectors once (from L2
// at 50,000 determinants) with all loads of an element in flight, and takes up
// to 3 m FP64 operations per element; 8 to 17 us at 50,000 elements, half of it
// the launch and the tail of the sums.  With the subspace solve below, a
// product costs 6 launches instead of 12: a solve at 50,000 determinants 34.8
// -> 15.4 ms.  The sums of a warp's lanes are folded value against value (half of
// the values kept by each half of the lanes, and so on): M + 1 FP64 additions per
// warp for M values instead of 5 M.
enum : int { kProject, kRitz, kRestart, kOrth1, kOrth2 };

struct PassArgs {
  double *T, *W;
  size_t n;
  int m, keep;
  const double *coef;   // kRitz, kRestart: Ct; kOrth1, kOrth2: h
  const double *theta;
  const double *diag;
  double *t;
  bool precondition;
  int iter;
  double tol;
  double *Hs, *h;       // outputs of the sums
  double *part;         // partial sums of the blocks
  unsigned *ticket;     // zero between launches
  DavState *st;
};

// Sums over the warp of v[0 .. M), M a power of two up to 32: on return lane l
// holds the sum of v[l % M].
template <int M>
__device__ __forceinline__ double fold_sums(double (&v)[M]) {
  const unsigned lane = threadIdx.x & 31u;
#pragma unroll
  for (int o = M / 2; o; o >>= 1) {
    const bool up = (lane & (unsigned)o) != 0u;
#pragma unroll
    for (int j = 0; j < o; ++j) {
      const double give = up ? v[j] : v[j + o], have = up ? v[j + o] : v[j];
      v[j] = have + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double s = v[0];
#pragma unroll
  for (int o = M; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

template <int MODE, int MAXM>
__global__ void __launch_bounds__(kPassThreads) k_pass(PassArgs A) {
  constexpr int kWarps = kPassThreads / 32;
  __shared__ double cf[MODE == kRestart ? kKeep * kMaxSub : kMaxSub];
  __shared__ double red[kWarps][kMaxSub + 1];
  __shared__ double sum[kMaxSub + 1];
  __shared__ double fin[kPassThreads];
  __shared__ bool last;
  if (A.st->stop) return;
  const int m = A.m, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = MODE == kRestart ? A.keep : 1;
  const int nh = MODE == kOrth2 ? 0 : (MODE == kRestart ? K : m);  // sums T_j . something
  const bool extra = MODE != kProject && MODE != kOrth1;           // r . r or t . t
  const int nval = nh + (extra ? 1 : 0);
  // coefficients of the T_j (with the factors of the basis vectors)
  if (MODE == kRitz || MODE == kRestart)
    for (int e = tid; e < K * m; e += kPassThreads) {
      const int k = e / m, j = e - k * m;
      cf[e] = A.coef[(size_t)k * kMaxSub + j] * A.st->scale[j];
    }
  if (MODE == kOrth1 || MODE == kOrth2)
    for (int e = tid; e < m; e += kPassThreads) cf[e] = -A.coef[e];
  const double theta = (MODE == kRitz || MODE == kRestart) ? *A.theta : 0.0;
  double acc[MAXM], ex = 0.0;
#pragma unroll
  for (int j = 0; j < MAXM; ++j) acc[j] = 0.0;
  __syncthreads();
  const size_t n = A.n;
  for (size_t i = (size_t)blockIdx.x * kPassThreads + tid; i < n;
       i += (size_t)gridDim.x * kPassThreads) {
    double *T = A.T + i, *W = A.W + i;
    double v[MAXM];
#pragma unroll
    for (int j = 0; j < MAXM; ++j) v[j] = j < m ? T[(size_t)j * n] : 0.0;
    if (MODE == kProject) {
      const double w = W[(size_t)(m - 1) * n];
#pragma unroll
      for (int j = 0; j < MAXM; ++j)
        if (j < m) acc[j] = fma(v[j], w, acc[j]);
      continue;
    }
    if (MODE == kOrth1 || MODE == kOrth2) {
      double t = A.t[i];
#pragma unroll
      for (int j = 0; j < MAXM; ++j)
        if (j < m) t = fma(cf[j], v[j], t);
      A.t[i] = t;
      if (MODE == kOrth2) {
        ex = fma(t, t, ex);
      } else {
#pragma unroll
        for (int j = 0; j < MAXM; ++j)
          if (j < m) acc[j] = fma(v[j], t, acc[j]);
      }
      continue;
    }
    double x = 0.0, wx = 0.0, xs[kKeep];
    if (MODE == kRestart) {
      double ws[kKeep];
#pragma unroll
      for (int k = 0; k < kKeep; ++k) xs[k] = ws[k] = 0.0;
#pragma unroll
      for (int j = 0; j < MAXM; ++j)
        if (j < m) {
          const double w = W[(size_t)j * n];
#pragma unroll
          for (int k = 0; k < kKeep; ++k)
            if (k < K) {
              xs[k] = fma(cf[k * m + j], v[j], xs[k]);
              ws[k] = fma(cf[k * m + j], w, ws[k]);
            }
        }
#pragma unroll
      for (int k = 0; k < kKeep; ++k)
        if (k < K) {
          T[(size_t)k * n] = xs[k];
          W[(size_t)k * n] = ws[k];
        }
      x = xs[0];
      wx = ws[0];
    } else {
      double w[MAXM];
#pragma unroll
      for (int j = 0; j < MAXM; ++j) w[j] = j < m ? W[(size_t)j * n] : 0.0;
#pragma unroll
      for (int j = 0; j < MAXM; ++j)
        if (j < m) {
          x = fma(cf[j], v[j], x);
          wx = fma(cf[j], w[j], wx);
        }
    }
    const double r = fma(-theta, x, wx);
    double t = r;
    if (A.precondition) {
      double d = theta - A.diag[i];
      if (fabs(d) < 1e-8) d = d < 0.0 ? -1e-8 : 1e-8;
      t = fabs(d) <= 1e30 ? r * recip_fast(d) : r / d;
    }
    A.t[i] = t;
    if (MODE == kRestart) {
#pragma unroll
      for (int k = 0; k < kKeep; ++k)
        if (k < K) acc[k] = fma(xs[k], t, acc[k]);
    } else {
#pragma unroll
      for (int j = 0; j < MAXM; ++j)
        if (j < m) acc[j] = fma(v[j], t, acc[j]);
    }
    ex = fma(r, r, ex);
  }
  if (nh) {
    const double s = fold_sums<MAXM>(acc);
    if (lane < nh) red[warp][lane] = s;
  }
  if (extra) {
    for (int o = 16; o; o >>= 1) ex += __shfl_xor_sync(0xffffffffu, ex, o);
    if (lane == 0) red[warp][nh] = ex;
  }
  __syncthreads();
  if (tid < nval) {
    double s = red[0][tid];
    for (int w = 1; w < kWarps; ++w) s += red[w][tid];
    A.part[(size_t)tid * gridDim.x + blockIdx.x] = s;
    __threadfence();
  }
  __syncthreads();
  if (tid == 0) last = atomicAdd(A.ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the blocks' sums: 8 lanes per value, then the 8 in order
  for (int j0 = 0; j0 < nval; j0 += kPassThreads / 8) {
    const int j = j0 + (tid >> 3), p = tid & 7;
    double s = 0.0;
    if (j < nval) {
      const double *q = A.part + (size_t)j * gridDim.x;
#pragma unroll 8
      for (unsigned e = p; e < gridDim.x; e += 8) s += __ldcg(q + e);
    }
    fin[tid] = s;
    __syncthreads();
    if (p == 0 && j < nval) {
      double t = fin[tid];
      for (int u = 1; u < 8; ++u) t += fin[tid + u];
      sum[j] = t;
    }
    __syncthreads();
  }
  DavState *st = A.st;
  if (MODE == kProject) {
    const double sm = st->scale[m - 1];
    for (int j = tid; j < m; j += kPassThreads) {
      const double v = sum[j] * st->scale[j] * sm;
      A.Hs[j * kMaxSub + (m - 1)] = v;
      A.Hs[(m - 1) * kMaxSub + j] = v;
    }
  } else {
    // v_j (v_j . t) = T_j scale_j^2 (T_j . t); restarted vectors have scale 1
    for (int j = tid; j < nh; j += kPassThreads) {
      const double sj = MODE == kRestart ? 1.0 : st->scale[j];
      A.h[j] = sum[j] * sj * sj;
    }
  }
  if (MODE == kRestart && tid < K) st->scale[tid] = 1.0;
  if (tid == 0) {
    *A.ticket = 0u;
    if (MODE == kRitz || MODE == kRestart) {
      const double rr = sum[nh];
      st->iter = A.iter;
      st->theta = theta;
      st->res2 = rr;
      if (!isfinite(theta) || !isfinite(rr)) st->stop = kStopBad;
      else if (sqrt(rr > 0.0 ? rr : 0.0) <= A.tol) st->stop = kStopConverged;
    }
    if (MODE == kOrth2) {
      st->scale[m] = 1.0 / sqrt(sum[0]);
      if (!(sum[0] > 1e-28)) st->stop = kStopSpent;  // the correction lies in the basis
    }
  }
}

// *out = 1 / sqrt(*norm2)
__global__ void k_inverse_norm(const double *norm2, double *out) { *out = 1.0 / sqrt(*norm2); }

// v *= 1 / sqrt(*norm2)
__global__ void k_normalize(double *v, size_t n, const double *norm2) {
  const double s = 1.0 / sqrt(*norm2);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    v[i] *= s;
}

// The lowest eigenpairs of the symmetric m x m subspace matrix Hs (leading
// dimension kMaxSub), one CTA.
//
// GB300 executes about 1.7 FP64 operations per clock per SM, against some 126
// FP32 ones, so the eigenvectors are found in FP32 and only the wanted ones
// (the lowest; the kKeep lowest at a restart) refined in FP64:
//   1. Jacobi rotations in the parallel (round-robin) ordering (Brent and Luk,
//      1985; Golub and Van Loan, Sec. 8.5) on Hs - Hs_00 in FP32: a sweep is
//      M - 1 rounds (M = m rounded up to even; the extra index has no
//      couplings), each round pairs every index with one other, so its M / 2
//      rotations act on disjoint planes and each 2 x 2 block of the matrix is
//      updated by one thread.  The matrix grew by a row since the last call, so
//      the sweeps start from that call's eigenbasis (two or three instead of
//      six).
//   2. Per wanted eigenpair, a warp iterates in FP64: theta = x.Hx,
//      r = Hx - theta x, x <- x - Q (L - theta)^-1 Q^T r with the FP32
//      eigenbasis Q, L as the approximate inverse (its own component left
//      out), normalised.  Each step shrinks the error by about the FP32
//      eigenbasis's own (1e-4), until |r| is at FP64 rounding.
//   3. Several eigenvectors are orthonormalised by two passes of Gram-Schmidt
//      and ordered by their FP64 eigenvalues.
// A small residual shows an eigenpair, not which one.  The next FP32 eigenvalue d
// is a lower bound of every eigenvalue that was not refined, up to: the
// off-diagonal norm left (Weyl's bound); 4e-3 |d|, for an eigenbasis off
// orthonormal by at most 2e-3 (Ostrowski's bound; each of up to 28 x 12 x 31
// warm-started rotations of a column scales it by 1 + 2e-7 at most); and 1e-5 of the
// matrix for the FP32 rounding.  Unless the lowest refined eigenvalue is below d by
// that much, and when a pair's residual stays above 1e-13 of the matrix or two
// pairs turned out to be the same (eigenvalues too close for FP32 to tell
// apart), the whole matrix goes through FP64 Jacobi: FP32 eigenvectors
// orthonormalised in FP64, Q^T Hs Q, FP64 sweeps to an off-diagonal norm of 1e-13
// of the diagonal's.
// m = 16: 15 us against 135 for the FP64 Jacobi that every product took.
constexpr int kEigThreads = 256;

// 1/sqrt(x) to FP64 accuracy from the FP32 estimate rsqrtf and two
// Newton-Raphson steps y <- y(3 - xy^2)/2 (2^-23 -> 2^-92), for x in
// [1e-30, 1e30]; with recip_fast it avoids the FP64 division and square-root
// sequences.
__device__ __forceinline__ double rsqrt_fast(double x) {
  double y = (double)rsqrtf((float)x);
  y = y * fma(-0.5 * x, y * y, 1.5);
  return y * fma(-0.5 * x, y * y, 1.5);
}

// The Jacobi rotation (c, s) that zeroes a_pq: tau = (a_qq - a_pp) / (2 a_pq),
// t = sign(tau) / (|tau| + sqrt(1 + tau^2)), c = 1 / sqrt(1 + t^2), s = t c
// (Golub and Van Loan, Alg. 8.5.1), with the fast reciprocals when every
// operand is in their range and the exact operations otherwise.
__device__ __forceinline__ void rotation(double app, double aqq, double apq, double *c,
                                         double *s) {
  const double d = aqq - app, a2 = 2.0 * apq;
  const bool fast = fabs(a2) > 1e-30 && fabs(a2) < 1e30 && fabs(d) < 1e15 * fabs(a2);
  double t;
  if (fast) {
    const double tau = d * recip_fast(a2);  // |tau| < 1e15
    const double y = fma(tau, tau, 1.0);
    const double den = fabs(tau) + y * rsqrt_fast(y);  // in [1, 2e15]
    t = (tau >= 0.0 ? 1.0 : -1.0) * recip_fast(den);
  } else {
    const double tau = d / a2;
    t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
  }
  const double cs = rsqrt_fast(fma(t, t, 1.0));  // 1 + t^2 in [1, 2]
  *c = cs;
  *s = t * cs;
}

constexpr int kEigPer = (kMaxSub * kMaxSub + kEigThreads - 1) / kEigThreads;

struct EigScratch {
  int rp[kMaxSub / 2], rq[kMaxSub / 2];
  double rc[kMaxSub / 2], rs[kMaxSub / 2];
  double red[2][kEigThreads / 32];
  int done;
};

// Parallel-order Jacobi sweeps in FP64 on A (symmetric, m x m) accumulating
// into Q, until the off-diagonal norm is at most sqrt(thr) of the diagonal's or
// after max_sweeps.  One thread per pair forms its rotation from the round's
// matrix, then the CTA applies all of them to the columns (and to Q), then to
// the rows.  Every thread of the CTA calls it.
__device__ void jacobi_sweeps(double (*A)[kMaxSub + 1], double (*Q)[kMaxSub + 1], int m,
                              int max_sweeps, double thr, EigScratch &E) {
  const int tid = threadIdx.x;
  const int M = m + (m & 1);
  const int half = M / 2;
  for (int sweep = 0; sweep < max_sweeps && m > 1; ++sweep) {
    double off = 0.0, dg = 0.0;
    for (int e = tid; e < m * m; e += kEigThreads) {
      const int i = e / m, k = e - (e / m) * m;
      const double a = A[i][k];
      if (i == k) dg += a * a;
      else off += a * a;
    }
    for (int o = 16; o; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      dg += __shfl_xor_sync(0xffffffffu, dg, o);
    }
    if ((tid & 31) == 0) {
      E.red[0][tid >> 5] = off;
      E.red[1][tid >> 5] = dg;
    }
    __syncthreads();
    if (tid == 0) {
      double so = 0.0, sd = 0.0;
      for (int w = 0; w < kEigThreads / 32; ++w) {
        so += E.red[0][w];
        sd += E.red[1][w];
      }
      E.done = so <= thr * sd;
    }
    __syncthreads();
    if (E.done) break;
    for (int r = 0; r < M - 1; ++r) {
      if (tid < half) {
        const int pa = tid == 0 ? 0 : 1 + (tid - 1 + r) % (M - 1);
        const int pb = 1 + (M - 2 - tid + r) % (M - 1);
        const int p = pa < pb ? pa : pb, q = pa < pb ? pb : pa;
        double cs = 1.0, sn = 0.0;
        if (q < m) {
          const double apq = A[p][q];
          if (fabs(apq) >= 1e-300) rotation(A[p][p], A[q][q], apq, &cs, &sn);
        }
        E.rc[tid] = cs;
        E.rs[tid] = sn;
        E.rp[tid] = p;
        E.rq[tid] = q;
      }
      __syncthreads();
      for (int e = tid; e < half * m; e += kEigThreads) {  // columns p, q of A and Q
        const int k = e / m, i = e - (e / m) * m;
        const int p = E.rp[k], q = E.rq[k];
        if (q >= m || E.rs[k] == 0.0) continue;
        const double cs = E.rc[k], sn = E.rs[k];
        const double aip = A[i][p], aiq = A[i][q];
        A[i][p] = cs * aip - sn * aiq;
        A[i][q] = sn * aip + cs * aiq;
        const double qip = Q[i][p], qiq = Q[i][q];
        Q[i][p] = cs * qip - sn * qiq;
        Q[i][q] = sn * qip + cs * qiq;
      }
      __syncthreads();
      for (int e = tid; e < half * m; e += kEigThreads) {  // rows p, q of A
        const int k = e / m, j = e - (e / m) * m;
        const int p = E.rp[k], q = E.rq[k];
        if (q >= m || E.rs[k] == 0.0) continue;
        const double cs = E.rc[k], sn = E.rs[k];
        const double apj = A[p][j], aqj = A[q][j];
        A[p][j] = cs * apj - sn * aqj;
        A[q][j] = sn * apj + cs * aqj;
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The FP32 rotation that zeroes apq by the hardware's approximate reciprocal
// and reciprocal square root (an error of some 1e-7 is made good by the
// refinement): t = sign(d) h / (|d| + sqrt(d^2 + h^2)), d = aqq - app, h = 2 apq.
__device__ __forceinline__ float2 rotation_fast(float app, float aqq, float apq) {
  const float d = aqq - app, h = 2.0f * apq;
  const float q = fmaf(d, d, h * h);
  if (!(q > 1e-35f) || h == 0.0f) return make_float2(1.0f, 0.0f);
  const float t = (d >= 0.0f ? h : -h) * rcp_approx(fmaf(q, rsqrt_approx(q), fabsf(d)));
  const float c = rsqrt_approx(fmaf(t, t, 1.0f));
  return make_float2(c, t * c);
}

// FP32 sweeps on A[0] (m x m, zero beyond) accumulating into Q[0], until the
// off-diagonal norm is 1e-4 of the matrix's (the refinement's contraction; a
// sweep costs as much as three of its steps).  Positions 2k and 2k + 1 are
// rotated against each other, a block of A (or a row's pair of Q) per thread,
// and the results written one place on in the round-robin into the other
// buffer, so a round has one barrier; after the M - 1 rounds of a sweep every
// index is back in its place.  Returns the buffer that holds the result; *off2
// and *all2 get the squares of its off-diagonal norm (infinite when the sweeps
// ran out) and of its norm.
__device__ int jacobi_fast(float (*A)[kMaxSub][kMaxSub + 1], float (*Q)[kMaxSub][kMaxSub + 1],
                           int m, float (*red)[kEigThreads / 32], float *off2, float *all2) {
  const int tid = threadIdx.x, M = m + (m & 1), half = M / 2;
  constexpr int kItems = (kMaxSub * kMaxSub / 4 + kMaxSub * kMaxSub / 2) / kEigThreads;
  const int items = half * half + M * half;  // blocks of A, then (row, pair) of Q
  auto next = [&](int pos) {
    if (pos == 0 || half == 1) return pos;
    if (pos & 1) return pos == 1 ? 2 : pos - 2;
    return pos == M - 2 ? M - 1 : pos + 2;
  };
  int it_k[kItems], it_l[kItems], to_l0[kItems], to_l1[kItems], to_k0[kItems], to_k1[kItems];
#pragma unroll
  for (int u = 0; u < kItems; ++u) {
    const int e = tid + u * kEigThreads;
    it_k[u] = e / max(half, 1);
    it_l[u] = e - it_k[u] * half;
    to_l0[u] = next(2 * it_l[u]);
    to_l1[u] = next(2 * it_l[u] + 1);
    to_k0[u] = next(2 * it_k[u]);
    to_k1[u] = next(2 * it_k[u] + 1);
  }
  int b = 0;
  *off2 = m > 1 ? __int_as_float(0x7f800000) : 0.0f;
  *all2 = 0.0f;
  for (int sweep = 0; sweep < 12 && m > 1; ++sweep) {
    float off = 0.0f, all = 0.0f;
    for (int e = tid; e < kMaxSub * M; e += kEigThreads) {
      const int i = e / kMaxSub, k = e % kMaxSub;
      if (k < M) {
        const float a = A[b][i][k];
        all = fmaf(a, a, all);
        if (i != k) off = fmaf(a, a, off);
      }
    }
    for (int o = 16; o; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      all += __shfl_xor_sync(0xffffffffu, all, o);
    }
    if ((tid & 31) == 0) {
      red[0][tid >> 5] = off;
      red[1][tid >> 5] = all;
    }
    __syncthreads();
    off = all = 0.0f;
#pragma unroll
    for (int w = 0; w < kEigThreads / 32; ++w) {
      off += red[0][w];
      all += red[1][w];
    }
    *all2 = all;
    if (!(off > 1e-8f * all)) {  // uniform
      *off2 = off;
      break;
    }
    for (int r = 0; r < M - 1; ++r, b ^= 1) {
      const float(*Ab)[kMaxSub + 1] = A[b];
      const float(*Qb)[kMaxSub + 1] = Q[b];
      float(*An)[kMaxSub + 1] = A[b ^ 1];
      float(*Qn)[kMaxSub + 1] = Q[b ^ 1];
#pragma unroll
      for (int u = 0; u < kItems; ++u) {
        if (tid + u * kEigThreads >= items) break;
        const int k = it_k[u], pl = 2 * it_l[u], ql = pl + 1;
        const float2 R = rotation_fast(Ab[pl][pl], Ab[ql][ql], Ab[pl][ql]);
        if (k < half) {
          const int pk = 2 * k, qk = pk + 1;
          const float x = Ab[pk][pl], y = Ab[pk][ql], z = Ab[qk][pl], w = Ab[qk][ql];
          const float2 L = rotation_fast(Ab[pk][pk], Ab[qk][qk], Ab[pk][qk]);
          const float x1 = L.x * x - L.y * z, z1 = L.y * x + L.x * z;
          const float y1 = L.x * y - L.y * w, w1 = L.y * y + L.x * w;
          An[to_k0[u]][to_l0[u]] = R.x * x1 - R.y * y1;
          An[to_k0[u]][to_l1[u]] = R.y * x1 + R.x * y1;
          An[to_k1[u]][to_l0[u]] = R.x * z1 - R.y * w1;
          An[to_k1[u]][to_l1[u]] = R.y * z1 + R.x * w1;
        } else {
          const float x = Qb[k - half][pl], y = Qb[k - half][ql];
          Qn[k - half][to_l0[u]] = R.x * x - R.y * y;
          Qn[k - half][to_l1[u]] = R.y * x + R.x * y;
        }
      }
      __syncthreads();
    }
  }
  __syncthreads();
  return b;
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// want lowest eigenpairs: theta[0 .. want), eigenvector k in Ct[k * kMaxSub + j].
// Qw keeps the FP32 eigenbasis; with `warm` it holds that of the leading
// m - 1 rows and columns, and the sweeps start in its basis (an arrowhead).
__global__ void __launch_bounds__(kEigThreads, 1) k_small_eig(const double *Hs, int m, int want,
                                                           bool warm, float *Qw, double *theta,
                                                           double *Ct, const int *stop) {
  __shared__ double H[kMaxSub][kMaxSub + 1];
  __shared__ double A[kMaxSub][kMaxSub + 1];
  __shared__ double Q[kMaxSub][kMaxSub + 1];
  __shared__ float A2[2][kMaxSub][kMaxSub + 1];
  __shared__ float Q2[2][kMaxSub][kMaxSub + 1];
  __shared__ double X[kKeep][kMaxSub], th[kKeep];
  __shared__ float gv[kKeep][kMaxSub], redf[2][kEigThreads / 32];
  __shared__ int of_rank[kMaxSub], failed, lowest;
  __shared__ double gsr[kMaxSub];
  __shared__ double nrm;
  __shared__ EigScratch E;
  if (stop && *stop) return;
  const int tid = threadIdx.x;
  const double shift = Hs[0];
#pragma unroll
  for (int e = tid; e < kMaxSub * kMaxSub; e += kEigThreads) {
    const int i = e / kMaxSub, k = e % kMaxSub;
    const bool in = i < m && k < m;
    const double h = in ? Hs[e] : 0.0;
    float q = i == k ? 1.0f : 0.0f;
    if (warm && i < m - 1 && k < m - 1) q = Qw[e];
    H[i][k] = h;
    A2[0][i][k] = (float)(in && i == k ? h - shift : h);
    Q2[0][i][k] = q;
  }
  if (tid == 0) {
    failed = 0;
    lowest = want >= m ? 1 : 0;  // the lowest of all pairs is among the refined ones
  }
  __syncthreads();
  if (warm) {  // A = Q^T A Q
    float p[kMaxSub * kMaxSub / kEigThreads];
    for (int side = 0; side < 2; ++side) {
#pragma unroll
      for (int u = 0; u < kMaxSub * kMaxSub / kEigThreads; ++u) {
        const int e = tid + u * kEigThreads, i = e / kMaxSub, k = e % kMaxSub;
        p[u] = 0.0f;
        if (i < m && k < m) {
#pragma unroll 8
          for (int l = 0; l < m; ++l)
            p[u] = side ? fmaf(Q2[0][l][i], A2[0][l][k], p[u]) : fmaf(A2[0][i][l], Q2[0][l][k], p[u]);
        }
      }
      __syncthreads();
#pragma unroll
      for (int u = 0; u < kMaxSub * kMaxSub / kEigThreads; ++u) {
        const int e = tid + u * kEigThreads, i = e / kMaxSub, k = e % kMaxSub;
        if (i < m && k < m) A2[0][i][k] = p[u];
      }
      __syncthreads();
    }
  }
  float off2, all2;
  const int buf = jacobi_fast(A2, Q2, m, redf, &off2, &all2);
  const float(*Af)[kMaxSub + 1] = A2[buf];
  const float(*Qf)[kMaxSub + 1] = Q2[buf];
#pragma unroll
  for (int e = tid; e < kMaxSub * kMaxSub; e += kEigThreads) {
    const int i = e / kMaxSub, k = e % kMaxSub;
    if (i < m && k < m) Qw[e] = Qf[i][k];
  }
  if (tid < m) {  // rank of each FP32 eigenvalue (ties by index)
    const float d = Af[tid][tid];
    int rk = 0;
    for (int j = 0; j < m; ++j) rk += (Af[j][j] < d) || (Af[j][j] == d && j < tid);
    of_rank[rk] = tid;
  }
  __syncthreads();
  const int w = tid >> 5, lane = tid & 31;
  if (w < want) {  // a warp per wanted pair
    const int own = of_rank[w];
    const bool in = lane < m;
    const float lam = in ? Af[lane][lane] : 0.0f;
    float scale = in ? fabsf(lam) : 0.0f;
    for (int o = 16; o; o >>= 1) scale = fmaxf(scale, __shfl_xor_sync(0xffffffffu, scale, o));
    scale += fabsf((float)shift);
    const float d = want < m ? Af[of_rank[want]][of_rank[want]] : 0.0f;
    const float bound = d - (sqrtf(2.0f * off2 + 2e-10f * all2) + 4e-3f * fabsf(d));
    double x = in ? (double)Qf[lane][own] : 0.0;
    x *= rsqrt_fast(warp_sum(x * x));
    double t = 0.0;
    float last = __int_as_float(0x7f800000);
    for (int it = 0; it < 16; ++it) {
      X[w][lane] = x;
      __syncwarp();
      double y = 0.0;
      if (m <= 16) {  // two lanes per row
        const int i = lane & 15, l0 = (lane >> 4) * 8;
        if (i < m)
          for (int l = l0; l < l0 + 8 && l < m; ++l) y = fma(H[i][l], X[w][l], y);
        y += __shfl_xor_sync(0xffffffffu, y, 16);
      } else if (in) {
        for (int l = 0; l < m; ++l) y = fma(H[lane][l], X[w][l], y);
      }
      if (!in) y = 0.0;
      t = warp_sum(x * y);
      const float r = (float)fma(-t, x, y);
      float rr = r * r;
      for (int o = 16; o; o >>= 1) rr += __shfl_xor_sync(0xffffffffu, rr, o);
      const float rn = sqrtf(rr);
      if (rn <= 4e-15f * scale) break;  // at rounding
      if (!(rn < 0.5f * last) || it == 15) {  // no longer falling
        if (!(rn <= 1e-13f * scale) && lane == 0) failed = 1;
        break;
      }
      last = rn;
      // the step from the FP32 eigenbasis
      gv[w][lane] = r;
      __syncwarp();
      float g = 0.0f;
      if (in)
#pragma unroll 8
        for (int l = 0; l < m; ++l) g = fmaf(Qf[l][lane], gv[w][l], g);
      const float gap = lam - (float)(t - shift);
      g = (in && lane != own && fabsf(gap) > 1e-6f * scale) ? __fdividef(g, gap) : 0.0f;
      __syncwarp();
      gv[w][lane] = g;
      __syncwarp();
      float dx = 0.0f;
      if (in)
#pragma unroll 8
        for (int l = 0; l < m; ++l) dx = fmaf(Qf[lane][l], gv[w][l], dx);
      __syncwarp();
      x -= (double)dx;
      x *= rsqrt_fast(warp_sum(x * x));
    }
    X[w][lane] = x;
    if (lane == 0) {
      th[w] = t;
      if ((float)(t - shift) < bound) lowest = 1;
    }
  }
  __syncthreads();
  if (!failed && lowest) {
    if (want > 1 && w == 0) {  // orthonormal: two passes of Gram-Schmidt, one vector after another
      for (int k = 0; k < want; ++k) {
        double x = X[k][lane];
        for (int pass = 0; pass < 2 && k > 0; ++pass) {
          double dots[kKeep];
#pragma unroll
          for (int j = 0; j < kKeep; ++j) dots[j] = j < k ? warp_sum(x * X[j][lane]) : 0.0;
#pragma unroll
          for (int j = 0; j < kKeep; ++j)
            if (j < k) x = fma(-dots[j], X[j][lane], x);
        }
        const double x2 = warp_sum(x * x);
        if (!(x2 > 0.25) && lane == 0) failed = 1;  // found before
        x *= rsqrt_fast(x2);
        X[k][lane] = x;
        __syncwarp();
      }
    }
    __syncthreads();
  }
  if (!failed && lowest) {
    auto place = [&](int k) {  // rank of pair k (ties by number)
      int rk = 0;
      for (int j = 0; j < want; ++j) rk += (th[j] < th[k]) || (th[j] == th[k] && j < k);
      return rk;
    };
    for (int k = w; k < want; k += kEigThreads / 32) {
      const int rk = want > 1 ? place(k) : 0;
      if (lane < m) Ct[(size_t)rk * kMaxSub + lane] = X[k][lane];
      if (lane == 0) theta[rk] = th[k];
    }
    return;
  }
  for (int e = tid; e < m * m; e += kEigThreads) {
    const int i = e / m, k = e - (e / m) * m;
    Q[i][k] = (double)Qf[i][k];
  }
  __syncthreads();
  // orthonormal columns in FP64: two passes of classical Gram-Schmidt each
  for (int k = 0; k < m; ++k) {
    for (int pass = 0; pass < 2; ++pass) {
      if (tid < k) {
        double t = 0.0;
        for (int i = 0; i < m; ++i) t = fma(Q[i][tid], Q[i][k], t);
        gsr[tid] = t;
      }
      __syncthreads();
      if (tid < m) {
        double t = Q[tid][k];
        for (int j = 0; j < k; ++j) t = fma(-gsr[j], Q[tid][j], t);
        Q[tid][k] = t;
      }
      __syncthreads();
    }
    if (tid < 32) {
      double v = tid < m ? Q[tid][k] * Q[tid][k] : 0.0;
      v = warp_sum(v);
      if (tid == 0) nrm = v;
    }
    __syncthreads();
    if (tid < m) Q[tid][k] *= rsqrt_fast(nrm);
    __syncthreads();
  }
  // A = Q^T Hs Q, through A = Hs Q and registers
  for (int e = tid; e < m * m; e += kEigThreads) {
    const int i = e / m, j = e - (e / m) * m;
    double t = 0.0;
    for (int l = 0; l < m; ++l) t = fma(H[i][l], Q[l][j], t);
    A[i][j] = t;
  }
  __syncthreads();
  double keep[kEigPer];
  for (int u = 0; u < kEigPer; ++u) {
    const int e = tid + u * kEigThreads;
    double t = 0.0;
    if (e < m * m) {
      const int i = e / m, j = e - (e / m) * m;
      for (int k = 0; k < m; ++k) t = fma(Q[k][i], A[k][j], t);
    }
    keep[u] = t;
  }
  __syncthreads();
  for (int u = 0; u < kEigPer; ++u) {
    const int e = tid + u * kEigThreads;
    if (e < m * m) A[e / m][e - (e / m) * m] = keep[u];
  }
  __syncthreads();
  jacobi_sweeps(A, Q, m, 8, 1e-26, E);
  for (int i = tid; i < m; i += kEigThreads) {
    const double d = A[i][i];
    int rk = 0;
    for (int j = 0; j < m; ++j) rk += (A[j][j] < d) || (A[j][j] == d && j < i);
    if (rk >= want) continue;
    theta[rk] = d;
    for (int k = 0; k < m; ++k) Ct[(size_t)rk * kMaxSub + k] = Q[k][i];
  }
}

// Hs = diag(theta[0..K)) after a restart.
__global__ void k_restart_hs(double *Hs, const double *theta, int K, const int *stop) {
  if (*stop) return;
  for (int e = threadIdx.x; e < kMaxSub * kMaxSub; e += blockDim.x) {
    const int i = e / kMaxSub, k = e - (e / kMaxSub) * kMaxSub;
    Hs[e] = (i == k && i < K) ? theta[i] : 0.0;
  }
}

// Largest |v_i| (lowest index among equal magnitudes): per-block candidates,
// then one block reduces them and flips the vector's sign if that entry is
// negative.
__global__ void k_absmax_part(const double *v, size_t n, double *bval, unsigned long long *bidx) {
  __shared__ double sv[256];
  __shared__ unsigned long long si[256];
  double best = -1.0;
  unsigned long long bi = ~0ull;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const double a = fabs(v[i]);
    if (a > best) {  // strided ascending: first index wins among equals
      best = a;
      bi = i;
    }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = 128; s; s >>= 1) {
    if (threadIdx.x < s) {
      const double o = sv[threadIdx.x + s];
      const unsigned long long oi = si[threadIdx.x + s];
      if (o > sv[threadIdx.x] || (o == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = o;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    bval[blockIdx.x] = sv[0];
    bidx[blockIdx.x] = si[0];
  }
}

__global__ void __launch_bounds__(256) k_absmax_sign(const double *bval,
                                                     const unsigned long long *bidx, int nb,
                                                     const double *v, double *sign) {
  __shared__ double sv[256];
  __shared__ unsigned long long si[256];
  double best = -1.0;
  unsigned long long bi = ~0ull;
  auto take = [&](double o, unsigned long long oi) {
    if (o > best || (o == best && oi < bi)) {
      best = o;
      bi = oi;
    }
  };
  for (int b = threadIdx.x; b < nb; b += 256) take(bval[b], bidx[b]);
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = 128; s; s >>= 1) {
    if ((int)threadIdx.x < s) {
      take(sv[threadIdx.x + s], si[threadIdx.x + s]);
      sv[threadIdx.x] = best;
      si[threadIdx.x] = bi;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *sign = (bi != ~0ull && v[bi] < 0.0) ? -1.0 : 1.0;
}

__global__ void k_scale_by(double *v, size_t n, const double *s) {
  const double f = *s;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    v[i] *= f;
}

__global__ void k_unit(double *v, size_t n, const double *diag) {
  // e_{argmin H_ii}, lowest index among equal values (one block scans)
  __shared__ double sv[256];
  __shared__ unsigned long long si[256];
  double best = INFINITY;
  unsigned long long bi = 0;
  for (size_t i = threadIdx.x; i < n; i += blockDim.x)
    if (diag[i] < best) {
      best = diag[i];
      bi = i;
    }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = 128; s; s >>= 1) {
    if (threadIdx.x < s) {
      const double o = sv[threadIdx.x + s];
      const unsigned long long oi = si[threadIdx.x + s];
      if (o < sv[threadIdx.x] || (o == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = o;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  for (size_t i = threadIdx.x; i < n; i += blockDim.x) v[i] = (i == si[0]) ? 1.0 : 0.0;
}

// A warp per row: the lanes scan the row's columns for the diagonal.
__global__ void k_csr_diag(const int64_t *rp, const int32_t *col, const double *val, uint32_t n,
                           double *diag) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t warps = (gridDim.x * blockDim.x) >> 5;
  for (uint32_t r = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; r < n; r += warps) {
    const int64_t e = rp[r + 1];
    double d = 0.0;
    for (int64_t k0 = rp[r]; k0 < e; k0 += 32) {
      const int64_t k = k0 + lane;
      const uint32_t hit = __ballot_sync(0xffffffffu, k < e && col[k] == (int32_t)r);
      if (hit) {
        d = val[k0 + __ffs(hit) - 1];
        break;
      }
    }
    if (lane == 0) diag[r] = d;
  }
}

// Number of keys of a[n] absent from the sorted list b[m] (binary search).
__global__ void k_count_missing(const uint64_t *a, size_t n, const uint64_t *b, size_t m,
                                unsigned long long *cnt) {
  unsigned long long c = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t k = a[i];
    size_t lo = 0, hi = m;
    while (lo < hi) {
      const size_t mid = (lo + hi) >> 1;
      if (b[mid] < k) lo = mid + 1;
      else hi = mid;
    }
    c += (lo == m || b[lo] != k);
  }
  if (c) atomicAdd(cnt, c);
}

__global__ void k_pack_dets(const asci_det *d, size_t n, uint64_t *keys) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    keys[i] = pack_key((uint32_t)d[i].alpha, (uint32_t)d[i].beta);
}

}  // namespace

// ------------------------------ host side ----------------------------------

struct Csr {
  const int64_t *row_ptr;
  const int32_t *col;
  const double *val;
  size_t n;
};

// Beta groups of key-ordered determinants and their neighbour graph.
struct BetaGraph {
  uint32_t G = 0;
  uint32_t *of_row = nullptr, *gstart = nullptr, *gbeta = nullptr, *nbr = nullptr;
  int64_t *nbr_ptr = nullptr;
  uint2 *mates = nullptr, *span = nullptr;  // rows in alpha order
  bool by_mates = true;                     // k_ham_rows: which of its two ways
};

// The row kernel looks at each of a row's mates (32 a step, loads that do not wait
// for one another), or searches its alpha string in the `doubles` groups a beta
// double away (32 at a time, ceil(log2 of a group's length) loads that do).  Build of
// n determinants (two calls, mates / searches): 16 orbitals, random walk of 1e5, 117
// mates against 705 groups of 11, 5.1 / 6.8 ms; 3335 mates, 784 groups of 8, 6.1 / 6.4;
// products 300 x 300 and 3432 x 8, 1.8 to 2.6 mates a group and load, equal; 2500 x
// 40, 152 groups of 40, 3.65 / 3.40; 12870 x 8, 16.8 / 15.7; 40000 of 20 orbitals x
// 4, 26.4 / 13.2.
static bool mates_are_fewer(double mates, double doubles, uint32_t n, uint32_t G) {
  int loads = 1;
  while (((uint64_t)G << loads) < (uint64_t)n) ++loads;
  return mates <= 2.0 * loads * doubles;
}

static int beta_graph(const uint64_t *keys, uint32_t n, const DevInts &I, BetaGraph *bg,
                      Arena &arena) {
  cudaStream_t s = arena.stream();
  uint32_t *head, *gid;
  ASCI_TRY(arena.alloc(&head, n));
  ASCI_TRY(arena.alloc(&gid, n));
  k_beta_heads<<<blocks_for(n, 256), 256, 0, s>>>(keys, n, head);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(scan_exclusive_u32(head, gid, n, arena));
  // rows in alpha order
  uint64_t *akey, *akey_alt;
  unsigned long long *d_tot, tot[2];
  ASCI_TRY(arena.alloc(&akey, n));
  ASCI_TRY(arena.alloc(&akey_alt, n));
  ASCI_TRY(arena.alloc(&d_tot, 2));
  ASCI_TRY(arena.alloc(&bg->mates, n));
  ASCI_TRY(arena.alloc(&bg->span, n));
  ASCI_TRY_CUDA(cudaMemsetAsync(d_tot, 0, sizeof(tot), s));
  k_alpha_keys<<<blocks_for(n, 256), 256, 0, s>>>(keys, n, akey);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(radix_sort_u64_varying(&akey, &akey_alt, n, 32, 32 + I.n,
                                  ((1ull << I.n) - 1ull) << 32, arena));
  k_alpha_mates<<<blocks_for(n, 256), 256, 0, s>>>(keys, akey, n, head, gid, bg->mates, bg->span,
                                                    d_tot);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaMemcpyAsync(tot, d_tot, sizeof(tot), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  const uint32_t G = (uint32_t)tot[1];
  ASCI_TRY(arena.alloc(&bg->of_row, n));
  ASCI_TRY(arena.alloc(&bg->gstart, (size_t)G + 1));
  ASCI_TRY(arena.alloc(&bg->gbeta, G));
  k_beta_groups<<<blocks_for(n, 256), 256, 0, s>>>(keys, n, head, gid, bg->of_row, bg->gstart,
                                                    bg->gbeta);
  ASCI_CHECK_LAUNCH();
  // which way: by the mates a row has and the beta doubles that G strings of all
  // would have, then by the doubles they do have
  const int nb = I.nb, nv = I.n - I.nb;
  double strings = 1.0;
  for (int k = 0; k < nb; ++k) strings *= (double)(I.n - k) / (k + 1);
  const double per_row = (double)tot[0] / n;
  bg->by_mates = mates_are_fewer(
      per_row, G / strings * (0.25 * nb * (nb - 1) * nv * (nv - 1)), n, G);
  // the group graph: count, scan, list
  const HamGeom g = ham_geom(G);
  const size_t slots = (size_t)G * g.gy;
  uint64_t *off, total = 0;
  ASCI_TRY(arena.alloc(&off, slots + 1));
  for (bool counted = false; !counted;) {
    const int reach = bg->by_mates ? 2 : 4;
    ASCI_TRY_CUDA(cudaMemsetAsync(off + slots, 0, sizeof(uint64_t), s));
    k_beta_pairs<false><<<dim3(g.gx, g.gy), kRowThreads, 0, s>>>(bg->gbeta, G, g.chunk, g.gy,
                                                                  reach, off, nullptr);
    ASCI_CHECK_LAUNCH();
    ASCI_TRY(scan_exclusive_u64(off, off, slots + 1, arena));
    ASCI_TRY_CUDA(cudaMemcpyAsync(&total, off + slots, sizeof(total), cudaMemcpyDeviceToHost, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    counted = bg->by_mates || !mates_are_fewer(per_row, (double)total / G, n, G);
    if (!counted) bg->by_mates = true;
  }
  ASCI_TRACE("hamiltonian rows: n=%u groups=%u mates=%llu pairs=%llu by %s", n, G, tot[0],
             (unsigned long long)total, bg->by_mates ? "mates" : "searches");
  ASCI_TRY(arena.alloc(&bg->nbr_ptr, (size_t)G + 1));
  k_row_ptr<<<blocks_for((size_t)G + 1, 256), 256, 0, s>>>(off, G, g.gy, bg->nbr_ptr);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(arena.alloc(&bg->nbr, total));
  k_beta_pairs<true><<<dim3(g.gx, g.gy), kRowThreads, 0, s>>>(bg->gbeta, G, g.chunk, g.gy,
                                                               bg->by_mates ? 2 : 4, off, bg->nbr);
  ASCI_CHECK_LAUNCH();
  bg->G = G;
  return ASCI_OK;
}

static unsigned row_blocks(uint32_t n) {
  return blocks_for((size_t)n * 32, kRowWarps * 32, 152 * 16);
}

// Counting pass and row pointers (rp[n + 1], device) of key-ordered keys.
static int ham_count(const DevInts &I, const uint64_t *keys, uint32_t n, const double *diag,
                     const BetaGraph &bg, int64_t *rp, size_t *nnz, Arena &arena) {
  cudaStream_t s = arena.stream();
  ASCI_TRY_CUDA(cudaMemsetAsync(rp + n, 0, sizeof(int64_t), s));
  auto *k = bg.by_mates ? k_ham_rows<false, true> : k_ham_rows<false, false>;
  k<<<row_blocks(n), kRowWarps * 32, 0, s>>>(I, keys, n, bg.of_row, bg.gstart, bg.gbeta, bg.nbr_ptr,
                                             bg.nbr, bg.mates, bg.span, diag, rp, nullptr, nullptr);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(scan_exclusive_u64(reinterpret_cast<uint64_t *>(rp), reinterpret_cast<uint64_t *>(rp),
                              (size_t)n + 1, arena));
  int64_t total = 0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&total, rp + n, sizeof(total), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  *nnz = (size_t)total;
  return ASCI_OK;
}

static int ham_fill(const DevInts &I, const uint64_t *keys, uint32_t n, const double *diag,
                    const BetaGraph &bg, int64_t *rp, int32_t *col, double *val, Arena &arena) {
  auto *k = bg.by_mates ? k_ham_rows<true, true> : k_ham_rows<true, false>;
  k<<<row_blocks(n), kRowWarps * 32, 0, arena.stream()>>>(I, keys, n, bg.of_row, bg.gstart, bg.gbeta,
                                                          bg.nbr_ptr, bg.nbr, bg.mates, bg.span,
                                                          diag, rp, col, val);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

static int spmv(const Csr &H, const double *x, double *y, cudaStream_t s,
                const int *stop = nullptr) {
  if (!H.n) return ASCI_OK;
  k_spmv<<<blocks_for(H.n * 32, 256, 152 * 32), 256, 0, s>>>(H.row_ptr, H.col, H.val,
                                                             (uint32_t)H.n, x, y, stop);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

// out[k * s1] (and out2[k * s2]) = V_k . b for k < m
// Scratch of the dot products: partial sums and the per-vector tickets (zero
// between calls).
struct DotScratch {
  double *part;
  unsigned *ticket;
};

static int dot_scratch(DotScratch *d, Arena &arena) {
  ASCI_TRY(arena.alloc(&d->part, (size_t)kMaxSub * kDotBlocks));
  ASCI_TRY(arena.alloc(&d->ticket, kMaxSub));
  ASCI_TRY_CUDA(cudaMemsetAsync(d->ticket, 0, kMaxSub * sizeof(unsigned), arena.stream()));
  return ASCI_OK;
}

static int dots(const double *V, size_t ld, int m, const double *b, size_t n,
                const DotScratch &d, double *out, int s1, double *out2, int s2, cudaStream_t s) {
  const int nblk = (int)std::min<size_t>(kDotBlocks, std::max<size_t>(1, (n + 1023) / 1024));
  k_dots<<<dim3(nblk, m), kDotThreads, 0, s>>>(V, ld, b, n, d.part, d.ticket, out, s1, out2, s2);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

template <int MODE>
static int run_pass(const PassArgs &A, unsigned blocks, cudaStream_t s) {
  auto *k = A.m <= 8 ? k_pass<MODE, 8> : (A.m <= 16 ? k_pass<MODE, 16> : k_pass<MODE, 32>);
  k<<<blocks, kPassThreads, 0, s>>>(A);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

struct DavidsonResult {
  double energy = 0.0, residual = 0.0;
  int iterations = 0;
  bool converged = false;
};

// Algorithm 5 on one device (see the file comment); vec receives the unit Ritz
// vector with its largest component positive.
static int davidson(const Csr &H, const double *diag, const double *guess,
                    const asci_davidson_opts &o, double *vec, DavidsonResult *res, Arena &arena) {
  cudaStream_t s = arena.stream();
  const size_t n = H.n;
  const int mmax = (int)std::min<size_t>((size_t)o.max_subspace, n);
  const unsigned gb = blocks_for(n, 256);
  const int keep = std::min(kKeep, mmax - 1);  // Ritz vectors kept at a restart
  double *V, *W, *Hs, *Ct, *th, *h, *sc, *x, *pass_part;
  unsigned *pass_ticket;
  float *Qw;
  DavState *st;
  DotScratch part;
  ASCI_TRY(arena.alloc(&V, ((size_t)mmax + 1) * n));  // the last correction has a place too
  ASCI_TRY(arena.alloc(&W, (size_t)mmax * n));
  ASCI_TRY(arena.alloc(&Hs, (size_t)kMaxSub * kMaxSub));
  ASCI_TRY(arena.alloc(&Ct, (size_t)kMaxSub * kMaxSub));
  ASCI_TRY(arena.alloc(&th, kMaxSub));
  ASCI_TRY(arena.alloc(&h, kMaxSub));
  ASCI_TRY(dot_scratch(&part, arena));
  ASCI_TRY(arena.alloc(&sc, 4));  // |v|^2, sign
  ASCI_TRY(arena.alloc(&x, n));
  ASCI_TRY(arena.alloc(&pass_part, (size_t)(kMaxSub + 1) * kPassBlocks));
  ASCI_TRY(arena.alloc(&pass_ticket, 1));
  ASCI_TRY(arena.alloc(&Qw, (size_t)kMaxSub * kMaxSub));
  ASCI_TRY(arena.alloc(&st, 1));
  ASCI_TRY_CUDA(cudaMemsetAsync(Hs, 0, sizeof(double) * kMaxSub * kMaxSub, s));
  ASCI_TRY_CUDA(cudaMemsetAsync(pass_ticket, 0, sizeof(unsigned), s));
  ASCI_TRY_CUDA(cudaMemsetAsync(st, 0, sizeof(DavState), s));
  // v0: the guess, or the unit vector of the smallest H_ii; normalised
  if (guess) {
    ASCI_TRY_CUDA(cudaMemcpyAsync(V, guess, n * sizeof(double), cudaMemcpyDefault, s));
  } else {
    k_unit<<<1, 256, 0, s>>>(V, n, diag);
    ASCI_CHECK_LAUNCH();
  }
  ASCI_TRY(dots(V, n, 1, V, n, part, sc + 2, 1, nullptr, 0, s));
  double g2 = 0.0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&g2, sc + 2, sizeof(double), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  if (!(g2 > 0.0) || !std::isfinite(g2)) {
    record_error("Davidson guess is zero or not finite", __FILE__, __LINE__);
    return ASCI_EINVAL;
  }
  k_inverse_norm<<<1, 1, 0, s>>>(sc + 2, &st->scale[0]);
  ASCI_CHECK_LAUNCH();
  const int *stop = &st->stop;
  const unsigned pb = blocks_for(n, kPassThreads, kPassBlocks);
  auto pass_args = [&](int m, int iter) {
    PassArgs A{};
    A.T = V;
    A.W = W;
    A.n = n;
    A.m = m;
    A.keep = keep;
    A.theta = th;
    A.diag = diag;
    A.t = V;
    A.precondition = iter > 1;
    A.iter = iter;
    A.tol = o.tol;
    A.Hs = Hs;
    A.h = h;
    A.part = pass_part;
    A.ticket = pass_ticket;
    A.st = st;
    return A;
  };
  // Iterations are enqueued kAhead at a time between two looks at the state:
  // the host's round trip is paid once for them, and those behind the one that
  // stopped return at once.
  constexpr int kAhead = 8;
  struct Step {
    int m;
    bool restarted;
  };
  std::vector<Step> steps(1);  // steps[i]: product i (1-based)
  int m = 1, it = 0;
  DavState hst{};
  for (bool more = true; more;) {
    for (int a = 0; a < kAhead && more; ++a) {
      // the newest basis vector's product and column of V^T H V
      ASCI_TRY(spmv(H, V + (size_t)(m - 1) * n, W + (size_t)(m - 1) * n, s, stop));
      ++it;
      const bool restart = m == mmax && (size_t)m < n;
      steps.push_back(Step{m, restart});
      PassArgs A = pass_args(m, it);
      ASCI_TRY(run_pass<kProject>(A, pb, s));
      k_small_eig<<<1, kEigThreads, 0, s>>>(Hs, m, restart ? keep : 1, it > 1 && !steps[it - 1].restarted,
                                            Qw, th, Ct, stop);
      ASCI_CHECK_LAUNCH();
      A.coef = Ct;
      A.t = V + (size_t)(restart ? keep : m) * n;
      if (restart) {  // thick restart: the `keep` lowest Ritz vectors and their products
        ASCI_TRY(run_pass<kRestart>(A, pb, s));
        k_restart_hs<<<1, 256, 0, s>>>(Hs, th, keep, stop);
        ASCI_CHECK_LAUNCH();
        m = keep;
      } else {
        ASCI_TRY(run_pass<kRitz>(A, pb, s));
      }
      if (it >= o.max_iter || (size_t)steps[it].m >= n) {
        more = false;
        break;
      }
      // the correction, orthogonalised by two passes of classical Gram-Schmidt
      A.m = m;
      A.coef = h;
      ASCI_TRY(run_pass<kOrth1>(A, pb, s));
      ASCI_TRY(run_pass<kOrth2>(A, pb, s));
      ++m;
    }
    ASCI_TRY_CUDA(cudaMemcpyAsync(&hst, st, sizeof(hst), cudaMemcpyDeviceToHost, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    if (hst.stop) more = false;
  }
  if (hst.stop == kStopBad) {
    record_error("Davidson produced a non-finite value", __FILE__, __LINE__);
    return ASCI_ECUDA;
  }
  const Step fin = steps[hst.iter];
  const double theta = hst.theta, rn = std::sqrt(std::max(hst.res2, 0.0));
  res->iterations = hst.iter;
  res->converged = rn <= o.tol || (size_t)fin.m >= n;
  // the Ritz vector of the last residual: a restart left it in V_0
  if (fin.restarted) {
    x = V;
  } else {
    k_combine<<<gb, 256, 0, s>>>(V, n, fin.m, Ct, st->scale, n, x);
    ASCI_CHECK_LAUNCH();
  }
  // unit Ritz vector, largest component positive
  {
    const int nb = (int)std::min<size_t>(296, std::max<size_t>(1, (n + 255) / 256));
    double *bval;
    unsigned long long *bidx;
    ASCI_TRY(arena.alloc(&bval, nb));
    ASCI_TRY(arena.alloc(&bidx, nb));
    ASCI_TRY(dots(x, n, 1, x, n, part, sc + 2, 1, nullptr, 0, s));
    k_normalize<<<gb, 256, 0, s>>>(x, n, sc + 2);
    ASCI_CHECK_LAUNCH();
    k_absmax_part<<<nb, 256, 0, s>>>(x, n, bval, bidx);
    ASCI_CHECK_LAUNCH();
    k_absmax_sign<<<1, 256, 0, s>>>(bval, bidx, nb, x, sc + 3);
    ASCI_CHECK_LAUNCH();
    k_scale_by<<<gb, 256, 0, s>>>(x, n, sc + 3);
    ASCI_CHECK_LAUNCH();
    ASCI_TRY_CUDA(cudaMemcpyAsync(vec, x, n * sizeof(double), cudaMemcpyDefault, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  }
  res->energy = theta;
  res->residual = rn;
  return ASCI_OK;
}

static int check_davidson_opts(const asci_davidson_opts &o) {
  if (o.max_subspace < 2 || o.max_subspace > kMaxSub || o.max_iter < 1 || !(o.tol >= 0.0) ||
      !std::isfinite(o.tol))
    return ASCI_EINVAL;
  return ASCI_OK;
}

// Packed keys of a determinant list, validated (range, counts, duplicates);
// na / nb from the first determinant.
static int det_keys(const asci_det *dets, size_t n, int norb, uint64_t *keys, int *na, int *nb,
                    Arena &arena) {
  cudaStream_t s = arena.stream();
  asci_det d0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&d0, dets, sizeof(d0), cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  *na = __builtin_popcountll(d0.alpha);
  *nb = __builtin_popcountll(d0.beta);
  unsigned *err;
  uint64_t *sk, *sk_alt;
  ASCI_TRY(arena.alloc(&err, 1));
  ASCI_TRY(arena.alloc(&sk, n));
  ASCI_TRY(arena.alloc(&sk_alt, n));
  ASCI_TRY_CUDA(cudaMemsetAsync(err, 0, sizeof(unsigned), s));
  k_det_keys<<<blocks_for(n, 256), 256, 0, s>>>(dets, n, norb, *na, *nb, keys, err);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaMemcpyAsync(sk, keys, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
  ASCI_TRY(radix_sort_u64_varying(&sk, &sk_alt, n, 0, 64, key_bits(norb), arena));
  k_adjacent_equal<<<blocks_for(n, 256), 256, 0, s>>>(sk, n, err);
  ASCI_CHECK_LAUNCH();
  unsigned herr = 0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  if (herr) {
    record_error(herr & kDuplicate  ? "duplicate determinants"
                 : herr & kBadCount ? "determinants with different electron counts"
                                    : "determinant bits at or above norb",
                 __FILE__, __LINE__);
    return ASCI_EINVAL;
  }
  return ASCI_OK;
}

static int stage_tables(const asci_ints *ints, int na, int nb, Arena &arena, DevInts *I) {
  const size_t n = (size_t)ints->norb;
  const double *h1, *eri;
  ASCI_TRY(to_device(ints->h1, n * n, &h1, arena));
  ASCI_TRY(to_device(ints->eri, n * n * n * n, &eri, arena));
  unsigned *err;
  ASCI_TRY(arena.alloc(&err, 1));
  cudaStream_t s = arena.stream();
  ASCI_TRY_CUDA(cudaMemsetAsync(err, 0, sizeof(unsigned), s));
  k_finite<<<blocks_for(n * n, 256), 256, 0, s>>>(h1, n * n, err);
  ASCI_CHECK_LAUNCH();
  k_finite<<<blocks_for(n * n * n * n, 256), 256, 0, s>>>(eri, n * n * n * n, err);
  ASCI_CHECK_LAUNCH();
  unsigned herr = 0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&herr, err, sizeof(herr), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  if (herr || !std::isfinite(ints->ecore)) {
    record_error("non-finite integral", __FILE__, __LINE__);
    return ASCI_EINVAL;
  }
  return build_tables(h1, eri, (int)n, na, nb, ints->ecore, false, arena, I);
}

// H over key-ordered packed keys, allocated in the arena.
static int ham_build(const DevInts &I, const uint64_t *keys, size_t n, Arena &arena, Csr *H,
                     double **diag_out) {
  double *diag;
  int64_t *rp;
  ASCI_TRY(arena.alloc(&diag, n));
  ASCI_TRY(arena.alloc(&rp, n + 1));
  ASCI_TRY(diagonal_packed(I, keys, n, diag, arena));
  BetaGraph bg;
  ASCI_TRY(beta_graph(keys, (uint32_t)n, I, &bg, arena));
  size_t nnz = 0;
  ASCI_TRY(ham_count(I, keys, (uint32_t)n, diag, bg, rp, &nnz, arena));
  int32_t *col;
  double *val;
  ASCI_TRY(arena.alloc(&col, nnz));
  ASCI_TRY(arena.alloc(&val, nnz));
  ASCI_TRY(ham_fill(I, keys, (uint32_t)n, diag, bg, rp, col, val, arena));
  H->row_ptr = rp;
  H->col = col;
  H->val = val;
  H->n = n;
  *diag_out = diag;
  return ASCI_OK;
}

static size_t csr_nnz(const Csr &H, cudaStream_t s) {
  int64_t e = 0;
  if (cudaMemcpyAsync(&e, H.row_ptr + H.n, sizeof(e), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return 0;
  return (size_t)e;
}

// The ASCI loop (Algorithm 1); see asci_loop in the public header.
static int loop_impl(const asci_det *dets_in, const double *coeffs_in, size_t nd,
                     const asci_ints *ints, const asci_loop_opts &o, asci_det *out_dets,
                     double *out_coeffs, size_t *out_n, double *energy, asci_loop_stats *st,
                     cudaStream_t s) {
  Arena arena(s);
  const int norb = ints->norb;
  const asci_det *dets;
  const double *coeffs;
  ASCI_TRY(to_device(dets_in, nd, &dets, arena));
  ASCI_TRY(to_device(coeffs_in, nd, &coeffs, arena));
  uint64_t *keys, *keys_alt;
  double *c, *c_alt;
  int na = 0, nb = 0;
  ASCI_TRY(arena.alloc(&keys, nd));
  ASCI_TRY(arena.alloc(&keys_alt, nd));
  ASCI_TRY(det_keys(dets, nd, norb, keys, &na, &nb, arena));
  DevInts I;
  ASCI_TRY(stage_tables(ints, na, nb, arena, &I));
  const double *h1d, *erid;
  ASCI_TRY(to_device(ints->h1, (size_t)norb * norb, &h1d, arena));
  ASCI_TRY(to_device(ints->eri, (size_t)norb * norb * norb * norb, &erid, arena));
  asci_ints dints = *ints;
  dints.h1 = h1d;
  dints.eri = erid;
  // the start in key order
  ASCI_TRY(arena.alloc(&c, nd));
  ASCI_TRY(arena.alloc(&c_alt, nd));
  ASCI_TRY_CUDA(cudaMemcpyAsync(c, coeffs, nd * sizeof(double), cudaMemcpyDeviceToDevice, s));
  const uint64_t used = key_bits(norb);
  ASCI_TRY(radix_sort_u64_f64(&keys, &keys_alt, &c, &c_alt, nd, 0, 64, arena, &used));
  double *sc;
  DotScratch part;
  ASCI_TRY(dot_scratch(&part, arena));
  ASCI_TRY(arena.alloc(&sc, 2));
  // E_0 = c.Hc / c.c on the start
  double E = 0.0;
  {
    Arena a2(s);
    Csr H;
    double *diag, *y;
    ASCI_TRY(ham_build(I, keys, nd, a2, &H, &diag));
    ASCI_TRY(a2.alloc(&y, nd));
    ASCI_TRY(spmv(H, c, y, s));
    ASCI_TRY(dots(c, nd, 1, y, nd, part, sc, 1, nullptr, 0, s));
    ASCI_TRY(dots(c, nd, 1, c, nd, part, sc + 1, 1, nullptr, 0, s));
    double hs[2];
    ASCI_TRY_CUDA(cudaMemcpyAsync(hs, sc, sizeof(hs), cudaMemcpyDeviceToHost, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    if (!(hs[1] > 0.0)) {
      record_error("start coefficients are all zero", __FILE__, __LINE__);
      return ASCI_EINVAL;
    }
    E = hs[0] / hs[1];
  }
  if (st) st->start_energy = E;
  size_t m = nd;
  // per-step buffers live in their own arena; the current wavefunction is
  // carried between steps in buffers of the loop's arena
  uint64_t *cur_k = keys;
  double *cur_c = c;
  const size_t cap = std::max(nd, (size_t)o.ntdets);
  uint64_t *buf_k[2];
  double *buf_c[2];
  for (int b = 0; b < 2; ++b) {
    ASCI_TRY(arena.alloc(&buf_k[b], cap));
    ASCI_TRY(arena.alloc(&buf_c[b], cap));
  }
  int which = 0;
  for (int step = 0; step < o.max_steps; ++step) {
    Arena sa(s);
    StageTimer tm(s);
    double t_search = 0.0, t_build = 0.0, t_dav = 0.0;
    // 1. search from (psi_k, c_k, E_k)
    tm.start();
    asci_det *pd, *cand;
    double *cs;
    ASCI_TRY(sa.alloc(&pd, m));
    ASCI_TRY(sa.alloc(&cand, o.ntdets));
    ASCI_TRY(sa.alloc(&cs, o.ntdets));
    k_keys_to_dets<<<blocks_for(m, 256), 256, 0, s>>>(cur_k, m, pd);
    ASCI_CHECK_LAUNCH();
    size_t U = 0;
    asci_opts so = o.search;
    ASCI_TRY(asci_search(pd, cur_c, m, E, &dints, std::min<size_t>(o.ncdets, m), o.ntdets, &so,
                         cand, cs, &U, nullptr, s));
    if (U) {  // E_k equal to a candidate's H_ii leaves its score undefined
      unsigned *ferr;
      ASCI_TRY(sa.alloc(&ferr, 1));
      ASCI_TRY_CUDA(cudaMemsetAsync(ferr, 0, sizeof(unsigned), s));
      k_finite<<<blocks_for(U, 256), 256, 0, s>>>(cs, U, ferr);
      ASCI_CHECK_LAUNCH();
      unsigned hf = 0;
      ASCI_TRY_CUDA(cudaMemcpyAsync(&hf, ferr, sizeof(hf), cudaMemcpyDeviceToHost, s));
      ASCI_TRY_CUDA(cudaStreamSynchronize(s));
      if (hf) {
        record_error("a candidate's score is not finite (E equals its H_ii)", __FILE__, __LINE__);
        return ASCI_EINVAL;
      }
    }
    // 2. merge: psi_k valued by c, candidates by S; top ntdets, key order
    const size_t tot = m + U;
    uint64_t *uk, *sel_k, *sel_k_alt;
    double *uv, *sel_v, *sel_v_alt;
    ASCI_TRY(sa.alloc(&uk, tot));
    ASCI_TRY(sa.alloc(&uv, tot));
    ASCI_TRY_CUDA(cudaMemcpyAsync(uk, cur_k, m * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
    ASCI_TRY_CUDA(cudaMemcpyAsync(uv, cur_c, m * sizeof(double), cudaMemcpyDeviceToDevice, s));
    if (U) {
      k_pack_dets<<<blocks_for(U, 256), 256, 0, s>>>(cand, U, uk + m);
      ASCI_CHECK_LAUNCH();
      ASCI_TRY_CUDA(cudaMemcpyAsync(uv + m, cs, U * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    const size_t keep = std::min<size_t>(tot, o.ntdets);
    ASCI_TRY(sa.alloc(&sel_k, keep));
    ASCI_TRY(sa.alloc(&sel_v, keep));
    ASCI_TRY(sa.alloc(&sel_k_alt, keep));
    ASCI_TRY(sa.alloc(&sel_v_alt, keep));
    size_t nsel = 0;
    ASCI_TRY(select_topn_packed(uk, uv, tot, o.ntdets, sel_k, sel_v, &nsel, sa));
    ASCI_TRY(radix_sort_u64_f64(&sel_k, &sel_k_alt, &sel_v, &sel_v_alt, nsel, 0, 64, sa, &used));
    // determinants that entered (selected keys absent from psi_k)
    unsigned long long entered = 0;
    {
      unsigned long long *dc;
      ASCI_TRY(sa.alloc(&dc, 1));
      ASCI_TRY_CUDA(cudaMemsetAsync(dc, 0, sizeof(*dc), s));
      k_count_missing<<<blocks_for(nsel, 256), 256, 0, s>>>(sel_k, nsel, cur_k, m, dc);
      ASCI_CHECK_LAUNCH();
      ASCI_TRY_CUDA(cudaMemcpyAsync(&entered, dc, sizeof(entered), cudaMemcpyDeviceToHost, s));
      ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    }
    const bool changed = nsel != m || entered != 0;
    tm.stop(&t_search);
    // 3. H on the new space and its lowest eigenpair
    tm.start();
    Csr H;
    double *diag;
    ASCI_TRY(ham_build(I, sel_k, nsel, sa, &H, &diag));
    tm.stop(&t_build);
    tm.start();
    DavidsonResult dr;
    double *nc = buf_c[which];
    ASCI_TRY(davidson(H, diag, sel_v, o.davidson, nc, &dr, sa));
    tm.stop(&t_dav);
    tm.read();
    if (!dr.converged) {
      record_error("Davidson did not converge within max_iter", __FILE__, __LINE__);
      return ASCI_ETIMEOUT;
    }
    ASCI_TRY_CUDA(cudaMemcpyAsync(buf_k[which], sel_k, nsel * sizeof(uint64_t),
                                  cudaMemcpyDeviceToDevice, s));
    if (st) {
      st->energy[step] = dr.energy;
      st->ndets[step] = nsel;
      st->nnz[step] = csr_nnz(H, s);
      st->davidson_iters[step] = dr.iterations;
      st->t_search[step] = t_search;
      st->t_hamiltonian[step] = t_build;
      st->t_davidson[step] = t_dav;
      st->new_dets[step] = entered;
      st->steps = step + 1;
    }
    const double Eold = E;
    E = dr.energy;
    cur_k = buf_k[which];
    cur_c = buf_c[which];
    m = nsel;
    which ^= 1;
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    if (std::fabs(E - Eold) <= o.etol || !changed) break;
  }
  // outputs: the final space in key order and its vector
  asci_det *od;
  double *oc;
  ASCI_TRY(out_buffer(out_dets, m, &od, arena));
  ASCI_TRY(out_buffer(out_coeffs, m, &oc, arena));
  k_keys_to_dets<<<blocks_for(m, 256), 256, 0, s>>>(cur_k, m, od);
  ASCI_CHECK_LAUNCH();
  if (oc != cur_c)
    ASCI_TRY_CUDA(cudaMemcpyAsync(oc, cur_c, m * sizeof(double), cudaMemcpyDeviceToDevice, s));
  ASCI_TRY(finish_out(out_dets, od, m, s));
  ASCI_TRY(finish_out(out_coeffs, oc, m, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  *out_n = m;
  *energy = E;
  return ASCI_OK;
}

}  // namespace asci

using namespace asci;

extern "C" {

void asci_default_davidson_opts(asci_davidson_opts *o) {
  if (!o) return;
  o->max_subspace = 16;
  o->max_iter = 300;
  o->tol = 1e-8;
}

void asci_default_loop_opts(asci_loop_opts *o) {
  if (!o) return;
  o->ncdets = 10000;
  o->ntdets = 100000;
  o->max_steps = 8;
  o->etol = 1e-6;
  asci_default_opts(&o->search);
  asci_default_davidson_opts(&o->davidson);
}

int asci_hamiltonian(const asci_det *dets, size_t n, const asci_ints *ints, int64_t *row_ptr,
                     int32_t *col, double *val, size_t capacity, size_t *nnz,
                     void *cuda_stream) {
  if (nnz) *nnz = 0;
  if (!dets || !ints || !ints->h1 || !ints->eri || !row_ptr || !nnz) return ASCI_EINVAL;
  if (capacity && (!col || !val)) return ASCI_EINVAL;
  if (ints->norb < 1 || ints->norb > 32 || n == 0 || n >= (1ull << 31)) return ASCI_EINVAL;
  clear_last_error();
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Arena arena(s);
  const asci_det *dd;
  ASCI_TRY(to_device(dets, n, &dd, arena));
  uint64_t *keys, *keys_alt;
  uint32_t *perm, *perm_alt;
  int na, nb;
  ASCI_TRY(arena.alloc(&keys, n));
  ASCI_TRY(arena.alloc(&keys_alt, n));
  ASCI_TRY(arena.alloc(&perm, n));
  ASCI_TRY(arena.alloc(&perm_alt, n));
  ASCI_TRY(det_keys(dd, n, ints->norb, keys, &na, &nb, arena));
  DevInts I;
  ASCI_TRY(stage_tables(ints, na, nb, arena, &I));
  // key order, and whether the caller's order already is key order
  k_iota<<<blocks_for(n, 256), 256, 0, s>>>(perm, (uint32_t)n);
  ASCI_CHECK_LAUNCH();
  const uint64_t used = key_bits(ints->norb);
  ASCI_TRY(radix_sort_u64_u32(&keys, &keys_alt, &perm, &perm_alt, n, 0, 64, arena, &used));
  unsigned *flag, hflag = 0;
  ASCI_TRY(arena.alloc(&flag, 1));
  ASCI_TRY_CUDA(cudaMemsetAsync(flag, 0, sizeof(unsigned), s));
  k_not_identity<<<blocks_for(n, 256), 256, 0, s>>>(perm, (uint32_t)n, flag);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY_CUDA(cudaMemcpyAsync(&hflag, flag, sizeof(hflag), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  double *diag;
  ASCI_TRY(arena.alloc(&diag, n));
  ASCI_TRY(diagonal_packed(I, keys, n, diag, arena));
  BetaGraph bg;
  ASCI_TRY(beta_graph(keys, (uint32_t)n, I, &bg, arena));
  const bool same_order = hflag == 0;
  int64_t *rp, *urp;
  ASCI_TRY(out_buffer(row_ptr, n + 1, &urp, arena));
  if (same_order) rp = urp;
  else ASCI_TRY(arena.alloc(&rp, n + 1));
  size_t total = 0;
  ASCI_TRY(ham_count(I, keys, (uint32_t)n, diag, bg, rp, &total, arena));
  if (!same_order) {  // row pointers in the caller's order
    ASCI_TRY_CUDA(cudaMemsetAsync(urp + n, 0, sizeof(int64_t), s));
    k_user_counts<<<blocks_for(n, 256), 256, 0, s>>>(rp, perm, (uint32_t)n, urp);
    ASCI_CHECK_LAUNCH();
    ASCI_TRY(scan_exclusive_u64(reinterpret_cast<uint64_t *>(urp),
                                reinterpret_cast<uint64_t *>(urp), n + 1, arena));
  }
  if (total <= capacity) {
    int32_t *dc;
    double *dv;
    ASCI_TRY(out_buffer(col, total, &dc, arena));
    ASCI_TRY(out_buffer(val, total, &dv, arena));
    if (same_order) {
      ASCI_TRY(ham_fill(I, keys, (uint32_t)n, diag, bg, rp, dc, dv, arena));
    } else {
      // build in key order, then sort the entries on (caller row, caller column)
      if (total >= (1ull << 32)) {
        record_error("too many elements to reorder; pass the determinants in key order",
                     __FILE__, __LINE__);
        return ASCI_ENOMEM;
      }
      int32_t *kc;
      double *kv, *kv_alt;
      uint64_t *ek, *ek_alt;
      ASCI_TRY(arena.alloc(&kc, total));
      ASCI_TRY(arena.alloc(&kv, total));
      ASCI_TRY(arena.alloc(&kv_alt, total));
      ASCI_TRY(arena.alloc(&ek, total));
      ASCI_TRY(arena.alloc(&ek_alt, total));
      ASCI_TRY(ham_fill(I, keys, (uint32_t)n, diag, bg, rp, kc, kv, arena));
      k_user_entries<<<row_blocks((uint32_t)n), 256, 0, s>>>(rp, kc, perm, (uint32_t)n, ek);
      ASCI_CHECK_LAUNCH();
      ASCI_TRY(radix_sort_u64_f64(&ek, &ek_alt, &kv, &kv_alt, total, 0, 64, arena));
      k_low_cols<<<blocks_for(total, 256), 256, 0, s>>>(ek, total, dc);
      ASCI_CHECK_LAUNCH();
      ASCI_TRY_CUDA(cudaMemcpyAsync(dv, kv, total * sizeof(double), cudaMemcpyDeviceToDevice, s));
    }
    ASCI_TRY(finish_out(col, dc, total, s));
    ASCI_TRY(finish_out(val, dv, total, s));
  }
  ASCI_TRY(finish_out(row_ptr, urp, n + 1, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  *nnz = total;
  return ASCI_OK;
}

int asci_spmv(const int64_t *row_ptr, const int32_t *col, const double *val, size_t n,
              const double *x, double *y, void *cuda_stream) {
  if (!row_ptr || !col || !val || !x || !y || n >= (1ull << 31)) return ASCI_EINVAL;
  if (n == 0) return ASCI_OK;
  clear_last_error();
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Arena arena(s);
  const int64_t *rp;
  ASCI_TRY(to_device(row_ptr, n + 1, &rp, arena));
  int64_t nnz = 0;  // needed only to stage host arrays
  if (!is_device_ptr(col) || !is_device_ptr(val)) {
    ASCI_TRY_CUDA(cudaMemcpyAsync(&nnz, rp + n, sizeof(nnz), cudaMemcpyDefault, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  }
  const int32_t *dc;
  const double *dv, *dx;
  double *dy;
  ASCI_TRY(to_device(col, (size_t)nnz, &dc, arena));
  ASCI_TRY(to_device(val, (size_t)nnz, &dv, arena));
  ASCI_TRY(to_device(x, n, &dx, arena));
  ASCI_TRY(out_buffer(y, n, &dy, arena));
  Csr H = {rp, dc, dv, n};
  ASCI_TRY(spmv(H, dx, dy, s));
  ASCI_TRY(finish_out(y, dy, n, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  return ASCI_OK;
}

int asci_davidson(const int64_t *row_ptr, const int32_t *col, const double *val, size_t n,
                  const double *guess, const asci_davidson_opts *opts, double *energy,
                  double *vec, int32_t *iterations, double *residual, void *cuda_stream) {
  if (!row_ptr || !col || !val || !energy || !vec || n == 0 || n >= (1ull << 31))
    return ASCI_EINVAL;
  asci_davidson_opts o;
  asci_default_davidson_opts(&o);
  if (opts) o = *opts;
  ASCI_TRY(check_davidson_opts(o));
  clear_last_error();
  cudaStream_t s = (cudaStream_t)cuda_stream;
  Arena arena(s);
  const int64_t *rp;
  ASCI_TRY(to_device(row_ptr, n + 1, &rp, arena));
  int64_t nnz = 0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&nnz, rp + n, sizeof(nnz), cudaMemcpyDefault, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  const int32_t *dc;
  const double *dv, *dg = nullptr;
  ASCI_TRY(to_device(col, (size_t)nnz, &dc, arena));
  ASCI_TRY(to_device(val, (size_t)nnz, &dv, arena));
  if (guess) ASCI_TRY(to_device(guess, n, &dg, arena));
  Csr H = {rp, dc, dv, n};
  double *diag;
  ASCI_TRY(arena.alloc(&diag, n));
  k_csr_diag<<<blocks_for(n * 32, 256), 256, 0, s>>>(rp, dc, dv, (uint32_t)n, diag);
  ASCI_CHECK_LAUNCH();
  DavidsonResult r;
  ASCI_TRY(davidson(H, diag, dg, o, vec, &r, arena));
  *energy = r.energy;
  if (iterations) *iterations = r.iterations;
  if (residual) *residual = r.residual;
  if (!r.converged) {
    record_error("Davidson did not converge within max_iter", __FILE__, __LINE__);
    return ASCI_ETIMEOUT;
  }
  return ASCI_OK;
}

int asci_loop(const asci_det *dets, const double *coeffs, size_t ndets, const asci_ints *ints,
              const asci_loop_opts *opts, asci_det *out_dets, double *out_coeffs,
              size_t capacity, size_t *out_n, double *energy, asci_loop_stats *stats,
              void *cuda_stream) {
  if (out_n) *out_n = 0;
  if (stats) memset(stats, 0, sizeof(*stats));
  if (!dets || !coeffs || !ints || !ints->h1 || !ints->eri || !opts || !out_dets ||
      !out_coeffs || !out_n || !energy)
    return ASCI_EINVAL;
  const asci_loop_opts &o = *opts;
  if (ints->norb < 1 || ints->norb > 32 || ndets == 0 || ndets >= (1ull << 31) || o.ncdets == 0 ||
      o.ntdets == 0 || o.ntdets >= (1ull << 31) || capacity < o.ntdets || o.max_steps < 1 ||
      o.max_steps > ASCI_LOOP_MAX_STEPS || !(o.etol >= 0.0))
    return ASCI_EINVAL;
  ASCI_TRY(check_davidson_opts(o.davidson));
  clear_last_error();
  int r = loop_impl(dets, coeffs, ndets, ints, o, out_dets, out_coeffs, out_n, energy, stats,
                    (cudaStream_t)cuda_stream);
  if (r != ASCI_OK) *out_n = 0;
  return r;
}

}  // extern "C"
