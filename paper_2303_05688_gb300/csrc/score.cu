// Sort-and-accumulate (Sec. 2.2), the diagonal H_ii and the score of Eq. 1,
// exclusion of psi, and the top-N selection that replaces a full sort.
#include <algorithm>
#include <cstring>

#include "asci_internal.cuh"

namespace asci {

namespace {

struct SelState {
  uint64_t pre[2];      // fixed bits of R_N: {hi, lo}
  uint64_t thr[2];      // entries with R <= thr are selected, once done
  uint64_t remaining;   // rank of R_N among the entries that match the prefix
  unsigned done, ticket;
};

// ------------------------- segmented accumulate ----------------------------

__global__ void k_heads(const uint64_t *keys, size_t n, uint32_t *head) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    head[i] = (i == 0 || keys[i] != keys[i - 1]) ? 1u : 0u;
}

__global__ void k_head_index(const uint32_t *head, const uint32_t *pos, size_t n,
                             uint32_t *head_idx) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (head[i]) head_idx[pos[i]] = (uint32_t)i;
}

// Sum of each run of equal keys, in input order (deterministic).
__global__ void k_segment_sum(const uint64_t *keys, const double *vals, size_t n,
                              const uint32_t *head_idx, size_t u, uint64_t *ukeys,
                              double *usums) {
  for (size_t s = (size_t)blockIdx.x * blockDim.x + threadIdx.x; s < u;
       s += (size_t)gridDim.x * blockDim.x) {
    size_t b = head_idx[s], e = (s + 1 < u) ? head_idx[s + 1] : n;
    double acc = 0.0;
    for (size_t i = b; i < e; ++i) acc += vals[i];
    ukeys[s] = keys[b];
    usums[s] = acc;
  }
}

// ------------------------------- diagonal ----------------------------------

__device__ double diag_value(const DevInts &I, uint32_t A, uint32_t B) {
  const int n = I.n;
  double s = I.ecore;
  for (uint32_t m = A; m; m &= m - 1) {
    const int p = __ffs(m) - 1;
    const double *jkp = I.jk + p * n, *jjp = I.jj + p * n;
    s += I.h1[p * n + p];
    for (uint32_t r = m & (m - 1); r; r &= r - 1) s += jkp[__ffs(r) - 1];
    for (uint32_t r = B; r; r &= r - 1) s += jjp[__ffs(r) - 1];
  }
  for (uint32_t m = B; m; m &= m - 1) {
    const int p = __ffs(m) - 1;
    const double *jkp = I.jk + p * n;
    s += I.h1[p * n + p];
    for (uint32_t r = m & (m - 1); r; r &= r - 1) s += jkp[__ffs(r) - 1];
  }
  return s;
}

__global__ void k_diag(DevInts I, const uint64_t *keys, size_t n, double *out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    uint64_t k = keys[i];
    out[i] = diag_value(I, key_alpha(k), key_beta(k));
  }
}

template <typename T>
__global__ void k_compact(const T *in, const uint32_t *keep, const uint32_t *pos, size_t n,
                          T *out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (keep[i]) out[pos[i]] = in[i];
}

// ------------------------------ selection ----------------------------------
//
// The rank of an entry is the 128-bit word R = (~bits(|S|), key): ascending R
// is |S| descending, then key ascending.  Keys are distinct, so R is too, and
// the top N are exactly the entries with R <= R_N.  R_N is found digit by digit
// from the most significant end (a radix select).

__device__ __forceinline__ void rank_words(uint64_t key, double s, uint64_t *hi, uint64_t *lo) {
  *hi = ~((uint64_t)__double_as_longlong(fabs(s)));
  *lo = key;
}

__global__ void k_select_hist(const uint64_t *keys, const double *scores, size_t n, int digit,
                              uint64_t pre_hi, uint64_t pre_lo, uint64_t m_hi, uint64_t m_lo,
                              unsigned long long *hist) {
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    uint64_t hi, lo;
    rank_words(keys[i], scores[i], &hi, &lo);
    if (((hi & m_hi) == pre_hi) && ((lo & m_lo) == pre_lo)) {
      uint32_t d = digit >= 8 ? (uint32_t)(hi >> ((digit - 8) * 8)) & 0xffu
                              : (uint32_t)(lo >> (digit * 8)) & 0xffu;
      atomicAdd(&h[d], 1u);
    }
  }
  __syncthreads();
  if (h[threadIdx.x]) atomicAdd(&hist[threadIdx.x], (unsigned long long)h[threadIdx.x]);
}

// Top-N selection on the device: the same digit choice with digits of 11 bits
// (six per word, the last of 9), made by the last block of each round, so that
// the rounds follow one another without the host.  A round whose selection is
// settled returns at once; the host enqueues all of them.  (With 8-bit digits
// and the choice on the host, a selection waited for a copy per digit: up to 16
// round trips, 0.4 ms.)  Lists of at most 16384 entries take one CTA instead.
constexpr int kSelBits = 11, kSelBins = 1 << kSelBits, kSelRounds = 12;
__host__ __device__ inline int sel_shift(int round) {
  const int d = round % 6;
  return d == 5 ? 0 : 64 - kSelBits * (d + 1);
}

// The state and the bins before the first round, for the n largest.
__global__ void k_select_init(SelState *st, uint32_t *hist, uint64_t n) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (i < kSelBins) hist[i] = 0;
  if (i > 0) return;
  SelState s{};
  s.remaining = n;
  *st = s;
}

__global__ void __launch_bounds__(256) k_select_round(const uint64_t *keys, const double *scores,
                                                      size_t n, int round, SelState *st,
                                                      uint32_t *hist) {
  __shared__ uint32_t h[kSelBins];
  __shared__ uint32_t part[256];
  __shared__ bool last;
  if (st->done) return;
  for (int i = threadIdx.x; i < kSelBins; i += 256) h[i] = 0;
  const uint64_t p_hi = st->pre[0], p_lo = st->pre[1];
  const int word = round / 6, sh = sel_shift(round);
  // the bits fixed so far: every higher digit of the word (and the high word)
  const int top = round % 6 == 0 ? 64 : sel_shift(round - 1);
  const uint64_t mask = top == 64 ? 0ull : ~0ull << top;
  const uint32_t bins = round % 6 == 5 ? 1u << 9 : (uint32_t)kSelBins;
  __syncthreads();
  // warp-uniform loop: equal digits of a warp are counted with one atomic
  // (the leading digits are the exponents, nearly all alike)
  const uint32_t lane = threadIdx.x & 31u;
  for (size_t i0 = (size_t)blockIdx.x * 256 + (threadIdx.x & ~31u); i0 < n;
       i0 += (size_t)gridDim.x * 256) {
    const size_t i = i0 + lane;
    uint32_t d = kSelBins;
    if (i < n) {
      const uint64_t hi = ~((uint64_t)__double_as_longlong(fabs(scores[i])));
      bool in;
      uint64_t w = hi;
      if (word == 0) {
        in = (hi & mask) == p_hi;
      } else {
        in = hi == p_hi;
        if (in) {
          w = keys[i];
          in = (w & mask) == p_lo;
        }
      }
      if (in) d = (uint32_t)(w >> sh) & (bins - 1u);
    }
    if (!__any_sync(0xffffffffu, d < (uint32_t)kSelBins)) continue;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    if (d < (uint32_t)kSelBins && (int)lane == __ffs(peers) - 1) atomicAdd(&h[d], __popc(peers));
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kSelBins; i += 256)
    if (h[i]) atomicAdd(&hist[i], h[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // thread t: bins [8 t, 8 t + 8); the bin that holds the remaining-th entry
  constexpr int kPer = kSelBins / 256;
  uint32_t c[kPer], own = 0;
  for (int k = 0; k < kPer; ++k) {
    c[k] = __ldcg(&hist[threadIdx.x * kPer + k]);
    hist[threadIdx.x * kPer + k] = 0;
    own += c[k];
  }
  part[threadIdx.x] = own;
  __syncthreads();
  for (int o = 1; o < 256; o <<= 1) {
    const uint32_t y = (int)threadIdx.x >= o ? part[threadIdx.x - o] : 0u;
    __syncthreads();
    part[threadIdx.x] += y;
    __syncthreads();
  }
  const uint64_t remaining = st->remaining;
  uint64_t below = part[threadIdx.x] - own;
  __syncthreads();
  if (threadIdx.x == 0) st->ticket = 0u;
  if (below < remaining && below + own >= remaining) {
    int k = 0;
    for (; k < kPer - 1 && below + c[k] < remaining; ++k) below += c[k];
    const uint64_t digit = (uint64_t)(threadIdx.x * kPer + k);
    const uint64_t pre = st->pre[word] | (digit << sh);
    st->pre[word] = pre;
    st->remaining = remaining - below;
    // the whole bin is selected: every lower bit of the threshold is set
    const bool whole = c[k] == remaining - below;
    if (whole || round == kSelRounds - 1) {
      const uint64_t low = whole ? ~(~0ull << sh) : 0ull;
      st->thr[0] = word == 0 ? pre | low : st->pre[0];
      st->thr[1] = word == 0 ? ~0ull : pre | low;
      st->done = 1;
    }
  }
}

// The whole selection of at most kSmallSelect entries by one CTA: the same
// digits, as many as it takes, then the selected entries in input order.
constexpr size_t kSmallSelect = 16384;

__global__ void __launch_bounds__(1024) k_select_small(const uint64_t *keys, const double *scores,
                                                       uint32_t n, uint32_t N, uint64_t *out_keys,
                                                       double *out_scores, SelState *st) {
  __shared__ uint32_t h[kSelBins];
  __shared__ uint32_t warp_sum[32];
  __shared__ uint64_t pre[2], thr[2];
  __shared__ uint32_t remaining, done;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
  if (tid == 0) {
    pre[0] = pre[1] = 0;
    remaining = N;
    done = 0;
  }
  // exclusive prefix of v over the CTA
  auto scan = [&](uint32_t v) {
    uint32_t x = v;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if ((int)lane >= o) x += y;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t w = warp_sum[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
        if ((int)lane >= o) w += y;
      }
      warp_sum[lane] = w;
    }
    __syncthreads();
    const uint32_t before = warp ? warp_sum[warp - 1] : 0u;
    return before + x - v;
  };
  for (int round = 0; round < kSelRounds; ++round) {
    for (uint32_t i = tid; i < kSelBins; i += 1024) h[i] = 0;
    __syncthreads();
    if (done) break;
    const int word = round / 6, sh = sel_shift(round);
    const int top = round % 6 == 0 ? 64 : sel_shift(round - 1);
    const uint64_t mask = top == 64 ? 0ull : ~0ull << top, p_hi = pre[0], p_lo = pre[1];
    const uint32_t bins = round % 6 == 5 ? 1u << 9 : (uint32_t)kSelBins;
    for (uint32_t i0 = tid & ~31u; i0 < n; i0 += 1024) {
      const uint32_t i = i0 + lane;
      uint32_t d = kSelBins;
      if (i < n) {
        const uint64_t hi = ~((uint64_t)__double_as_longlong(fabs(scores[i])));
        const uint64_t w = word == 0 ? hi : keys[i];
        if (word == 0 ? (hi & mask) == p_hi : (hi == p_hi && (w & mask) == p_lo))
          d = (uint32_t)(w >> sh) & (bins - 1u);
      }
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      if (d < (uint32_t)kSelBins && (int)lane == __ffs(peers) - 1) atomicAdd(&h[d], __popc(peers));
    }
    __syncthreads();
    const uint32_t c0 = h[2 * tid], c1 = h[2 * tid + 1], want = remaining;
    const uint32_t below = scan(c0 + c1);
    if (below < want && below + c0 + c1 >= want) {
      const bool second = below + c0 < want;
      const uint32_t under = below + (second ? c0 : 0u);
      const uint64_t p = pre[word] | ((uint64_t)(2 * tid + (second ? 1u : 0u)) << sh);
      const bool whole = (second ? c1 : c0) == want - under;
      pre[word] = p;
      remaining = want - under;
      if (whole || round == kSelRounds - 1) {
        const uint64_t low = whole ? ~(~0ull << sh) : 0ull;
        thr[0] = word == 0 ? p | low : pre[0];
        thr[1] = word == 0 ? ~0ull : p | low;
        done = 1;
      }
    }
    __syncthreads();
  }
  __syncthreads();
  const uint64_t t_hi = thr[0], t_lo = thr[1];
  uint32_t at = 0;
  for (uint32_t i0 = 0; i0 < n; i0 += 1024) {
    const uint32_t i = i0 + tid;
    bool in = false;
    if (i < n) {
      const uint64_t hi = ~((uint64_t)__double_as_longlong(fabs(scores[i])));
      in = hi < t_hi || (hi == t_hi && keys[i] <= t_lo);
    }
    const uint32_t pos = at + scan(in ? 1u : 0u);
    if (in && pos < N) {
      out_keys[pos] = keys[i];
      out_scores[pos] = scores[i];
    }
    at += warp_sum[31];
    __syncthreads();
  }
  if (tid == 0) {
    st->thr[0] = t_hi;
    st->thr[1] = t_lo;
  }
}

__global__ void k_select_marks(const uint64_t *keys, const double *scores, size_t n,
                               const SelState *st, uint32_t *flag) {
  const uint64_t t_hi = st->thr[0], t_lo = st->thr[1];
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t hi = ~((uint64_t)__double_as_longlong(fabs(scores[i])));
    flag[i] = (hi < t_hi || (hi == t_hi && keys[i] <= t_lo)) ? 1u : 0u;
  }
}

// Marked entries of both arrays, at most m of them.
__global__ void k_select_compact(const uint64_t *keys, const double *scores, const uint32_t *flag,
                                 const uint32_t *pos, size_t n, size_t m, uint64_t *out_keys,
                                 double *out_scores) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    if (flag[i] && pos[i] < m) {
      out_keys[pos[i]] = keys[i];
      out_scores[pos[i]] = scores[i];
    }
}

__global__ void k_select_flags(const uint64_t *keys, const double *scores, size_t n,
                               uint64_t t_hi, uint64_t t_lo, uint32_t *flag) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    uint64_t hi, lo;
    rank_words(keys[i], scores[i], &hi, &lo);
    flag[i] = (hi < t_hi || (hi == t_hi && lo <= t_lo)) ? 1u : 0u;
  }
}

inline unsigned grid_for(size_t n, unsigned cap = 152 * 16) {
  size_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  return (unsigned)(b < cap ? b : cap);
}

}  // namespace

int compact_u64(const uint64_t *in, const uint32_t *keep, const uint32_t *pos, size_t n,
                uint64_t *out, Arena &arena) {
  if (!n) return ASCI_OK;
  k_compact<uint64_t><<<grid_for(n), 256, 0, arena.stream()>>>(in, keep, pos, n, out);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

int compact_f64(const double *in, const uint32_t *keep, const uint32_t *pos, size_t n, double *out,
                Arena &arena) {
  if (!n) return ASCI_OK;
  k_compact<double><<<grid_for(n), 256, 0, arena.stream()>>>(in, keep, pos, n, out);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

// Number of kept entries = pos[n-1] + keep[n-1] (host read).
int kept_count(const uint32_t *keep, const uint32_t *pos, size_t n, size_t *host_count,
               Arena &arena) {
  *host_count = 0;
  if (!n) return ASCI_OK;
  uint32_t h[2];
  cudaStream_t s = arena.stream();
  ASCI_TRY_CUDA(cudaMemcpyAsync(&h[0], pos + n - 1, 4, cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaMemcpyAsync(&h[1], keep + n - 1, 4, cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  *host_count = (size_t)h[0] + h[1];
  return ASCI_OK;
}

int sort_accumulate(uint64_t **keys, uint64_t **keys_alt, double **vals, double **vals_alt,
                    size_t n, uint64_t *ukeys, double *usums, size_t *host_u, Arena &arena) {
  *host_u = 0;
  if (!n) return ASCI_OK;
  ASCI_TRY(radix_sort_u64_f64(keys, keys_alt, vals, vals_alt, n, 0, 64, arena));
  uint32_t *head, *pos, *head_idx;
  ASCI_TRY(arena.alloc(&head, n));
  ASCI_TRY(arena.alloc(&pos, n));
  cudaStream_t s = arena.stream();
  k_heads<<<grid_for(n), 256, 0, s>>>(*keys, n, head);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(scan_exclusive_u32(head, pos, n, arena));
  size_t u = 0;
  ASCI_TRY(kept_count(head, pos, n, &u, arena));
  ASCI_TRY(arena.alloc(&head_idx, u));
  k_head_index<<<grid_for(n), 256, 0, s>>>(head, pos, n, head_idx);
  ASCI_CHECK_LAUNCH();
  k_segment_sum<<<grid_for(u), 256, 0, s>>>(*keys, *vals, n, head_idx, u, ukeys, usums);
  ASCI_CHECK_LAUNCH();
  *host_u = u;
  return ASCI_OK;
}

int diagonal_packed(const DevInts &I, const uint64_t *keys, size_t n, double *out, Arena &arena) {
  if (!n) return ASCI_OK;
  k_diag<<<grid_for(n), 256, 0, arena.stream()>>>(I, keys, n, out);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

int select_topn_packed(const uint64_t *keys, const double *scores, size_t n, size_t N,
                       uint64_t *out_keys, double *out_scores, size_t *host_out_n,
                       Arena &arena, double *host_min) {
  *host_out_n = 0;
  if (!n || !N) return ASCI_OK;
  cudaStream_t s = arena.stream();
  const size_t m = std::min(n, N);
  *host_out_n = m;
  if (N >= n) {  // everything is selected
    ASCI_TRY_CUDA(cudaMemcpyAsync(out_keys, keys, n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, s));
    ASCI_TRY_CUDA(cudaMemcpyAsync(out_scores, scores, n * sizeof(double), cudaMemcpyDeviceToDevice,
                                  s));
    if (host_min) ASCI_TRY(abs_min(scores, n, host_min, arena));
    return ASCI_OK;
  }
  SelState *st;
  ASCI_TRY(arena.alloc(&st, 1));
  if (n <= kSmallSelect) {
    k_select_small<<<1, 1024, 0, s>>>(keys, scores, (uint32_t)n, (uint32_t)N, out_keys, out_scores,
                                      st);
    ASCI_CHECK_LAUNCH();
  } else {
    uint32_t *flag, *pos, *hist;
    ASCI_TRY(arena.alloc(&flag, n));
    ASCI_TRY(arena.alloc(&pos, n));
    ASCI_TRY(arena.alloc(&hist, (size_t)kSelBins));
    k_select_init<<<kSelBins / 256, 256, 0, s>>>(st, hist, N);
    ASCI_CHECK_LAUNCH();
    for (int round = 0; round < kSelRounds; ++round) {
      k_select_round<<<grid_for(n, 152 * 4), 256, 0, s>>>(keys, scores, n, round, st, hist);
      ASCI_CHECK_LAUNCH();
    }
    k_select_marks<<<grid_for(n), 256, 0, s>>>(keys, scores, n, st, flag);
    ASCI_CHECK_LAUNCH();
    ASCI_TRY(scan_exclusive_u32(flag, pos, n, arena));
    k_select_compact<<<grid_for(n), 256, 0, s>>>(keys, scores, flag, pos, n, m, out_keys,
                                                 out_scores);
    ASCI_CHECK_LAUNCH();
  }
  if (host_min) {
    // the selected entry of largest R has the smallest |S|: thr bounds it from
    // below (its free low bits are set)
    SelState done;
    ASCI_TRY_CUDA(cudaMemcpyAsync(&done, st, sizeof(done), cudaMemcpyDeviceToHost, s));
    ASCI_TRY_CUDA(cudaStreamSynchronize(s));
    const uint64_t bits = ~done.thr[0];
    memcpy(host_min, &bits, sizeof(bits));
  }
  return ASCI_OK;
}

// Building blocks of a selection across ranks: the histogram of one byte of
// the rank word over the entries that match a prefix, and the entries at or
// below a rank threshold.
int select_histogram(const uint64_t *keys, const double *scores, size_t n, int digit,
                     const uint64_t pre[2], const uint64_t msk[2], uint64_t hist[256],
                     Arena &arena) {
  cudaStream_t s = arena.stream();
  unsigned long long *dhist;
  ASCI_TRY(arena.alloc(&dhist, 256));
  ASCI_TRY_CUDA(cudaMemsetAsync(dhist, 0, 256 * sizeof(unsigned long long), s));
  if (n) {
    k_select_hist<<<grid_for(n), 256, 0, s>>>(keys, scores, n, digit, pre[0], pre[1], msk[0],
                                              msk[1], dhist);
    ASCI_CHECK_LAUNCH();
  }
  ASCI_TRY_CUDA(cudaMemcpyAsync(hist, dhist, 256 * sizeof(uint64_t), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  return ASCI_OK;
}

int select_below(const uint64_t *keys, const double *scores, size_t n, const uint64_t thr[2],
                 uint64_t *out_keys, double *out_scores, size_t *host_out_n, Arena &arena) {
  *host_out_n = 0;
  if (!n) return ASCI_OK;
  cudaStream_t s = arena.stream();
  uint32_t *flag, *pos;
  ASCI_TRY(arena.alloc(&flag, n));
  ASCI_TRY(arena.alloc(&pos, n));
  k_select_flags<<<grid_for(n), 256, 0, s>>>(keys, scores, n, thr[0], thr[1], flag);
  ASCI_CHECK_LAUNCH();
  ASCI_TRY(scan_exclusive_u32(flag, pos, n, arena));
  size_t m = 0;
  ASCI_TRY(kept_count(flag, pos, n, &m, arena));
  ASCI_TRY(compact_u64(keys, flag, pos, n, out_keys, arena));
  ASCI_TRY(compact_f64(scores, flag, pos, n, out_scores, arena));
  *host_out_n = m;
  return ASCI_OK;
}

}  // namespace asci
