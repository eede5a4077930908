// Device-wide primitives: exclusive scan and a stable LSD radix sort.
//
// The sort is the "sort" of the paper's sort-and-accumulate (Sec. 2.2); it is
// written for this library: 8-bit digits, one kernel that counts every digit of
// the keys, and one kernel per digit that ranks each tile's keys stably, learns
// from the tiles before it where its runs begin, and moves the keys.
#include "asci_internal.cuh"

namespace asci {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

template <typename T>
__device__ T block_exclusive_scan(T v, T *total) {
  __shared__ T warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    T y = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    T w = lane < nw ? warp_sums[lane] : T(0);
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      T y = __shfl_up_sync(0xffffffffu, w, d);
      if (lane >= d) w += y;
    }
    if (lane < nw) warp_sums[lane] = w;
  }
  __syncthreads();
  T warp_prefix = warp ? warp_sums[warp - 1] : T(0);
  if (total) *total = warp_sums[(blockDim.x >> 5) - 1];
  __syncthreads();
  return warp_prefix + x - v;
}

// Scan inputs: an array, or a value computed from each index.
template <typename T>
struct ArrayIn {
  const T *p;
  __device__ T operator()(size_t i) const { return p[i]; }
};

// Pairs of item i (the constraint-batched generation's item format, alpha
// operation in the low opbits, group above it): the beta singles and doubles
// for o = 0, the single itself and its alpha-beta doubles for an alpha
// single, one pair for an alpha double; times the group's core determinants.
// Index T (one past the end) is 0, so the scan's last entry is the total.
struct ItemWeightIn {
  const uint64_t *items;
  const uint32_t *grp_count;
  uint64_t T, npd0, npd1;
  uint32_t omask, sa;
  int opbits;
  __device__ uint64_t operator()(size_t i) const {
    if (i >= T) return 0;
    const uint32_t lo = (uint32_t)items[i];
    const uint32_t k = lo >> opbits, o = lo & omask;
    const uint64_t npd = (o == 0) ? npd0 : (o <= sa ? npd1 : 1ull);
    return npd * grp_count[k];
  }
};

// 1 where item i starts a new target alpha string (its high word changes);
// index T (one past the end) is 0, so the scan's last entry is the count.
struct ItemHeadIn {
  const uint64_t *items;
  uint64_t T;
  __device__ uint32_t operator()(size_t i) const {
    if (i >= T) return 0u;
    return (i == 0 || (items[i] >> 32) != (items[i - 1] >> 32)) ? 1u : 0u;
  }
};

// Shared-memory index of tile element e, padded by one element per 128 bytes
// so that the transposed pass (thread t on elements 16t .. 16t+15) falls on
// distinct banks: without the pad every thread of a warp hits one or two banks.
template <typename T>
__device__ __forceinline__ int scan_pad(int e) {
  return e + e / (int)(128 / sizeof(T));
}

__device__ __forceinline__ uint64_t ld_relaxed(const uint64_t *p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(uint64_t *p, uint64_t v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
constexpr uint32_t kLookLimit = 1u << 18;  // polls before a tile counts for itself

__device__ __forceinline__ uint64_t warp_sum(uint64_t v) {
  for (int d = 16; d; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// Exclusive scan in one pass, a tile per CTA: the single-pass scan with decoupled look
// back of Merrill and Garland (2016).  words[0] numbers the tiles in the
// order in which CTAs start; words[1 + t] is tile t's sum (below 2^62) under a
// state: 0 unknown, 1 the tile's own sum, 2 the sum of it and all before.  A tile
// publishes its sum, then its first warp adds up the tiles before it, 32 at a
// time, back to the nearest one that knows its prefix; those tiles are running or
// done and publish before they wait, so the wait ends.  Should one not answer
// within kLookLimit polls, the warp sums its input itself (in and out may be the
// same array: a tile writes only after it has published, so an input whose word
// is still unknown after it was read was read unchanged).
//
// Bound: memory and the look back's latency: 57.7 M item weights 248 us (312 for
// reduce, scan of the partial sums and scan, which read twice), 1e5 words 4 (9 in
// three launches).
template <typename T, typename In>
__global__ void __launch_bounds__(kScanThreads, 5) k_scan(In in, T *out, size_t n, uint64_t *words) {
  __shared__ T tile[kScanTile + kScanTile / (128 / sizeof(T))];
  __shared__ uint32_t s_tile;
  __shared__ uint64_t s_before;
  if (threadIdx.x == 0) {
    s_tile = words ? atomicAdd(reinterpret_cast<uint32_t *>(words), 1u) : 0u;
    s_before = 0;
  }
  __syncthreads();
  const uint32_t t = s_tile;
  const size_t base = (size_t)t * kScanTile;
  // coalesced load into shared memory
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    size_t idx = base + (size_t)i * kScanThreads + threadIdx.x;
    tile[scan_pad<T>(i * kScanThreads + threadIdx.x)] = idx < n ? in(idx) : T(0);
  }
  __syncthreads();
  T v[kScanItems];
  T s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = tile[scan_pad<T>(threadIdx.x * kScanItems + i)];
    s += v[i];
  }
  T total;
  T pre = block_exclusive_scan<T>(s, &total);
  if (words && threadIdx.x < 32) {
    constexpr uint64_t kSum = 1ull << 62, kPrefix = 2ull << 62, kValue = kSum - 1;
    uint64_t *st = words + 1;
    const int lane = (int)threadIdx.x;
    if (lane == 0) {
      st_relaxed(st + t, (t ? kSum : kPrefix) | (uint64_t)total);
      __threadfence();
    }
    uint64_t before = 0;
    uint32_t p = t, polls = 0;  // tiles [p, t) are in `before`
    while (p > 0) {
      const uint64_t w = (uint32_t)lane < p ? ld_relaxed(st + (p - 1u - (uint32_t)lane)) : kPrefix;
      const uint32_t unknown = __ballot_sync(0xffffffffu, (w >> 62) == 0);
      const uint32_t prefix = __ballot_sync(0xffffffffu, (w >> 62) == 2);
      const int known = unknown ? __ffs(unknown) - 1 : 32;
      const int first = prefix ? __ffs(prefix) - 1 : 32;
      const int take = first < known ? first + 1 : known;
      before += warp_sum(lane < take ? w & kValue : 0ull);
      if (first < known) break;
      p -= (uint32_t)take;
      if (take == 0 && ++polls > kLookLimit) {
        T own = 0;
        for (int e = lane; e < kScanTile; e += 32) {
          const size_t idx = (size_t)(p - 1u) * kScanTile + e;
          if (idx < n) own += in(idx);
        }
        const uint64_t sum = (uint64_t)(T)warp_sum((uint64_t)own);
        __threadfence();
        if (__any_sync(0xffffffffu, (ld_relaxed(st + (p - 1u)) >> 62) != 0)) continue;
        before += sum;
        --p;
      }
    }
    if (lane == 0) {
      if (t) st_relaxed(st + t, kPrefix | (before + (uint64_t)total));
      s_before = before;
    }
  }
  __syncthreads();
  pre += (T)s_before;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    tile[scan_pad<T>(threadIdx.x * kScanItems + i)] = pre;
    pre += v[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    size_t idx = base + (size_t)i * kScanThreads + threadIdx.x;
    if (idx < n) out[idx] = tile[scan_pad<T>(i * kScanThreads + threadIdx.x)];
  }
}

template <typename T, typename In>
int scan_exclusive_by(In in, T *out, size_t n, Arena &arena) {
  if (n == 0) return ASCI_OK;
  const size_t nb = (n + kScanTile - 1) / kScanTile;
  cudaStream_t s = arena.stream();
  uint64_t *words = nullptr;
  if (nb > 1) {
    ASCI_TRY(arena.alloc(&words, nb + 1));
    ASCI_TRY_CUDA(cudaMemsetAsync(words, 0, (nb + 1) * sizeof(uint64_t), s));
  }
  k_scan<T, In><<<(unsigned)nb, kScanThreads, 0, s>>>(in, out, n, words);
  ASCI_CHECK_LAUNCH();
  return ASCI_OK;
}

template <typename T>
int scan_exclusive(const T *in, T *out, size_t n, Arena &arena) {
  return scan_exclusive_by<T>(ArrayIn<T>{in}, out, n, arena);
}

// ----------------------------- radix sort ---------------------------------

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortItems = 16;  // per thread
constexpr int kSortTile = kSortThreads * kSortItems;
constexpr int kRadix = 256;

// The digits of a sort that vary, lowest first (at most eight).
struct DigitShifts {
  int count;
  int shift[8];
};

// Counts of every digit in one pass over the keys (hist[digit][value]).
__global__ void __launch_bounds__(512) k_digit_counts(const uint64_t *keys, size_t n,
                                                      DigitShifts D, uint32_t *hist) {
  extern __shared__ uint32_t h[];
  for (int i = threadIdx.x; i < D.count * kRadix; i += blockDim.x) h[i] = 0;
  __syncthreads();
  const size_t step = (size_t)gridDim.x * blockDim.x * 4;
  for (size_t base = (size_t)blockIdx.x * blockDim.x * 4; base < n; base += step) {
    uint64_t k[4] = {0, 0, 0, 0};
    uint32_t ok = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const size_t i = base + (size_t)r * blockDim.x + threadIdx.x;
      if (i < n) {
        k[r] = keys[i];
        ok |= 1u << r;
      }
    }
    for (int d = 0; d < D.count; ++d) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const uint32_t v = (uint32_t)(k[r] >> D.shift[d]) & 0xffu;
        // kept together from one addition to the next: 57.7 M keys of four digits take
        // 154 us, without this 445 (557 without the branch)
        __syncwarp();
        if ((ok >> r) & 1u) atomicAdd(&h[d * kRadix + v], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < D.count * kRadix; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

// A word of the tiles' digit counts: the value (a count or a prefix, both at most
// n < 2^32) below a tag, 4 x (number of the pass) + state.  The words of one pass
// are distinct from those of the passes before, so they are cleared once a sort.
constexpr uint32_t kTileCount = 1u;   // the tile's own count of the digit
constexpr uint32_t kTilePrefix = 2u;  // the count in this tile and all before it
constexpr int kLook = 8;               // predecessors read at a time

// Shared memory of the scatter: the tile's keys (and values) in digit order,
// per-warp digit counters, and each digit's offset from the tile to the output.
template <typename V, bool kHasVals>
constexpr size_t scatter_smem() {
  return (size_t)kSortTile * sizeof(uint64_t) + (kHasVals ? (size_t)kSortTile * sizeof(V) : 0) +
         (size_t)(kSortWarps + 1) * kRadix * sizeof(uint32_t);
}

// Stable scatter by one digit, a tile per CTA, the digits' starts by decoupled look back
// (as in the Onesweep sort of Adinets and Merrill, 2022).  Warp w owns elements
// [w*32*kSortItems, ...) of the tile in rounds of 32 consecutive elements, so tile
// order is preserved.  Tiles are numbered in the order in which CTAs start, so a
// tile's predecessors are running or done; each publishes its digit counts before
// it looks at theirs, so the wait below always ends.  Thread d adds up digit d of
// the tiles before, kLook at a time, back to the nearest one that knows its prefix.
// (Should a predecessor not answer within kLookLimit polls, the CTA counts the
// keys before its tile itself.)  The tile is then placed in shared memory in digit
// order and each digit's run is written with consecutive threads on consecutive
// addresses.
//
// Bound: shared-memory wavefronts (78% of their rate) before memory: 16 bytes a
// key and digit, at 2.8 TB/s.  Against a histogram kernel, its scan and a scatter
// that ranked twice, a digit of 57.7 M keys 620 -> 330 us with its share of the
// counts, of 1e5 keys 30 (five launches) -> 9.
template <typename V, bool kHasVals>
__global__ void __launch_bounds__(kSortThreads, 4)
    k_digit_scatter(const uint64_t *keys_in, const V *vals_in, uint64_t *keys_out, V *vals_out,
                    size_t n, int shift, uint32_t pass, const uint32_t *hist, uint64_t *words,
                    uint32_t *ticket) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ uint32_t s_tile;
  uint64_t *sk = reinterpret_cast<uint64_t *>(sm);
  V *sv = reinterpret_cast<V *>(sk + kSortTile);
  uint32_t *wb = reinterpret_cast<uint32_t *>(sm + (size_t)kSortTile * sizeof(uint64_t) +
                                              (kHasVals ? (size_t)kSortTile * sizeof(V) : 0));
  uint32_t *dmove = wb + kSortWarps * kRadix;  // from a key's place in the tile to the output
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_tile = atomicAdd(ticket, 1u);
  for (int i = threadIdx.x; i < kSortWarps * kRadix; i += kSortThreads) wb[i] = 0;
  __syncthreads();
  const uint32_t tile = s_tile;
  const size_t base = (size_t)tile * kSortTile;
  const size_t wbase = base + (size_t)warp * 32 * kSortItems;
  const uint32_t lt = (1u << lane) - 1u;
  // the tile's keys and their ranks among the warp's keys of the same digit stay in
  // registers; out-of-range slots get the digit kRadix, which no counter holds
  uint64_t k[kSortItems];
  uint32_t rank2[kSortItems / 2];  // two 16-bit ranks a word
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const size_t idx = wbase + (size_t)r * 32 + lane;
    k[r] = idx < n ? keys_in[idx] : 0ull;
  }
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const bool ok = wbase + (size_t)r * 32 + lane < n;
    const uint32_t d = ok ? (uint32_t)((k[r] >> shift) & 0xffu) : (uint32_t)kRadix;
    const uint32_t peers = __match_any_sync(0xffffffffu, d);
    uint32_t before = 0;
    if (ok) before = wb[warp * kRadix + d];
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) wb[warp * kRadix + d] = before + __popc(peers);
    __syncwarp();
    const uint32_t rk = before + __popc(peers & lt);
    rank2[r >> 1] = (r & 1) ? rank2[r >> 1] | (rk << 16) : rk;
  }
  __syncthreads();
  {
    const int dig = threadIdx.x;  // kSortThreads == kRadix
    uint32_t cnt = 0, first[kSortWarps];  // the warps' keys within the digit's run
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) {
      first[w] = cnt;
      cnt += wb[w * kRadix + dig];
    }
    uint64_t *mine = words + (size_t)tile * kRadix + dig;
    const uint64_t tag = (uint64_t)(4u * pass) << 32;
    st_relaxed(mine, tag | ((uint64_t)(tile ? kTileCount : kTilePrefix) << 32) | cnt);
    // starts of the digit in the tile and in the output: both sums stay below 2^32
    const uint64_t st = block_exclusive_scan<uint64_t>(((uint64_t)cnt << 32) | hist[dig], nullptr);
    const uint32_t dstart = (uint32_t)(st >> 32);
#pragma unroll
    for (int w = 0; w < kSortWarps; ++w) wb[w * kRadix + dig] = dstart + first[w];
    uint32_t before = 0;  // the digit's keys in the tiles before
    bool lost = false;
    if (tile) {
      uint32_t t = tile, polls = 0;  // tiles [t, tile) are in `before`
      bool done = false;
      while (!done) {
        uint64_t w[kLook];
#pragma unroll
        for (int j = 0; j < kLook; ++j) {
          const uint32_t b = (uint32_t)j + 1u <= t ? t - 1u - (uint32_t)j : 0u;
          w[j] = ld_relaxed(words + (size_t)b * kRadix + dig);
        }
        bool open = true;
#pragma unroll
        for (int j = 0; j < kLook; ++j) {
          const uint32_t hi = (uint32_t)(w[j] >> 32);
          open = open && !done && hi >= 4u * pass + kTileCount;
          if (open) {
            before += (uint32_t)w[j];
            --t;
            done = hi == 4u * pass + kTilePrefix;
          }
        }
        if (!done && ++polls > kLookLimit + tile) {
          lost = true;
          break;
        }
      }
    }
    if (__syncthreads_or(lost)) {
      dmove[dig] = 0;
      __syncthreads();
      for (size_t i = threadIdx.x; i < base; i += kSortThreads)
        atomicAdd(&dmove[(keys_in[i] >> shift) & 0xffu], 1u);
      __syncthreads();
      before = dmove[dig];
      __syncthreads();
    }
    if (tile) st_relaxed(mine, tag | ((uint64_t)kTilePrefix << 32) | (before + cnt));
    dmove[dig] = (uint32_t)st + before - dstart;
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortItems; ++r) {
    const size_t idx = wbase + (size_t)r * 32 + lane;
    if (idx < n) {
      const uint32_t d = (uint32_t)((k[r] >> shift) & 0xffu);
      const uint32_t pos = wb[warp * kRadix + d] + ((rank2[r >> 1] >> (16 * (r & 1))) & 0xffffu);
      sk[pos] = k[r];
      if (kHasVals) sv[pos] = vals_in[idx];
    }
  }
  __syncthreads();
  const uint32_t tn = (uint32_t)((n - base) < (size_t)kSortTile ? (n - base) : (size_t)kSortTile);
  for (uint32_t i = threadIdx.x; i < tn; i += kSortThreads) {
    const uint64_t key = sk[i];
    const uint32_t dg = (uint32_t)((key >> shift) & 0xffu);
    const uint32_t gpos = dmove[dg] + i;
    keys_out[gpos] = key;
    if (kHasVals) vals_out[gpos] = sv[i];
  }
}

// The whole sort of at most one tile (4096 keys) in one CTA: 16 warps of 256
// consecutive elements each, the digits that vary one after another in shared
// memory (the ranks as in the scatter above, so just as stable).  Through the tile
// kernels a list of one tile would take a launch a digit, the counts' launch and,
// where the varying bits are not given, a wait for them.
constexpr int kSmallThreads = 512;
constexpr int kSmallItems = kSortTile / kSmallThreads;
constexpr int kSmallWarps = kSmallThreads / 32;

template <typename V, bool kHasVals>
constexpr size_t small_smem() {
  return (size_t)kSortTile * (sizeof(uint64_t) + (kHasVals ? sizeof(V) : 0)) +
         (size_t)(kSmallWarps + 1) * kRadix * sizeof(uint32_t);
}

template <typename V, bool kHasVals>
__global__ void __launch_bounds__(kSmallThreads) k_sort_small(uint64_t *keys, V *vals, uint32_t n,
                                                              int begin_bit, int end_bit) {
  extern __shared__ __align__(16) unsigned char sm[];
  __shared__ uint32_t differ[2];
  uint64_t *sk = reinterpret_cast<uint64_t *>(sm);
  V *sv = reinterpret_cast<V *>(sk + kSortTile);
  uint32_t *wb = reinterpret_cast<uint32_t *>(sm + (size_t)kSortTile * (sizeof(uint64_t) +
                                                                        (kHasVals ? sizeof(V) : 0)));
  uint32_t *dstart = wb + kSmallWarps * kRadix;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t base = (uint32_t)warp * (32 * kSmallItems) + lane;
  if (threadIdx.x < 2) differ[threadIdx.x] = 0;
  const uint64_t k0 = keys[0];
  uint64_t k[kSmallItems], acc = 0;
  V v[kSmallItems];
#pragma unroll
  for (int r = 0; r < kSmallItems; ++r) {
    const uint32_t i = base + 32 * r;
    k[r] = i < n ? keys[i] : 0ull;
    if (kHasVals) v[r] = i < n ? vals[i] : V(0);
    if (i < n) acc |= k[r] ^ k0;
  }
  __syncthreads();
  const uint32_t a0 = __reduce_or_sync(0xffffffffu, (uint32_t)acc);
  const uint32_t a1 = __reduce_or_sync(0xffffffffu, (uint32_t)(acc >> 32));
  if (lane == 0) {
    if (a0) atomicOr(&differ[0], a0);
    if (a1) atomicOr(&differ[1], a1);
  }
  __syncthreads();
  const uint64_t mask = ((uint64_t)differ[1] << 32) | differ[0];
  const uint32_t lt = (1u << lane) - 1u;
  for (int shift = begin_bit; shift < end_bit; shift += 8) {
    const uint64_t dm = end_bit - shift < 8 ? (1ull << (end_bit - shift)) - 1ull : 0xffull;
    if (!((mask >> shift) & dm)) continue;  // uniform
    for (int i = threadIdx.x; i < kSmallWarps * kRadix; i += kSmallThreads) wb[i] = 0;
    __syncthreads();
    uint32_t rank[kSmallItems];  // among the warp's keys of the same digit
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r) {
      const bool ok = base + 32 * r < n;
      const uint32_t d = ok ? (uint32_t)((k[r] >> shift) & 0xffu) : (uint32_t)kRadix;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      uint32_t before = 0;
      if (ok) before = wb[warp * kRadix + d];
      __syncwarp();
      if (ok && lane == __ffs(peers) - 1) wb[warp * kRadix + d] = before + __popc(peers);
      __syncwarp();
      rank[r] = before + __popc(peers & lt);
    }
    __syncthreads();
    uint32_t cnt = 0;
    if (threadIdx.x < kRadix)
      for (int w = 0; w < kSmallWarps; ++w) {
        const uint32_t c = wb[w * kRadix + threadIdx.x];
        wb[w * kRadix + threadIdx.x] = cnt;
        cnt += c;
      }
    const uint32_t first = block_exclusive_scan<uint32_t>(cnt, nullptr);
    if (threadIdx.x < kRadix) dstart[threadIdx.x] = first;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r)
      if (base + 32 * r < n) {
        const uint32_t d = (uint32_t)((k[r] >> shift) & 0xffu);
        const uint32_t pos = dstart[d] + wb[warp * kRadix + d] + rank[r];
        sk[pos] = k[r];
        if (kHasVals) sv[pos] = v[r];
      }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSmallItems; ++r)
      if (base + 32 * r < n) {
        k[r] = sk[base + 32 * r];
        if (kHasVals) v[r] = sv[base + 32 * r];
      }
  }
#pragma unroll
  for (int r = 0; r < kSmallItems; ++r)
    if (base + 32 * r < n) {
      keys[base + 32 * r] = k[r];
      if (kHasVals) vals[base + 32 * r] = v[r];
    }
}

template <typename V, bool kHasVals>
int radix_sort_impl(uint64_t **keys, uint64_t **keys_alt, V **vals, V **vals_alt, size_t n,
                    int begin_bit, int end_bit, Arena &arena, const uint64_t *known_mask = nullptr) {
  if (n <= 1 || begin_bit >= end_bit) return ASCI_OK;
  if (n >= (1ull << 32)) return ASCI_EINVAL;
  cudaStream_t s = arena.stream();
  if (n <= (size_t)kSortTile) {
    static const cudaError_t small_attr = cudaFuncSetAttribute(
        k_sort_small<V, kHasVals>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)small_smem<V, kHasVals>());
    ASCI_TRY_CUDA(small_attr);
    k_sort_small<V, kHasVals><<<1, kSmallThreads, small_smem<V, kHasVals>(), s>>>(
        *keys, kHasVals ? *vals : nullptr, (uint32_t)n, begin_bit, end_bit);
    ASCI_CHECK_LAUNCH();
    return ASCI_OK;
  }
  const uint32_t ntiles = (uint32_t)((n + kSortTile - 1) / kSortTile);
  // once per instantiation (thread-safe static initialisation)
  static const cudaError_t attr = cudaFuncSetAttribute(
      k_digit_scatter<V, kHasVals>, cudaFuncAttributeMaxDynamicSharedMemorySize,
      (int)scatter_smem<V, kHasVals>());
  ASCI_TRY_CUDA(attr);
  uint64_t mask = 0;
  if (known_mask) mask = *known_mask;  // the caller knows which bits vary
  else ASCI_TRY(varying_bits_u64(*keys, n, &mask, arena));
  DigitShifts D;
  D.count = 0;
  for (int shift = begin_bit; shift < end_bit; shift += 8) {
    uint64_t dmask = (0xffull << shift);
    if (end_bit - shift < 8) dmask &= ((end_bit >= 64) ? ~0ull : ((1ull << end_bit) - 1));
    if (mask & dmask) D.shift[D.count++] = shift;  // else constant over the input
  }
  if (D.count == 0) return ASCI_OK;
  // the tiles' words, then the counts and the tickets of the passes
  uint64_t *words;
  const size_t nwords = (size_t)kRadix * ntiles, extra = (size_t)D.count * (kRadix + 1);
  ASCI_TRY(arena.alloc(&words, nwords + (extra + 1) / 2));
  ASCI_TRY_CUDA(cudaMemsetAsync(words, 0, (nwords + (extra + 1) / 2) * sizeof(uint64_t), s));
  uint32_t *hist = reinterpret_cast<uint32_t *>(words + nwords);
  uint32_t *ticket = hist + (size_t)D.count * kRadix;
  k_digit_counts<<<(unsigned)std::min<size_t>(152 * 4, (n + 2047) / 2048), 512,
                   (size_t)D.count * kRadix * sizeof(uint32_t), s>>>(*keys, n, D, hist);
  ASCI_CHECK_LAUNCH();
  for (int p = 0; p < D.count; ++p) {
    k_digit_scatter<V, kHasVals><<<ntiles, kSortThreads, scatter_smem<V, kHasVals>(), s>>>(
        *keys, kHasVals ? *vals : nullptr, *keys_alt, kHasVals ? *vals_alt : nullptr, n,
        D.shift[p], (uint32_t)(p + 1), hist + (size_t)p * kRadix, words, ticket + p);
    ASCI_CHECK_LAUNCH();
    uint64_t *t = *keys;
    *keys = *keys_alt;
    *keys_alt = t;
    if (kHasVals) {
      V *tv = *vals;
      *vals = *vals_alt;
      *vals_alt = tv;
    }
  }
  return ASCI_OK;
}

__global__ void k_varying(const uint64_t *keys, size_t n, unsigned long long *out) {
  uint64_t k0 = keys[0], acc = 0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    acc |= keys[i] ^ k0;
  for (int d = 16; d; d >>= 1) acc |= __shfl_xor_sync(0xffffffffu, acc, d);
  if ((threadIdx.x & 31) == 0 && acc) atomicOr(out, (unsigned long long)acc);
}

}  // namespace

int scan_exclusive_u32(const uint32_t *in, uint32_t *out, size_t n, Arena &arena) {
  return scan_exclusive<uint32_t>(in, out, n, arena);
}
int scan_exclusive_u64(const uint64_t *in, uint64_t *out, size_t n, Arena &arena) {
  return scan_exclusive<uint64_t>(in, out, n, arena);
}

int scan_item_weights(const uint64_t *items, uint64_t T, int opbits, const uint32_t *grp_count,
                      const ExcCounts &X, uint64_t *Wexcl, Arena &arena) {
  ItemWeightIn in{items, grp_count, T, (uint64_t)X.sb + X.dbb, 1ull + X.sb,
                  (1u << opbits) - 1u, X.sa, opbits};
  return scan_exclusive_by<uint64_t>(in, Wexcl, (size_t)T + 1, arena);
}

int scan_item_heads(const uint64_t *items, uint64_t T, uint32_t *excl, Arena &arena) {
  return scan_exclusive_by<uint32_t>(ItemHeadIn{items, T}, excl, (size_t)T + 1, arena);
}

int varying_bits_u64(const uint64_t *keys, size_t n, uint64_t *host_mask, Arena &arena) {
  *host_mask = 0;
  if (n == 0) return ASCI_OK;
  unsigned long long *d = nullptr;
  ASCI_TRY(arena.alloc(&d, 1));
  cudaStream_t s = arena.stream();
  ASCI_TRY_CUDA(cudaMemsetAsync(d, 0, sizeof(unsigned long long), s));
  unsigned blocks = (unsigned)((n + 255) / 256);
  if (blocks > 152 * 8) blocks = 152 * 8;
  k_varying<<<blocks, 256, 0, s>>>(keys, n, d);
  ASCI_CHECK_LAUNCH();
  unsigned long long h = 0;
  ASCI_TRY_CUDA(cudaMemcpyAsync(&h, d, sizeof(h), cudaMemcpyDeviceToHost, s));
  ASCI_TRY_CUDA(cudaStreamSynchronize(s));
  *host_mask = h;
  return ASCI_OK;
}

int radix_sort_u64(uint64_t **keys, uint64_t **keys_alt, size_t n, int begin_bit, int end_bit,
                   Arena &arena) {
  return radix_sort_impl<uint32_t, false>(keys, keys_alt, nullptr, nullptr, n, begin_bit, end_bit,
                                          arena);
}
int radix_sort_u64_varying(uint64_t **keys, uint64_t **keys_alt, size_t n, int begin_bit,
                           int end_bit, uint64_t varying, Arena &arena) {
  return radix_sort_impl<uint32_t, false>(keys, keys_alt, nullptr, nullptr, n, begin_bit, end_bit,
                                          arena, &varying);
}
int radix_sort_u64_u32(uint64_t **keys, uint64_t **keys_alt, uint32_t **vals, uint32_t **vals_alt,
                       size_t n, int begin_bit, int end_bit, Arena &arena,
                       const uint64_t *varying) {
  return radix_sort_impl<uint32_t, true>(keys, keys_alt, vals, vals_alt, n, begin_bit, end_bit,
                                         arena, varying);
}
int radix_sort_u64_f64(uint64_t **keys, uint64_t **keys_alt, double **vals, double **vals_alt,
                       size_t n, int begin_bit, int end_bit, Arena &arena,
                       const uint64_t *varying) {
  return radix_sort_impl<double, true>(keys, keys_alt, vals, vals_alt, n, begin_bit, end_bit,
                                       arena, varying);
}

}  // namespace asci
