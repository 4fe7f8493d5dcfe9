// sort.cu -- A3: stable LSD radix sort of (uint64 key, uint32 value) pairs,
// one kernel per 8-bit digit with decoupled look-back ("onesweep"): each CTA
// ranks one tile of keys in shared memory, publishes its per-digit counts,
// looks back over the preceding tiles for their running totals and scatters
// its keys straight to their final positions of that pass.
//
// The paper sorts the Z-curve keys with the search library's device sort
// (§2 "ArborX"); this is an independent GPU sort with the same result (a
// stable order of the codes, equal codes keeping input order).
#include "common.cuh"

namespace emst {

constexpr int kRadix = 256;
constexpr uint32_t kFlagAggregate = 1u << 30;
constexpr uint32_t kFlagPrefix = 2u << 30;
constexpr uint32_t kValueMask = (1u << 30) - 1u;
constexpr int kSpinLimit = 1 << 22;
constexpr int kLookWindow = 8;  // preceding tiles read per look-back round trip
// A tile is kSortThreads threads x items.  Each tile costs the others a step
// of their look-back, so there should be no more than a few hundred until
// larger ones no longer fit the registers; below that the GPU wants a tile
// per SM.  A sort of 8 digits (us) with 4 / 8 / 14 items: 600,000 keys 150 /
// 119 / 150, 1M - / 182 / 152, 2M - / 281 / 254 (core distances of 200,000
// points, whole call, 4 / 12 items: 519 / 538); 37M keys with 8 / 12 / 14 /
// 15 items 2,940 / 2,535 / 2,425 / 2,955 (15 spill; 18 at two CTAs per SM
// 2,820).  Before the ballots and the scatter ahead of the look-back, with
// 12 items: 200,000 keys 113, 1M 208, 8M 846, 37M 3,061.
constexpr int kSortThreads = 256;
constexpr int kSmallItems = 4, kMidItems = 8, kLargeItems = 14;
constexpr int64_t kMaxEarlyTiles = 300;  // of the two smaller shapes
constexpr int64_t kSmallMax = kMaxEarlyTiles * kSortThreads * kSmallItems;
constexpr int64_t kMidMax = kMaxEarlyTiles * kSortThreads * kMidItems;

// Tiles of a sort of up to n keys, whichever shape serves it.
static int64_t sort_tiles_for(int64_t n) {
  auto tiles = [](int64_t c, int items) { return (c + kSortThreads * items - 1) / (kSortThreads * items); };
  if (n <= kSmallMax) return tiles(n, kSmallItems);
  const int64_t large = tiles(n, kLargeItems);
  return large > kMaxEarlyTiles ? large : kMaxEarlyTiles;
}

constexpr int kWarps = kSortThreads / 32;
static_assert(kSortThreads == kRadix, "a sort pass gives each thread one digit");

// The words of P.sort_state: the digits' histograms, the passes' tile counters
// and the histogram's count of finished CTAs, then two look-back arrays that
// the passes use in turn (each clears the other for the next one), so one
// memset serves a whole sort.
constexpr int64_t kHistWords = 8 * kRadix;
constexpr int64_t kCounterWords = 64;  // [0..7] tile counters, [8] finished CTAs

int64_t sort_clear_words(int64_t n) {
  const int items = n <= kSmallMax ? kSmallItems : n <= kMidMax ? kMidItems : kLargeItems;
  return kHistWords + kCounterWords + kRadix * ((n + kSortThreads * items - 1) / (kSortThreads * items));
}

int64_t sort_state_words(int64_t n) { return kHistWords + kCounterWords + 2 * kRadix * sort_tiles_for(n); }

// Histograms of all digits in [digit_begin, digit_end) in one pass; the last
// CTA to finish turns them into exclusive prefix sums.
__global__ void __launch_bounds__(512) k_sort_hist(const uint64_t *__restrict__ keys, int64_t n,
                                                   int digit_begin, int digit_end, int bit0,
                                                   uint32_t *hist, uint32_t *finished) {
  __shared__ uint32_t sh[8][kRadix];
  __shared__ bool s_last;
  for (int t = threadIdx.x; t < 8 * kRadix; t += blockDim.x) (&sh[0][0])[t] = 0;
  wait_for_previous();
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) {
    uint64_t key = __ldg(keys + k) >> bit0;
    for (int d = digit_begin; d < digit_end; ++d)
      atomicAdd(&sh[d][(uint32_t)(key >> (8 * d)) & 0xffu], 1u);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 8 * kRadix; t += blockDim.x) {
    uint32_t v = (&sh[0][0])[t];
    if (v) atomicAdd(hist + t, v);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(finished, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // a warp per digit, eight bins per lane
  const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
  if (d < 8) {
    uint32_t *h = hist + d * kRadix + lane * 8;
    uint32_t v[8], sum = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      v[q] = __ldcg(h + q);
      sum += v[q];
    }
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    uint32_t run = x - sum;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      h[q] = run;
      run += v[q];
    }
  }
}

template <int ITEMS>
struct SortSmem {
  static constexpr int kTile = kSortThreads * ITEMS;
  uint64_t keys[kTile];
  uint32_t vals[kTile];
  uint32_t warp_hist[kWarps][kRadix];
  uint32_t global_base[kRadix];  // global position of local position 0 of each digit
  uint32_t warp_tot[kWarps];
  uint32_t tile_id;
};

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

template <int ITEMS, int BLOCKS>
__global__ void __launch_bounds__(kSortThreads, BLOCKS) k_sort_pass(
    const uint64_t *__restrict__ keys_in, const uint32_t *__restrict__ vals_in,
    uint64_t *__restrict__ keys_out, uint32_t *__restrict__ vals_out, int64_t n, int shift,
    const uint32_t *__restrict__ digit_offset, uint32_t *lookback, uint32_t *next_lookback,
    uint32_t *tile_counter, uint32_t *status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SortSmem<ITEMS> &S = *reinterpret_cast<SortSmem<ITEMS> *>(smem_raw);
  constexpr int kTile = SortSmem<ITEMS>::kTile;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  for (int t = tid; t < kWarps * kRadix; t += kSortThreads) (&S.warp_hist[0][0])[t] = 0;
  wait_for_previous();
  if (tid == 0) S.tile_id = atomicAdd(tile_counter, 1u);
  __syncthreads();
  const uint32_t tile = S.tile_id;
  const int64_t base = (int64_t)tile * kTile;
  const int count = (int)(n - base < kTile ? n - base : kTile);
  const int seg = warp * 32 * ITEMS;

  // Load: warp w owns a contiguous segment; item `it` of lane l sits at
  // seg + it*32 + l, so (it, lane) order is input order within the warp.
  uint64_t key[ITEMS];
  uint32_t val[ITEMS];
  uint32_t rank[(ITEMS + 1) / 2] = {};  // two of 16 bits each
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int idx = seg + it * 32 + lane;
    const bool ok = idx < count;
    key[it] = ok ? keys_in[base + idx] : 0ull;
    val[it] = ok ? vals_in[base + idx] : 0u;
  }
  // Rank within the warp, in input order: peers with the same digit in this
  // item (one ballot per bit: they wait on nothing, so the items' overlap,
  // where a match instruction per item took a third longer, 8M keys 846 ->
  // 630 us a sort), plus the warp's running count of that digit.  The leader
  // adds the group size to the warp's counter; the old value is the group's
  // base.  The warp issues the items' adds in order, so item it's base counts
  // exactly the keys of items < it.
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const bool ok = seg + it * 32 + lane < count;
    uint32_t dg = ok ? (uint32_t)(key[it] >> shift) & 0xffu : 0x100u + lane;
    uint32_t peers = __ballot_sync(0xffffffffu, ok);
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const bool p = (dg >> b) & 1u;
      const uint32_t m = __ballot_sync(0xffffffffu, p);
      peers &= p ? m : ~m;
    }
    const int leader = __ffs(peers) - 1;
    uint32_t first = 0u;
    if (ok && leader == lane) first = atomicAdd(&S.warp_hist[warp][dg], (uint32_t)__popc(peers));
    first = __shfl_sync(0xffffffffu, first, leader);
    rank[it / 2] |= (first + __popc(peers & lt)) << (16 * (it & 1));
  }
  __syncthreads();

  // Thread t owns digit t: its count in each warp, and the tile total.
  const int t = tid;
  uint32_t total = 0;
  uint32_t before[kWarps];
#pragma unroll
  for (int w = 0; w < kWarps; ++w) {
    before[w] = total;
    total += S.warp_hist[w][t];
  }
  // Publish this tile's count (tile 0 publishes a finished prefix at once).
  {
    volatile uint32_t *lb = lookback + (int64_t)tile * kRadix + t;
    *lb = (tile == 0 ? kFlagPrefix : kFlagAggregate) | total;
  }
  next_lookback[(int64_t)tile * kRadix + t] = 0u;
  // Exclusive scan of the totals over digits: local start of each digit, and
  // from it the first local position of each warp's keys of that digit.
  uint32_t x = total;
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) S.warp_tot[warp] = x;
  __syncthreads();
  uint32_t start = x - total;
  for (int q = 0; q < warp; ++q) start += S.warp_tot[q];
#pragma unroll
  for (int w = 0; w < kWarps; ++w) S.warp_hist[w][t] = start + before[w];
  __syncthreads();

  // Scatter into shared memory in tile-sorted order.  (Before the look-back:
  // the registers are free for it, and the tiles before this one publish
  // meanwhile.)
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    if (seg + it * 32 + lane < count) {
      const uint32_t dg = (uint32_t)(key[it] >> shift) & 0xffu;
      const uint32_t pos = S.warp_hist[warp][dg] + ((rank[it / 2] >> (16 * (it & 1))) & 0xffffu);
      S.keys[pos] = key[it];
      S.vals[pos] = val[it];
    }
  }
  // Look back over preceding tiles for digit t, kLookWindow tiles per round
  // trip: sum their counts in order up to the nearest finished prefix; a
  // tile that has not published yet is waited for.
  uint32_t excl = 0;
  if (tile > 0) {
    int64_t j = (int64_t)tile - 1;
    int spins = 0;
    for (;;) {
      uint32_t wv[kLookWindow];
#pragma unroll
      for (int w = 0; w < kLookWindow; ++w)
        wv[w] = j - w >= 0 ? *reinterpret_cast<const volatile uint32_t *>(lookback + (j - w) * kRadix + t)
                           : kFlagPrefix;  // before tile 0: a finished prefix of 0
      int used = 0;
      bool done = false, stall = false;
#pragma unroll
      for (int w = 0; w < kLookWindow; ++w) {
        if (done || stall) continue;
        const uint32_t f = wv[w] & ~kValueMask;
        if (f == 0u) { stall = true; continue; }
        excl += wv[w] & kValueMask;
        ++used;
        done = f == kFlagPrefix;
      }
      if (done) break;
      j -= used;
      if (stall) {
        if (++spins > kSpinLimit) {  // give up: results are invalid, the status says so
          atomicOr(status, kErrSpin);
          break;
        }
        __nanosleep(32);
      }
    }
    volatile uint32_t *mine = lookback + (int64_t)tile * kRadix + t;
    *mine = kFlagPrefix | ((excl + total) & kValueMask);
  }
  S.global_base[t] = digit_offset[t] + excl - start;
  __syncthreads();
  // Write out: consecutive threads write consecutive positions of a digit run.
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = it * kSortThreads + tid;
    if (i < count) {
      const uint64_t k = S.keys[i];
      const uint32_t out = S.global_base[(uint32_t)(k >> shift) & 0xffu] + (uint32_t)i;
      keys_out[out] = k;
      vals_out[out] = S.vals[i];
    }
  }
}

// One sort of tiles of kSortThreads x ITEMS keys.
template <int ITEMS, int BLOCKS>
static int sort_passes(Problem &P, int64_t n, int digit_begin, int digit_end, int src, int bit0, bool cleared) {
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  const size_t smem = sizeof(SortSmem<ITEMS>);
  if (dev >= 64 || !attr_set[dev]) {
    cudaFuncSetAttribute(k_sort_pass<ITEMS, BLOCKS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (dev < 64) attr_set[dev] = true;
  }
  const int64_t tiles = (n + SortSmem<ITEMS>::kTile - 1) / SortSmem<ITEMS>::kTile;
  uint32_t *hist = P.sort_state, *counters = hist + kHistWords;
  uint32_t *look[2] = {counters + kCounterWords, counters + kCounterWords + kRadix * tiles};
  if (!cleared)
    cudaMemsetAsync(hist, 0, sizeof(uint32_t) * (size_t)(kHistWords + kCounterWords + kRadix * tiles), P.stream);
  // keys per histogram CTA: its 2,048 bins go to memory one atomic each, which
  // with 512 keys was most of the pass (a sort of 200,000 keys with 512 / 2,048
  // / 4,096: 77.5 / 75.4 / 77.4 us, of 1M 125.6 / 123.5 / 121.5)
  const int64_t hist_keys = n > 400000 ? 4096 : 2048;
  int hgrid = (int)((n + hist_keys - 1) / hist_keys);
  if (hgrid > sm_count() * 4) hgrid = sm_count() * 4;
  launch_next(P, k_sort_hist, hgrid, 512, 0, P.keys[src], n, digit_begin, digit_end, bit0, hist, counters + 8);
  P.launches += 1;
  for (int d = digit_begin; d < digit_end; ++d) {
    launch_next(P, k_sort_pass<ITEMS, BLOCKS>, (unsigned)tiles, kSortThreads, smem, P.keys[src], P.vals[src], P.keys[src ^ 1], P.vals[src ^ 1], n, bit0 + 8 * d, hist + d * kRadix,
        look[0], look[1], counters + d, P.counters + 1);
    P.launches += 1;
    src ^= 1;
    uint32_t *t = look[0];
    look[0] = look[1];
    look[1] = t;
  }
  return src;
}

int radix_sort_pairs(Problem &P, int64_t n, int digit_begin, int digit_end, int src, int bit0,
                     bool cleared) {
  if (n <= 1 || digit_begin >= digit_end) return src;
  if (n <= kSmallMax) return sort_passes<kSmallItems, 4>(P, n, digit_begin, digit_end, src, bit0, cleared);
  if (n <= kMidMax) return sort_passes<kMidItems, 4>(P, n, digit_begin, digit_end, src, bit0, cleared);
  return sort_passes<kLargeItems, 3>(P, n, digit_begin, digit_end, src, bit0, cleared);
}

}  // namespace emst
