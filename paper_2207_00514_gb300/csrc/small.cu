// small.cu -- the whole EMST of a small problem in one cooperative launch.
//
// Up to kSmallMaxPoints points the general path is a sequence of about a
// hundred short launches with a host round trip per Boruvka round: at 333
// points nothing but launches, at 10,000 points launches plus searches that
// each wait on one lane's chain of 50 to 150 dependent node visits.  Here one
// cooperative kernel runs every step with grid barriers between them, and a
// query is one warp: the sorted points are cut into blocks of 32 consecutive
// curve positions and superblocks of 32 blocks, each with its box, so that a
// lane tests one box or one point and a search is a dozen warp-wide steps,
// nearest box first (Algorithm 2 with a fixed 32-ary hierarchy; the skip of
// same-component subtrees, the bounds and the tie rule are those of
// traverse.cuh).  The tree is unique under the total order (w, i, j), so it
// does not depend on the hierarchy.
//
// What bounds it: the latency of dependent L2 accesses, of the barriers (four
// and three a round, 1-2 us each) and, from some thousand points on, of the
// tile sorts (7 us each for 1,024 keys).  Measured (us per call, general path
// / this one): 333 points 345 / 113, 10,000 496-532 / 251-262, 16,384 512-611 /
// 290-338, 30,000 576-611 / 443-478, 32,768 552-657 / 445-517 by shape and
// dimension: they meet not far above, and a point's index has 16 bits in the
// sort keys.
#include <cstring>

#include "grid.cuh"

namespace emst {
namespace {

constexpr int kThreads = 512;
constexpr int kWarpsPerCta = kThreads / 32;
constexpr int kMaxTiles = 16;                  // tiles the rank merge looks through
constexpr int kMaxTile = 2048;                 // sort tile (a power of two)
static_assert(kMaxTiles * kMaxTile == kSmallMaxPoints, "every point fits the tiles");

// 128-bit sort keys, all distinct.
struct __align__(16) Key {
  uint64_t hi, lo;
};
__device__ __forceinline__ bool key_less(const Key &a, const Key &b) {
  return a.hi < b.hi || (a.hi == b.hi && a.lo < b.lo);
}

// A block's or superblock's box, 32 bytes: lo.w the label shared by all its
// points (kInvalid: several), hi.w their smallest original id.
struct __align__(16) BoxRec {
  float4 lo, hi;
};

struct SmallArgs {
  const float *src;       // the input (device memory, or pinned host memory mapped)
  float *copy;            // non-null: the device copy of a mapped input, written by the first step
  int n, dim, tile;
  uint32_t *counters;     // [0] edges, [1] status, [2..4] ~min, [5..7] max of the box, [8] barrier
  Key *tiles;             // n (+ padding): sorted tiles
  float4 *pts;            // n, curve order
  uint32_t *labels[2];
  uint32_t *bound[2];
  CompBest *comp[2];
  uint32_t *root;
  uint2 *res;
  BoxRec *blk, *sup;
  Key *ekeys;             // n: emitted edges as keys
  emst_edge *out;
};

// The curve key of a point: the 128-bit Z-curve code of build.cu (42 bits per
// axis in 3D, 64 in 2D, quantised in FP64) with its lowest 16 bits replaced
// by the point's index, which makes the keys distinct.
// lo, scale: the box's lower corner and 2^bits / extent (0 for a flat axis).
__device__ __forceinline__ Key curve_key(const float (&x)[3], const double *lo, const double *scale, int dim,
                                         uint32_t idx) {
  const double twoB = dim == 3 ? 4398046511104.0 : 18446744073709551616.0;
  const uint64_t qmax = dim == 3 ? ((1ull << 42) - 1ull) : ~0ull;
  uint64_t q[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (d >= dim) continue;
    const double t = __dmul_rn(__dsub_rn((double)x[d], lo[d]), scale[d]);
    q[d] = t >= twoB ? qmax : (uint64_t)t;
  }
  Key k;
  if (dim == 3) {
    const uint64_t H = interleave((uint32_t)(q[0] >> 21), (uint32_t)(q[1] >> 21), (uint32_t)(q[2] >> 21), 3);
    const uint64_t L = interleave((uint32_t)(q[0] & 0x1fffffu), (uint32_t)(q[1] & 0x1fffffu),
                                  (uint32_t)(q[2] & 0x1fffffu), 3);
    k.hi = (H << 1) | (L >> 62);
    k.lo = L << 2;
  } else {
    k.hi = interleave((uint32_t)(q[0] >> 32), (uint32_t)(q[1] >> 32), 0u, 2);
    k.lo = interleave((uint32_t)q[0], (uint32_t)q[1], 0u, 2);
  }
  k.lo = (k.lo & ~0xffffull) | idx;
  return k;
}

__device__ __forceinline__ Key shfl_xor_key(const Key &k, int j) {
  Key r;
  r.hi = __shfl_xor_sync(0xffffffffu, (unsigned long long)k.hi, j);
  r.lo = __shfl_xor_sync(0xffffffffu, (unsigned long long)k.lo, j);
  return r;
}

// Bitonic sort of the first `size` (a power of two, at least 32) keys of s, by
// the CTA.  The steps over distances below 32 stay in a warp's registers: 21
// barriers instead of 55 for 1,024 keys.
__device__ __forceinline__ void tile_sort(Key *s, int size) {
  const int lane = threadIdx.x & 31;
  // the steps k = k0 .. k1 over distances 16 .. 1, on rows of 32 keys
  auto rows = [&](int k0, int k1) {
    __syncthreads();
    for (int r = (int)threadIdx.x >> 5; r < size / 32; r += kWarpsPerCta) {
      const int e = r * 32 + lane;
      Key x = s[e];
      for (int k = k0; k <= k1; k <<= 1) {
        for (int j = k / 2 < 16 ? k / 2 : 16; j > 0; j >>= 1) {
          const Key y = shfl_xor_key(x, j);
          const bool keep_small = ((e & k) == 0) == ((lane & j) == 0);
          if (key_less(y, x) == keep_small) x = y;
        }
      }
      s[e] = x;
    }
  };
  rows(2, 32);
  for (int k = 64; k <= size; k <<= 1) {
    for (int j = k >> 1; j >= 32; j >>= 1) {
      __syncthreads();
      for (int t = threadIdx.x; t < size / 2; t += kThreads) {
        const int a = ((t & ~(j - 1)) << 1) | (t & (j - 1)), b = a | j;
        const Key x = s[a], y = s[b];
        if (key_less(y, x) == ((a & k) == 0)) {
          s[a] = y;
          s[b] = x;
        }
      }
    }
    rows(k, k);
  }
  __syncthreads();
}

// The rank of sorted-tile element e among all n: its place in its own tile
// plus the smaller keys of every other tile, one tile per lane of a group of
// kMaxTiles lanes, each by binary search.  Every lane of the warp calls.
__device__ __forceinline__ int merged_rank(const Key *tiles, int n, int tile, int e, const Key &key) {
  const int t = (int)(threadIdx.x & (kMaxTiles - 1));
  const int own = e / tile;
  int count = 0;
  const int begin = t * tile;
  if (t == own) {
    count = e - begin;
  } else if (begin < n) {
    int lo = 0, hi = n - begin < tile ? n - begin : tile;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      const Key m = tiles[begin + mid];
      if (key_less(m, key)) lo = mid + 1;
      else hi = mid;
    }
    count = lo;
  }
#pragma unroll
  for (int o = kMaxTiles / 2; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
  return count;
}

__device__ __forceinline__ float warp_min_any(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ float warp_max_any(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}
__device__ __forceinline__ uint32_t warp_min(uint32_t x) { return __reduce_min_sync(0xffffffffu, x); }

// Weights and bounds are compared as their bits (they are never negative):
// kNoBound lies above +inf, the weight of points farther apart than FP32 can
// square, which is an edge like any other.
__device__ __forceinline__ uint32_t box_bits(const float4 &p, const float4 &lo, const float4 &hi) {
  return __float_as_uint(box_dist(p.x, p.y, p.z, lo.x, lo.y, lo.z, hi.x, hi.y, hi.z));
}

// A warp's search for point p of component `me` within the cutoff r
// (inclusive).  Returns the best weight's bits `w`, its curve index `j` and
// original id `id` (j == kInvalid: none); `lb` is then the smallest rejected
// bound (kNoBound: no other component met).
struct Found {
  uint32_t w, j, id, lb;
};

__device__ __forceinline__ Found warp_search(const SmallArgs &A, const uint32_t *labels, const float4 &p,
                                             uint32_t me, uint32_t r) {
  const int lane = threadIdx.x & 31;
  const int nb = (A.n + 31) >> 5, ns = (nb + 31) >> 5;
  // this lane's best point
  uint32_t bw = kNoBound, bj = kInvalid, bid = kInvalid;
  uint32_t lb = kNoBound;  // the same on every lane, like r and found
  bool found = false;
  // a bound that ties the cutoff helps only with an id below the best one's
  auto best_id = [&]() { return warp_min(bw == r ? bid : kInvalid); };
  for (int s0 = 0; s0 < ns; s0 += 32) {
    uint32_t ds = kNoBound, smin = 0;
    if (s0 + lane < ns) {
      const float4 lo = A.sup[s0 + lane].lo, hi = A.sup[s0 + lane].hi;
      smin = __float_as_uint(hi.w);
      if (__float_as_uint(lo.w) != me) ds = box_bits(p, lo, hi);
    }
    for (;;) {
      uint32_t m = warp_min(ds);
      if (found && m == r) {
        const uint32_t b = best_id();
        if (ds == r && smin >= b) ds = kNoBound;
        m = warp_min(ds);
      }
      if (m > r || m == kNoBound) {
        lb = min(lb, m);
        break;
      }
      const int pick = __ffs(__ballot_sync(0xffffffffu, ds == m)) - 1;
      if (lane == pick) ds = kNoBound;
      const int b0 = (s0 + pick) << 5;
      uint32_t db = kNoBound, bmin = 0;
      if (b0 + lane < nb) {
        const float4 lo = A.blk[b0 + lane].lo, hi = A.blk[b0 + lane].hi;
        bmin = __float_as_uint(hi.w);
        if (__float_as_uint(lo.w) != me) db = box_bits(p, lo, hi);
      }
      for (;;) {
        uint32_t mb = warp_min(db);
        if (found && mb == r) {
          const uint32_t b = best_id();
          if (db == r && bmin >= b) db = kNoBound;
          mb = warp_min(db);
        }
        if (mb > r || mb == kNoBound) {
          lb = min(lb, mb);
          break;
        }
        const int pb = __ffs(__ballot_sync(0xffffffffu, db == mb)) - 1;
        if (lane == pb) db = kNoBound;
        const int k = ((b0 + pb) << 5) + lane;
        uint32_t d = kNoBound;
        if (k < A.n && labels[k] != me) {
          const float4 t = A.pts[k];
          d = __float_as_uint(sq_dist(p.x, p.y, p.z, t.x, t.y, t.z));
          const uint32_t id = __float_as_uint(t.w);
          if (d <= r && (d < bw || (d == bw && id < bid))) {
            bw = d;
            bj = (uint32_t)k;
            bid = id;
          }
        }
        const uint32_t md = warp_min(d);
        if (md != kNoBound && md <= r) {
          found = true;
          r = md;
        } else {
          lb = min(lb, md);
        }
      }
    }
  }
  Found f;
  f.lb = lb;
  f.w = warp_min(bw);
  const bool cand = bj != kInvalid && bw == f.w;
  f.id = warp_min(cand ? bid : kInvalid);
  const unsigned who = __ballot_sync(0xffffffffu, cand && bid == f.id);
  f.j = who ? __shfl_sync(0xffffffffu, bj, __ffs(who) - 1) : kInvalid;
  return f;
}

// The component minimum's update of traverse.cuh (offer_best), on arrays that
// this kernel also writes: no loads through the read-only path.
__device__ __forceinline__ uint32_t best_weight(const CompBest *c) {
  return (uint32_t)(__ldcg(reinterpret_cast<const unsigned long long *>(&c->key)) >> 32);
}
__device__ __forceinline__ void offer(CompBest *c, uint32_t w, uint32_t oi, uint32_t oj, uint32_t label,
                                      uint32_t *status) {
  CompBest want, cur;
  want.key = ((uint64_t)w << 32) | (uint64_t)min(oi, oj);
  want.mx = ((uint64_t)max(oi, oj) << 32) | (uint64_t)label;
  cur.key = __ldcg(reinterpret_cast<const unsigned long long *>(&c->key));
  if (want.key > cur.key) return;
  cur.mx = __ldcg(reinterpret_cast<const unsigned long long *>(&c->mx));
  for (int it = 0; it < (1 << 20); ++it) {
    if (want.key > cur.key || (want.key == cur.key && want.mx >= cur.mx)) return;
    const CompBest old = atomicCAS(c, cur, want);
    if (old.key == cur.key && old.mx == cur.mx) return;
    cur = old;
  }
  atomicOr(status, kErrCas);
}

// A warp's box of the points [first, first + 32 rows) with its smallest id.
__device__ __forceinline__ void write_box(const SmallArgs &A, int first, int rows, uint32_t label, BoxRec *out) {
  const int lane = threadIdx.x & 31;
  const float kInf = __int_as_float(0x7f800000);
  float lo[3] = {kInf, kInf, kInf}, hi[3] = {-kInf, -kInf, -kInf};
  uint32_t id = 0xffffffffu;
  for (int r = 0; r < rows; ++r) {
    const int k = first + r * 32 + lane;
    if (k < A.n) {
      const float4 t = A.pts[k];
      lo[0] = fminf(lo[0], t.x); lo[1] = fminf(lo[1], t.y); lo[2] = fminf(lo[2], t.z);
      hi[0] = fmaxf(hi[0], t.x); hi[1] = fmaxf(hi[1], t.y); hi[2] = fmaxf(hi[2], t.z);
      id = min(id, __float_as_uint(t.w));
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    lo[q] = warp_min_any(lo[q]);
    hi[q] = warp_max_any(hi[q]);
  }
  id = __reduce_min_sync(0xffffffffu, id);
  if (lane == 0) {
    out->lo = make_float4(lo[0], lo[1], lo[2], __uint_as_float(label));
    out->hi = make_float4(hi[0], hi[1], hi[2], __uint_as_float(id));
  }
}

__global__ void __launch_bounds__(kThreads, 2) k_small(SmallArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Key *s_keys = reinterpret_cast<Key *>(smem_raw);
  uint4 *todo = reinterpret_cast<uint4 *>(smem_raw);  // (between the sorts: at most 32 entries per warp)
  __shared__ double s_lo[3], s_scale[3];
  __shared__ uint32_t s_cnt[kWarpsPerCta];
  __shared__ uint32_t s_base;
  __shared__ int s_todo, s_taken;
  const float kInf = __int_as_float(0x7f800000);
  const int tid = threadIdx.x, lane = tid & 31;
  const int gtid = blockIdx.x * kThreads + tid, gthreads = gridDim.x * kThreads;
  // warps in an order that spreads consecutive ones over the CTAs
  const int gwarp = (tid >> 5) * gridDim.x + blockIdx.x, gwarps = gthreads >> 5;
  const int n = A.n, dim = A.dim;
  uint32_t *counters = A.counters, *status = A.counters + 1, *bar = A.counters + 8;
  uint32_t phase = 0;

  // --- scene box (counters start at zero: minima kept as maxima of ~bits)
  {
    float lo[3] = {kInf, kInf, kInf}, hi[3] = {-kInf, -kInf, -kInf};
    bool bad = false;
    for (int k = gtid; k < n; k += gthreads) {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (q >= dim) continue;
        const float x = A.src[k * dim + q];
        if (A.copy) A.copy[k * dim + q] = x;
        if (!isfinite(x)) { bad = true; continue; }
        lo[q] = fminf(lo[q], x);
        hi[q] = fmaxf(hi[q], x);
      }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(status, kErrNonFinite);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (q >= dim) continue;
      const uint32_t l = __reduce_max_sync(0xffffffffu, lo[q] <= hi[q] ? ~float_to_ordered(lo[q]) : 0u);
      const uint32_t h = __reduce_max_sync(0xffffffffu, lo[q] <= hi[q] ? float_to_ordered(hi[q]) : 0u);
      if (lane == 0 && h != 0u) {
        atomicMax(counters + 2 + q, l);
        atomicMax(counters + 5 + q, h);
      }
    }
  }
  if (!grid_barrier(bar, status, phase)) return;
  if (__ldcg(status) != 0u) return;  // non-finite input: the same value for every CTA
  const float *src = A.copy ? A.copy : A.src;
  if (tid < dim) {  // (the FP64 divisions here, not per point: few FP64 units)
    const double twoB = dim == 3 ? 4398046511104.0 : 18446744073709551616.0;
    const double lo = (double)ordered_to_float(~__ldcg(counters + 2 + tid));
    const double ext = __dsub_rn((double)ordered_to_float(__ldcg(counters + 5 + tid)), lo);
    s_lo[tid] = lo;
    s_scale[tid] = ext > 0.0 ? __ddiv_rn(twoB, ext) : 0.0;
  }
  __syncthreads();

  // --- curve keys, sorted tile by tile
  const int tile = A.tile, ntiles = (n + tile - 1) / tile;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const int begin = t * tile, cnt = n - begin < tile ? n - begin : tile;
    int size = 32;
    while (size < cnt) size <<= 1;
    for (int i = tid; i < size; i += kThreads) {
      Key k = {~0ull, ~0ull};
      if (i < cnt) {
        const int idx = begin + i;
        float x[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int q = 0; q < 3; ++q)
          if (q < dim) x[q] = src[idx * dim + q];
        k = curve_key(x, s_lo, s_scale, dim, (uint32_t)idx);
      }
      s_keys[i] = k;
    }
    tile_sort(s_keys, size);
    for (int i = tid; i < cnt; i += kThreads) A.tiles[begin + i] = s_keys[i];
    __syncthreads();
  }
  if (!grid_barrier(bar, status, phase)) return;

  // --- the tiles merged by rank; points, labels and round state in curve order
  const int group = lane / kMaxTiles, groups = 32 / kMaxTiles;
  for (int e0 = gwarp * groups; e0 < n; e0 += gwarps * groups) {
    const int e = e0 + group;
    Key k = {0, 0};
    if (e < n) k = A.tiles[e];
    const int rank = merged_rank(A.tiles, n, tile, e < n ? e : n - 1, k);
    if (e < n && (lane & (kMaxTiles - 1)) == 0) {
      const uint32_t idx = (uint32_t)(k.lo & 0xffffu);
      const float *s = src + (int)idx * dim;
      A.pts[rank] = make_float4(s[0], s[1], dim == 3 ? s[2] : 0.f, __uint_as_float(idx));
      A.labels[0][rank] = (uint32_t)rank;
      CompBest empty;
      empty.key = kEmptyKey;
      empty.mx = kEmptyKey;
      A.comp[0][rank] = empty;
    }
  }
  if (!grid_barrier(bar, status, phase)) return;

  // --- boxes of blocks and superblocks; the first round's curve-pair bounds
  const int nb = (n + 31) >> 5, ns = (nb + 31) >> 5;
  for (int b = gwarp; b < nb + ns; b += gwarps) {
    if (b >= nb) {
      const int s = b - nb;
      write_box(A, s * 1024, 32, n - s * 1024 == 1 ? (uint32_t)(n - 1) : kInvalid, A.sup + s);
    } else {
      const int k = b * 32 + lane;
      write_box(A, b * 32, 1, n - b * 32 == 1 ? (uint32_t)(n - 1) : kInvalid, A.blk + b);
      if (k < n) {
        const float4 t = A.pts[k];
        float w = kInf;
        if (k > 0) {
          const float4 u = A.pts[k - 1];
          w = sq_dist(u.x, u.y, u.z, t.x, t.y, t.z);
        }
        if (k + 1 < n) {
          const float4 u = A.pts[k + 1];
          w = fminf(w, sq_dist(t.x, t.y, t.z, u.x, u.y, u.z));
        }
        A.bound[0][k] = __float_as_uint(w);
      }
    }
  }
  if (!grid_barrier(bar, status, phase)) return;

  // --- Boruvka rounds
  int limit = 1;
  while ((1 << (limit - 1)) < n) ++limit;  // ceil(log2 n) + 1
  ++limit;
  // curve positions a warp looks at together
  int chunk = (n + gwarps - 1) / gwarps;
  if (chunk > 32) chunk = 32;
  for (int round = 0;; ++round) {
    if (round >= limit) {
      if (gtid == 0) atomicOr(status, kErrChain);
      return;
    }
    const int cur = round & 1;
    const uint32_t *labels = A.labels[cur];
    const uint32_t *bound = A.bound[cur];
    CompBest *comp = A.comp[cur];
    // queries: every warp looks at its positions, the CTA's warps share those
    // that need a search (neighbours on the curve often all do, or none)
    for (int base = 0; base < n; base += gwarps * chunk) {
      const int i = base + gwarp * chunk + lane;
      bool act = false;
      uint32_t me = 0;
      uint2 prev = make_uint2(0u, kInvalid);
      if (lane < chunk && i < n) {
        me = labels[i];
        if (round > 0) prev = A.res[i];
        if (prev.x <= min(bound[me], best_weight(comp + me))) {
          // the nearest neighbour found in an earlier round is still the nearest
          // while it lies in another component: components only grow
          const uint32_t other = prev.y != kInvalid ? labels[prev.y] : me;
          if (other != me) {
            if (prev.x <= best_weight(comp + me))
              offer(comp + me, prev.x, __float_as_uint(A.pts[i].w), __float_as_uint(A.pts[prev.y].w), other,
                    status);
          } else {
            act = true;
          }
        }
      }
      if (tid == 0) s_todo = s_taken = 0;
      __syncthreads();
      const unsigned b = __ballot_sync(0xffffffffu, act);
      int at = 0;
      if (lane == 0 && b) at = atomicAdd(&s_todo, __popc(b));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(b & ((1u << lane) - 1u));
      if (act) todo[at] = make_uint4((uint32_t)i, me, prev.x, 0u);
      __syncthreads();
      const int count = s_todo;
      for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(&s_taken, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= count) break;
        const uint4 e = todo[t];
        const int q = (int)e.x;
        const uint32_t r0 = __shfl_sync(0xffffffffu, min(bound[e.y], best_weight(comp + e.y)), 0);
        if (e.z > r0) continue;
        const float4 p = A.pts[q];
        const Found f = warp_search(A, labels, p, e.y, r0);
        if (lane == 0) {
          // nothing within r0: the smallest rejected bound is a lower bound of
          // the nearest other component from here on
          const uint32_t lb = f.lb != kNoBound ? f.lb : (r0 != kNoBound ? r0 : 0u);
          A.res[q] = make_uint2(f.j != kInvalid ? f.w : lb, f.j);
          if (f.j != kInvalid) offer(comp + e.y, f.w, __float_as_uint(p.w), f.id, labels[f.j], status);
        }
        __syncwarp();
      }
      __syncthreads();
    }
    if (!grid_barrier(bar, status, phase)) return;
    // merge: one thread per component (a label is the position of one of its points)
    for (int c0 = blockIdx.x * kThreads; c0 < n; c0 += gthreads) {
      const int c = c0 + tid;
      bool emit = false;
      Key ek = {0, 0};
      if (c < n && labels[c] == (uint32_t)c) {
        const CompBest b = comp[c];
        const uint32_t t = b.key == kEmptyKey ? kInvalid : (uint32_t)b.mx;
        uint32_t r = (uint32_t)c;
        emit = t != kInvalid;
        if (t != kInvalid) {
          uint32_t x = (uint32_t)c, y = t;
          for (int steps = 0;; ++steps) {
            const CompBest cb = comp[y];
            if (cb.key == kEmptyKey) { r = y; break; }
            const uint32_t z = (uint32_t)cb.mx;
            if (steps == 0) emit = z != x || x < y;
            if (z == x) { r = x < y ? x : y; break; }
            x = y;
            y = z;
            if (steps > n) { atomicOr(status, kErrChain); r = x; break; }
          }
          if (emit) ek.hi = (b.key & 0xffffffff00000000ull) | ((b.key & 0xffffull) << 16) | (b.mx >> 32);
        }
        CompBest empty;
        empty.key = kEmptyKey;
        empty.mx = kEmptyKey;
        A.comp[cur ^ 1][c] = empty;
        A.root[c] = r;
        if (r == (uint32_t)c) A.bound[cur ^ 1][c] = kNoBound;
      }
      const unsigned be = __ballot_sync(0xffffffffu, emit);
      if (lane == 0) s_cnt[tid >> 5] = __popc(be);
      __syncthreads();
      if (tid == 0) {
        uint32_t tot = 0;
        for (int w = 0; w < kWarpsPerCta; ++w) {
          const uint32_t v = s_cnt[w];
          s_cnt[w] = tot;
          tot += v;
        }
        s_base = tot ? atomicAdd(counters, tot) : 0u;
      }
      __syncthreads();
      const uint32_t at = s_base + s_cnt[tid >> 5] + __popc(be & ((1u << lane) - 1u));
      if (emit && at < (uint32_t)n) A.ekeys[at] = ek;
      __syncthreads();
    }
    if (!grid_barrier(bar, status, phase)) return;
    const uint32_t emitted = __ldcg(counters);
    if (emitted >= (uint32_t)(n - 1) || __ldcg(status) != 0u) break;  // (the same for every CTA)
    // relabel, the next round's curve-pair bounds, block and superblock labels
    for (int b = gwarp; b < nb + ns; b += gwarps) {
      if (b >= nb) {
        const int s = b - nb;
        uint32_t mn = 0xffffffffu, mx = 0u;
        for (int q = 0; q < 32; ++q) {
          const int k = s * 1024 + q * 32 + lane;
          if (k < n) {
            const uint32_t l = A.root[labels[k]];
            mn = min(mn, l);
            mx = max(mx, l);
          }
        }
        mn = __reduce_min_sync(0xffffffffu, mn);
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) A.sup[s].lo.w = __uint_as_float(mn == mx ? mn : kInvalid);
      } else {
        const int k = b * 32 + lane;
        const uint32_t l = k < n ? A.root[labels[k]] : kInvalid;
        uint32_t nxt = __shfl_down_sync(0xffffffffu, l, 1);
        if (lane == 31) nxt = k + 1 < n ? A.root[labels[k + 1]] : kInvalid;
        if (k < n) A.labels[cur ^ 1][k] = l;
        if (k + 1 < n && l != nxt) {
          const float4 t = A.pts[k], u = A.pts[k + 1];
          const uint32_t w = __float_as_uint(sq_dist(t.x, t.y, t.z, u.x, u.y, u.z));
          atomicMin(A.bound[cur ^ 1] + l, w);
          atomicMin(A.bound[cur ^ 1] + nxt, w);
        }
        const uint32_t mn = __reduce_min_sync(0xffffffffu, l);
        const uint32_t mx = __reduce_max_sync(0xffffffffu, k < n ? l : 0u);
        if (lane == 0) A.blk[b].lo.w = __uint_as_float(mn == mx ? mn : kInvalid);
      }
    }
    if (!grid_barrier(bar, status, phase)) return;
  }
  if (__ldcg(status) != 0u) return;

  // --- the edges in (w, i, j) order: the key holds all three
  const int m = n - 1;
  for (int t = blockIdx.x; t < (m + tile - 1) / tile; t += gridDim.x) {
    const int begin = t * tile, cnt = m - begin < tile ? m - begin : tile;
    int size = 32;
    while (size < cnt) size <<= 1;
    for (int i = tid; i < size; i += kThreads) {
      Key k = {~0ull, ~0ull};
      if (i < cnt) k = A.ekeys[begin + i];
      s_keys[i] = k;
    }
    tile_sort(s_keys, size);
    for (int i = tid; i < cnt; i += kThreads) A.tiles[begin + i] = s_keys[i];
    __syncthreads();
  }
  if (!grid_barrier(bar, status, phase)) return;
  for (int e0 = gwarp * groups; e0 < m; e0 += gwarps * groups) {
    const int e = e0 + group;
    Key k = {0, 0};
    if (e < m) k = A.tiles[e];
    const int rank = merged_rank(A.tiles, m, tile, e < m ? e : m - 1, k);
    if (e < m && (lane & (kMaxTiles - 1)) == 0) {
      emst_edge E;
      E.i = (uint32_t)(k.hi >> 16) & 0xffffu;
      E.j = (uint32_t)k.hi & 0xffffu;
      E.w = __uint_as_float((uint32_t)(k.hi >> 32));
      A.out[rank] = E;
    }
  }
}

}  // namespace

int small_emst(const float *points, int64_t n64, int dim, emst_edge *out, cudaStream_t stream) {
  const int n = (int)n64;
  const bool pts_dev = device_accessible(points), out_dev = device_accessible(out);
  // pinned host buffers are read and written in place, pageable ones staged
  const float *pts_map = pts_dev ? nullptr : static_cast<const float *>(mapped_host(points));
  emst_edge *out_map = out_dev ? nullptr : static_cast<emst_edge *>(mapped_host(out));
  const bool out_staged = !out_dev && !out_map;
  // scratch
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 255) & ~size_t(255);
    const size_t at = off;
    off += bytes;
    return at;
  };
  const int nb = (n + 31) / 32, ns = (nb + 31) / 32;
  const size_t o_counters = take(256), o_tiles = take(sizeof(Key) * n), o_pts = take(16 * (size_t)n),
               o_l0 = take(4 * (size_t)n), o_l1 = take(4 * (size_t)n), o_b0 = take(4 * (size_t)n),
               o_b1 = take(4 * (size_t)n), o_c0 = take(16 * (size_t)n), o_c1 = take(16 * (size_t)n),
               o_root = take(4 * (size_t)n), o_res = take(8 * (size_t)n), o_blk = take(sizeof(BoxRec) * nb),
               o_sup = take(sizeof(BoxRec) * ns), o_ek = take(sizeof(Key) * n),
               o_copy = take(pts_dev ? 0 : sizeof(float) * (size_t)n * dim),
               o_out = take(out_staged ? sizeof(emst_edge) * (size_t)n : 0);
  char *base = nullptr;
  if (scratch_alloc((void **)&base, off + 256, stream) != cudaSuccess) return EMST_ERR_OOM;
  SmallArgs A;
  A.n = n;
  A.dim = dim;
  A.tile = n <= kMaxTiles * 1024 ? 1024 : kMaxTile;
  A.counters = reinterpret_cast<uint32_t *>(base + o_counters);
  A.tiles = reinterpret_cast<Key *>(base + o_tiles);
  A.pts = reinterpret_cast<float4 *>(base + o_pts);
  A.labels[0] = reinterpret_cast<uint32_t *>(base + o_l0);
  A.labels[1] = reinterpret_cast<uint32_t *>(base + o_l1);
  A.bound[0] = reinterpret_cast<uint32_t *>(base + o_b0);
  A.bound[1] = reinterpret_cast<uint32_t *>(base + o_b1);
  A.comp[0] = reinterpret_cast<CompBest *>(base + o_c0);
  A.comp[1] = reinterpret_cast<CompBest *>(base + o_c1);
  A.root = reinterpret_cast<uint32_t *>(base + o_root);
  A.res = reinterpret_cast<uint2 *>(base + o_res);
  A.blk = reinterpret_cast<BoxRec *>(base + o_blk);
  A.sup = reinterpret_cast<BoxRec *>(base + o_sup);
  A.ekeys = reinterpret_cast<Key *>(base + o_ek);
  float *copy = reinterpret_cast<float *>(base + o_copy);
  A.out = out_dev ? out : out_map ? out_map : reinterpret_cast<emst_edge *>(base + o_out);
  A.src = pts_dev ? points : pts_map ? pts_map : copy;
  A.copy = pts_map ? copy : nullptr;
  int rc = EMST_OK;
  uint32_t host[2] = {0, 0};
  const size_t smem = sizeof(Key) * (size_t)A.tile;
  static int ctas_per_sm[64][2];  // by device and tile size, looked up once (every thread finds the same)
  int dev = 0;
  cudaGetDevice(&dev);
  const int kind = A.tile == kMaxTile ? 1 : 0;
  int occ = dev >= 0 && dev < 64 ? ctas_per_sm[dev][kind] : 0;
  bool ok = true;
  if (occ == 0) {
    ok = cudaFuncSetAttribute(k_small, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(sizeof(Key) * (size_t)kMaxTile)) == cudaSuccess &&
         cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_small, kThreads, smem) == cudaSuccess && occ >= 1;
    if (ok && dev >= 0 && dev < 64) ctas_per_sm[dev][kind] = occ;
  }
  if (ok) {
    // a warp per query while the GPU holds that many
    int grid = stream_sm_count(stream) * occ;
    const int want = (n + kWarpsPerCta - 1) / kWarpsPerCta;
    if (grid > want) grid = want;
    ok = cudaMemsetAsync(A.counters, 0, 256, stream) == cudaSuccess;
    if (A.src == copy)
      ok = ok && cudaMemcpyAsync(copy, points, sizeof(float) * (size_t)n * dim, cudaMemcpyHostToDevice,
                                 stream) == cudaSuccess;
    void *args[] = {&A};
    auto launch = [&](unsigned g) {
      return cudaLaunchCooperativeKernel(k_small, dim3(g), dim3(kThreads), args, smem, stream);
    };
    ok = ok && launch_cooperative(grid, launch) == cudaSuccess;
    if (ok && out_staged)
      ok = cudaMemcpyAsync(out, A.out, sizeof(emst_edge) * (size_t)(n - 1), cudaMemcpyDeviceToHost,
                           stream) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(host, A.counters, sizeof(host), cudaMemcpyDeviceToHost, stream) == cudaSuccess &&
         cudaStreamSynchronize(stream) == cudaSuccess;
  }
  if (!ok) rc = EMST_ERR_CUDA;
  else if (host[1] != 0) rc = status_from_bits(host[1]);
  else if (host[0] != (uint32_t)(n - 1)) rc = EMST_ERR_INTERNAL;
  cudaFreeAsync(base, stream);
  if (rc == EMST_ERR_CUDA) cudaGetLastError();
  return rc;
}

}  // namespace emst
