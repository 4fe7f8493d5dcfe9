// dendrogram.cu -- the single-linkage dendrogram of a spanning tree: the
// hierarchy that single-linkage clustering and HDBSCAN* read off the EMST
// (the introduction names clustering as a consumer; §4.5 builds the
// mutual-reachability tree for HDBSCAN*).
//
// Definition: Kruskal's merge sequence (§2, "MST computation") over the
// tree's own edges in the given order (non-decreasing weight).  Edge k makes
// cluster n + k.  The parent of edge k is the first later edge that touches
// C(k), the component of edges 0..k holding k.  A point's parent is its
// lowest-ranked incident edge.
//
// The merge sequence is serial (its depth is the height of the hierarchy,
// which single linkage makes long by chaining).  Here the tree is contracted
// as Boruvka's algorithm would, and the contracted edges are put back into
// chains (the idea of parallel dendrograms by recursive tree contraction):
//  - Level 0 is the tree itself.  At every level, each vertex takes its
//    lowest-ranked edge; the edges taken are contracted, the components they
//    form are the vertices of the next level and the edges left are its
//    edges.  Every level at least halves the vertices.
//  - A contracted edge x = (u, v) that u took has u alone on one side when it
//    merges (every other edge of u ranks above x), so within its component
//    the contracted edges form one chain in rank order, and they lie on the
//    path from that component, a leaf of the next level's hierarchy, up to
//    the root: x belongs below the first edge on that path that ranks above
//    it.  Going up the levels, that is the first component S holding x whose
//    own taken edge p ranks above x.  All edges with the same S form one
//    chain, ordered by rank, whose last one hangs under p on S's side.
//  - So the hierarchy is one sort of the edges by (S, rank).  Of two chain
//    neighbours the lower hangs under the higher, on the side of the higher
//    one that no vertex took it from.
//  - Sizes: x adds to its chain the points of the side(s) that took it: the
//    total of the chain that ends there, or one point when it is empty.
//    Those chains hold edges of lower levels only, so the totals follow level
//    by level, and a cluster's size is the running total along its chain.
// An edge's two sides are its endpoint slots 2k + side.
//
// Work is proportional to the edges (each level at most half the one before)
// plus one sort, where splitting the ranks in halves took every edge through
// every one of log2(n) levels.  Measured, whole call, halving / this: EMST
// tree of 8M halo points 5,665 / 2,361 us, of 6M 4,454 / 1,651, of 300,000
// 604 / 366; mutual-reachability tree (k_pts 8) of 6M 7,798 / 1,508.  What
// bounds it: scattered accesses (the contraction's walks and lowest-slot
// updates 1.29 ms of the 8M call, the sort 0.27, the scattered results 0.35).
#include <utility>

#include "grid.cuh"

namespace emst {
namespace {

constexpr int kDgBlock = 256;
constexpr int kContractThreads = 512;
constexpr int kContractWarps = kContractThreads / 32;
constexpr int kMaxLevels = 32;      // vertices at least halve: 31 levels reach any n
constexpr uint32_t kTook = 0x80000000u;  // a vertex id's flag: this endpoint took the edge

// A bijective mix of a vertex id (the MurmurHash3 32-bit finaliser): the
// union-find hooks the root of higher priority under the other, so trees
// stay shallow in expectation whatever order the vertices are united in
// (linking by random index).
__device__ __forceinline__ uint32_t prio(uint32_t x) {
  x ^= x >> 16;
  x *= 0x85ebca6bu;
  x ^= x >> 13;
  x *= 0xc2b2ae35u;
  x ^= x >> 16;
  return x;
}

// Root of x, optionally halving the path.  Every parent has a lower
// priority than its child and a parent is only ever replaced by an
// ancestor, so a walk is strictly descending and ends even when it reads
// stale (cached) entries: a stale entry is still an ancestor.  A stale root
// is caught by the hook's compare-and-swap in uf_unite.
template <bool HALVE>
__device__ __forceinline__ uint32_t uf_find(uint32_t *uf, uint32_t x) {
  for (;;) {
    const uint32_t p = uf[x];
    if (p == x) return x;
    const uint32_t g = uf[p];
    if (g == p) return p;
    if (HALVE) uf[x] = g;
    x = g;
  }
}

// The roots of a and b, the two walks advanced together so that their
// loads are in flight at once (each walk as in uf_find).
template <bool HALVE>
__device__ __forceinline__ void uf_find2(uint32_t *uf, uint32_t &a, uint32_t &b) {
  bool da = false, db = false;
  while (!(da && db)) {
    const uint32_t pa = da ? a : uf[a];
    const uint32_t pb = db ? b : uf[b];
    if (!da && pa == a) da = true;
    if (!db && pb == b) db = true;
    const uint32_t ga = da ? a : uf[pa];
    const uint32_t gb = db ? b : uf[pb];
    if (!da) {
      if (ga == pa) { a = pa; da = true; }
      else { if (HALVE) uf[a] = ga; a = ga; }
    }
    if (!db) {
      if (gb == pb) { b = pb; db = true; }
      else { if (HALVE) uf[b] = gb; b = gb; }
    }
  }
}

// Joins the sets of a and b, lock-free.  A failed hook returns the hooked
// root's actual parent, and the walk resumes there, so each retry climbs the
// real chain.  Hooking the higher-priority root under the other cannot close
// a cycle even when the other is stale: its actual root has a still lower
// priority.  False only if the retry bound runs out.
__device__ __forceinline__ bool uf_unite(uint32_t *uf, uint32_t a, uint32_t b) {
  uf_find2<true>(uf, a, b);
  for (int it = 0; it < (1 << 22); ++it) {
    if (a == b) return true;
    const bool ah = prio(a) > prio(b);
    const uint32_t hi = ah ? a : b, lo = ah ? b : a;
    const uint32_t old = atomicCAS(uf + hi, hi, lo);
    if (old == hi) return true;
    if (ah) a = uf_find<true>(uf, old);
    else b = uf_find<true>(uf, old);
  }
  return false;
}

// Adds v to a[idx] from a warp.  In up to two rounds, the lanes that share
// the target of the lowest remaining lane (the edges of one long chain) sum
// their values and one of them adds.  Lanes left after two rounds add on
// their own.  Every lane of the warp calls; `want` selects the participants.
__device__ __forceinline__ void warp_add(uint32_t *a, uint32_t idx, uint32_t v, bool want) {
  unsigned act = __ballot_sync(0xffffffffu, want);
  if (!want) return;
  const int lane = (int)(threadIdx.x & 31);
#pragma unroll
  for (int round = 0; round < 2; ++round) {
    const int leader = __ffs(act) - 1;
    const uint32_t lead_idx = __shfl_sync(act, idx, leader);
    const unsigned same = __ballot_sync(act, idx == lead_idx);
    if (idx == lead_idx) {
      const uint32_t r = __reduce_add_sync(same, v);
      if (lane == leader) atomicAdd(a + idx, r);
      return;
    }
    act &= ~same;
  }
  atomicAdd(a + idx, v);
}

// A vertex of any level (ids continue from level to level: points 0..n-1,
// then each level's components): x the lowest slot of an edge touching it
// (the edge it takes; kInvalid at the top), y the component of the next level
// that holds it.
// Work lists are 16-byte rows {rank, vertex of side 0, vertex of side 1, -}.
struct Contract {
  const emst_edge *e;
  int64_t n, m;
  uint2 *node;         // 2n
  uint32_t *uf;        // 2n
  uint32_t *total;     // n: points below each chain, by component id - n
  uint4 *rest[2];      // m / 2 + 1: the edges of a level above 0, alternating
  uint4 *done;         // m: contracted edges in level order, vertices flagged kTook
  uint64_t *keys;      // m, by rank: (chain << 32) | slot where the chain goes on below
  uint32_t *vals;      // m, by rank: points the edge adds to its chain
  uint32_t *child;     // 2m or null: the cluster on each slot
  uint32_t *out_parent;  // n + m or null
  uint32_t *counters;  // [1] status, [2] invalid input found before the contraction, [40] barrier
  uint32_t *per_level; // 4 x kMaxLevels: components, edges left, edges done, errors
};

// Input checks (ids below n, no loop edge, no NaN weight, weights not
// decreasing) and, in the same pass, every point's lowest slot.
__global__ void k_dg_check(const emst_edge *__restrict__ e, int64_t m, int64_t n, uint2 *node,
                           uint32_t *__restrict__ uf, uint32_t *counters) {
  wait_for_previous();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) uf[k] = (uint32_t)k;
  if (k >= m) return;
  const emst_edge x = e[k];
  bool bad = x.i >= n || x.j >= n || x.i == x.j || !(x.w == x.w);
  if (k + 1 < m && e[k + 1].w < x.w) bad = true;
  if (bad) {
    atomicOr(counters + 1, kErrBadInput);
    counters[2] = 1u;
    return;
  }
  const uint32_t s = 2 * (uint32_t)k;
  if (node[x.i].x > s) atomicMin(&node[x.i].x, s);
  if (node[x.j].x > s + 1) atomicMin(&node[x.j].x, s + 1);
}

// Places of this thread's entries in a list: one atomic per CTA.  Every
// thread of the CTA calls; s_cnt has kContractWarps + 1 words.
__device__ __forceinline__ uint32_t append_place(bool want, uint32_t *counter, uint32_t *s_cnt) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned b = __ballot_sync(0xffffffffu, want);
  if (lane == 0) s_cnt[warp] = __popc(b);
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t v = lane < kContractWarps ? s_cnt[lane] : 0u;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    uint32_t base = 0;
    if (lane == 31 && x) base = atomicAdd(counter, x);
    base = __shfl_sync(0xffffffffu, base, 31);
    if (lane < kContractWarps) s_cnt[lane] = base + x - v;
  }
  __syncthreads();
  const uint32_t at = s_cnt[warp] + __popc(b & ((1u << lane) - 1u));
  __syncthreads();
  return at;
}

// All levels of the contraction, then the chains and their totals, in one
// cooperative launch: the levels' sizes are known only on the device, and the
// upper ones are too small to be worth launches of their own.
__global__ void __launch_bounds__(kContractThreads, 3) k_dg_contract(Contract A) {
  __shared__ uint32_t s_cnt[kContractWarps + 1];
  const int64_t gthreads = (int64_t)gridDim.x * kContractThreads;
  const int64_t first = (int64_t)blockIdx.x * kContractThreads;
  const int tid = threadIdx.x;
  uint32_t *status = A.counters + 1, *bar = A.counters + 40;
  uint32_t *c_comp = A.per_level, *c_rest = c_comp + kMaxLevels, *c_done = c_rest + kMaxLevels,
           *c_err = c_done + kMaxLevels;
  uint32_t phase = 0;
  if (__ldcg(A.counters + 2) != 0u) return;  // (written before this launch only)
  const int64_t ids = 2 * A.n;       // room for vertex ids: every level halves
  const int64_t room = A.m / 2 + 1;  // and for the edges of a level above 0
  int64_t base = 0, nv = A.n, ne = A.m, dstart = 0;
  int levels = 0;
  for (int lv = 0; ne > 0 && lv < kMaxLevels; ++lv) {
    const uint4 *rest = A.rest[lv & 1];
    uint4 *next = A.rest[(lv + 1) & 1];
    // the edges some endpoint takes are contracted, the others left
    for (int64_t b = first; b < ne; b += gthreads) {
      const int64_t t = b + tid;
      bool take = false, keep = false;
      uint4 row = make_uint4(0, 0, 0, 0);
      if (t < ne) {
        if (lv == 0) {
          const emst_edge x = A.e[t];
          row = make_uint4((uint32_t)t, x.i, x.j, 0u);
        } else {
          row = rest[t];
        }
        const uint32_t u = row.y, v = row.z;
        const bool tu = A.node[u].x >> 1 == row.x, tv = A.node[v].x >> 1 == row.x;
        take = tu || tv;
        keep = !take;
        if (take) {
          if (!uf_unite(A.uf, u, v)) atomicOr(status, kErrSpin);
          row.y |= tu ? kTook : 0u;
          row.z |= tv ? kTook : 0u;
        }
      }
      const uint32_t d = append_place(take, c_done + lv, s_cnt);
      if (take) A.done[dstart + d] = row;
      const uint32_t r = append_place(keep, c_rest + lv, s_cnt);
      if (keep) {
        if (r < room) next[r] = row;
        else atomicOr(c_err + lv, 1u);  // more edges than half the vertices: not a tree
      }
    }
    if (!grid_barrier(bar, status, phase)) return;
    // a component per remaining root; a vertex without an edge: not a tree
    for (int64_t b = first; b < nv; b += gthreads) {
      const int64_t v = base + b + tid;
      const bool root = b + tid < nv && A.uf[v] == (uint32_t)v;
      const uint32_t id = append_place(root, c_comp + lv, s_cnt);
      if (b + tid < nv) {
        const uint32_t s = A.node[v].x;
        if (s == kInvalid) atomicOr(c_err + lv, 1u);
        if (root) {
          const int64_t g = base + nv + id;
          if (g < ids) {
            A.node[v].y = (uint32_t)g;
            A.uf[g] = (uint32_t)g;
          } else {
            atomicOr(c_err + lv, 1u);
          }
        }
        if (lv == 0 && s != kInvalid) {  // the points' own places in the result
          if (A.out_parent) A.out_parent[v] = (uint32_t)A.n + (s >> 1);
          if (A.child) A.child[s] = (uint32_t)v;
        }
      }
    }
    if (!grid_barrier(bar, status, phase)) return;
    if (__ldcg(c_err + lv) != 0u) {  // (nothing writes this level's word any more: the same for every CTA)
      if (first == 0 && tid == 0) atomicOr(status, kErrBadInput);
      return;
    }
    const int64_t left = (int64_t)__ldcg(c_rest + lv), comps = (int64_t)__ldcg(c_comp + lv);
    // every vertex's component; the remaining edges between components, and
    // each component's lowest slot
    for (int64_t t = first + tid; t < nv; t += gthreads) {
      const uint32_t v = (uint32_t)(base + t), r = uf_find<true>(A.uf, v);
      if (r != v) A.node[v].y = A.node[r].y;
    }
    for (int64_t t = first + tid; t < left; t += gthreads) {
      uint4 row = next[t];
      uint32_t u = row.y, v = row.z;
      uf_find2<true>(A.uf, u, v);
      if (u == v) {  // an edge inside a component: it closes a cycle
        if (lv + 1 < kMaxLevels) atomicOr(c_err + lv + 1, 1u);  // (seen by the next level's check)
        continue;
      }
      row.y = A.node[u].y;
      row.z = A.node[v].y;
      next[t] = row;
      const uint32_t s = 2 * row.x;
      if (A.node[row.y].x > s) atomicMin(&A.node[row.y].x, s);
      if (A.node[row.z].x > s + 1) atomicMin(&A.node[row.z].x, s + 1);
    }
    if (!grid_barrier(bar, status, phase)) return;
    dstart += ne - left;
    base += nv;
    nv = comps;
    ne = left;
    levels = lv + 1;
  }
  if (ne > 0) {
    if (first == 0 && tid == 0) atomicOr(status, kErrBadInput);
    return;
  }
  // chains, level by level (totals of lower chains are complete)
  int64_t d0 = 0;
  for (int lv = 0; lv < levels; ++lv) {
    const int64_t d1 = d0 + (int64_t)__ldcg(c_done + lv);
    for (int64_t b = d0 + first; b < d1; b += gthreads) {
      const int64_t t = b + tid;
      uint32_t c = 0, w = 0;
      if (t < d1) {
        const uint4 row = A.done[t];
        const bool tu = (row.y & kTook) != 0u, tv = (row.z & kTook) != 0u;
        const uint32_t u = row.y & ~kTook, v = row.z & ~kTook;
        auto points = [&](uint32_t g) { return g < A.n ? 1u : max(1u, A.total[g - A.n]); };
        w = (tu ? points(u) : 0u) + (tv ? points(v) : 0u);
        c = A.node[u].y;
        uint2 nd = A.node[c];
        while (nd.x != kInvalid && (nd.x >> 1) < row.x) {
          c = nd.y;
          nd = A.node[c];
        }
        c -= (uint32_t)A.n;
        A.keys[row.x] = ((uint64_t)c << 32) | (uint64_t)(2 * row.x + (tu && !tv ? 1u : 0u));
        A.vals[row.x] = w;
      }
      warp_add(A.total, c, w, t < d1);
    }
    d0 = d1;
    if (lv + 1 < levels && !grid_barrier(bar, status, phase)) return;
  }
}

// The sorted edges' running totals along their chains, in tiles: first each
// tile's total since its last chain start (and whether it has one) ...
constexpr int kScanItems = 8;
constexpr int kScanTile = kDgBlock * kScanItems;

struct Segment {  // points since the last chain start; head: there is one
  uint32_t sum;
  bool head;
};
__device__ __forceinline__ Segment join(const Segment &a, const Segment &b) {
  Segment r;
  r.sum = b.head ? b.sum : a.sum + b.sum;
  r.head = a.head || b.head;
  return r;
}

// A thread's kScanItems consecutive elements from q0 on, and their total.
__device__ __forceinline__ Segment load_items(const uint64_t *__restrict__ keys,
                                              const uint32_t *__restrict__ vals, int64_t m, int64_t q0,
                                              uint64_t (&k)[kScanItems + 1], uint32_t (&v)[kScanItems],
                                              uint32_t &heads) {
  Segment s = {0u, false};
  heads = 0;
  uint64_t before = q0 > 0 && q0 < m ? __ldg(keys + q0 - 1) : ~0ull;
#pragma unroll
  for (int j = 0; j <= kScanItems; ++j) k[j] = q0 + j < m ? __ldg(keys + q0 + j) : ~0ull;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    v[j] = q0 + j < m ? __ldg(vals + q0 + j) : 0u;
    const bool head = (k[j] >> 32) != (before >> 32);
    before = k[j];
    heads |= head ? 1u << j : 0u;
    s.sum = head ? v[j] : s.sum + v[j];
    s.head = s.head || head;
  }
  return s;
}

// Inclusive scan of one Segment per thread over the CTA (exclusive result in
// `before`: the elements of the CTA ahead of this thread).
__device__ __forceinline__ Segment scan_segments(Segment s, Segment &before) {
  __shared__ uint32_t s_sum[kDgBlock / 32];
  __shared__ bool s_head[kDgBlock / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Segment x = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    Segment y;
    y.sum = __shfl_up_sync(0xffffffffu, x.sum, o);
    y.head = __shfl_up_sync(0xffffffffu, (int)x.head, o) != 0;
    if (lane >= o) x = join(y, x);
  }
  if (lane == 31) {
    s_sum[warp] = x.sum;
    s_head[warp] = x.head;
  }
  __syncthreads();
  Segment base = {0u, false};
  for (int w = 0; w < warp; ++w) base = join(base, Segment{s_sum[w], s_head[w]});
  Segment up;
  up.sum = __shfl_up_sync(0xffffffffu, x.sum, 1);
  up.head = __shfl_up_sync(0xffffffffu, (int)x.head, 1) != 0;
  before = lane == 0 ? base : join(base, up);
  return join(base, x);
}

__global__ void __launch_bounds__(kDgBlock) k_dg_tiles(const uint64_t *__restrict__ keys,
                                                       const uint32_t *__restrict__ vals, int64_t m,
                                                       uint2 *__restrict__ tiles, const uint32_t *status) {
  wait_for_previous();
  if (*status != 0u) return;
  uint64_t k[kScanItems + 1];
  uint32_t v[kScanItems], heads;
  const int64_t q0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  Segment before;
  const Segment s = scan_segments(load_items(keys, vals, m, q0, k, v, heads), before);
  if (threadIdx.x == kDgBlock - 1) tiles[blockIdx.x] = make_uint2(s.sum, s.head ? 1u : 0u);
}

// ... then every cluster: its size, and the cluster it merges into.
__global__ void __launch_bounds__(kDgBlock) k_dg_finish(const uint64_t *__restrict__ keys,
                                                        const uint32_t *__restrict__ vals, int64_t m,
                                                        int64_t n, const uint2 *__restrict__ tiles,
                                                        const uint2 *__restrict__ node,
                                                        uint32_t *__restrict__ size_out,
                                                        uint32_t *__restrict__ child,
                                                        uint32_t *__restrict__ out_parent,
                                                        const uint32_t *status) {
  wait_for_previous();
  __shared__ uint32_t s_carry;
  if (*status != 0u) return;
  uint64_t k[kScanItems + 1];
  uint32_t v[kScanItems], heads;
  const int64_t q0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  const Segment mine = load_items(keys, vals, m, q0, k, v, heads);
  // what the chain that reaches into this tile gathered in the tiles before:
  // back to the last one with a chain start
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    uint32_t sum = 0;
    for (int64_t t = (int64_t)blockIdx.x - 1; t >= 0; t -= 32) {
      const uint2 x = t - lane >= 0 ? __ldg(tiles + (t - lane)) : make_uint2(0u, 0u);
      const unsigned b = __ballot_sync(0xffffffffu, x.y != 0u);
      const int stop = b ? __ffs(b) - 1 : 31;  // tiles t .. t - stop count
      sum += __reduce_add_sync(0xffffffffu, lane <= stop ? x.x : 0u);
      if (b) break;
    }
    if (lane == 0) s_carry = sum;
  }
  Segment before;
  scan_segments(mine, before);  // (its barrier also publishes s_carry)
  uint32_t run = before.head ? before.sum : s_carry + before.sum;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    if (q0 + j >= m) break;
    run = (heads >> j) & 1u ? v[j] : run + v[j];
    const uint32_t rank = (uint32_t)k[j] >> 1;
    const bool last = q0 + j + 1 >= m || (k[j + 1] >> 32) != (k[j] >> 32);
    // the chain's next edge, on the side it left open, or the edge above the chain
    const uint32_t ps = last ? __ldg(&node[n + (int64_t)(k[j] >> 32)].x) : (uint32_t)k[j + 1];
    if (size_out) size_out[rank] = run;
    if (out_parent) out_parent[n + rank] = ps == kInvalid ? kInvalid : (uint32_t)n + (ps >> 1);
    if (child && ps != kInvalid) child[ps] = (uint32_t)n + rank;
  }
}

// Linkage rows {a, b, w, size}, the two children ordered a < b.
__global__ void k_dg_rows(const emst_edge *__restrict__ e, int64_t m,
                          const uint32_t *__restrict__ size_out, const uint2 *__restrict__ child,
                          uint4 *__restrict__ link, const uint32_t *status) {
  wait_for_previous();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m || *status != 0u) return;
  const uint2 c = child[k];
  link[k] = make_uint4(min(c.x, c.y), max(c.x, c.y), __float_as_uint(e[k].w), size_out[k]);
}

}  // namespace

int dendrogram_impl(const emst_edge *edges, int64_t n, uint4 *out_link, uint32_t *out_parent,
                    cudaStream_t s) {
  if (n < 0 || n > EMST_MAX_POINTS) return EMST_ERR_INVALID_ARG;
  if (n == 0) return EMST_OK;
  const int64_t m = n - 1;
  if (m > 0 && !edges) return EMST_ERR_INVALID_ARG;
  const bool link_dev = !out_link || device_accessible(out_link);
  const bool par_dev = !out_parent || device_accessible(out_parent);
  if (m == 0) {
    if (out_parent) {
      const uint32_t root = kInvalid;
      if (cudaMemcpyAsync(out_parent, &root, 4, cudaMemcpyDefault, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return EMST_ERR_CUDA;
    }
    return EMST_OK;
  }
  const bool edges_dev = device_accessible(edges);
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 255) & ~size_t(255);
    const size_t at = off;
    off += bytes > 0 ? bytes : 1;
    return at;
  };
  const int64_t tiles = (m + kScanTile - 1) / kScanTile;
  // counters, per-level counters and totals first: cleared together
  const size_t o_counters = take(256), o_levels = take(4 * kMaxLevels * sizeof(uint32_t));
  const size_t o_total = take(4 * (size_t)n), clear = off;
  const size_t o_node = take(8 * (size_t)(2 * n)), o_uf = take(4 * (size_t)(2 * n));
  const size_t o_rest0 = take(16 * (size_t)(m / 2 + 1)), o_rest1 = take(16 * (size_t)(m / 2 + 1));
  const size_t o_done = take(16 * (size_t)m);
  const size_t o_k0 = take(8 * (size_t)m), o_k1 = take(8 * (size_t)m);
  const size_t o_v0 = take(4 * (size_t)m), o_v1 = take(4 * (size_t)m);
  const size_t o_sort = take(4 * (size_t)sort_state_words(m));
  const size_t o_child = take(out_link ? 8 * (size_t)m : 0);
  const size_t o_tiles = take(8 * (size_t)tiles);
  const size_t o_edges = edges_dev ? 0 : take(sizeof(emst_edge) * (size_t)m);
  const size_t o_link = (out_link && !link_dev) ? take(16 * (size_t)m) : 0;
  const size_t o_pout = (out_parent && !par_dev) ? take(4 * (size_t)(n + m)) : 0;
  char *base = nullptr;
  if (scratch_alloc((void **)&base, off, s) != cudaSuccess) return EMST_ERR_OOM;
  int rc = EMST_OK;
  uint32_t host_status = 0;
  auto U = [&](size_t o) { return reinterpret_cast<uint32_t *>(base + o); };
  const emst_edge *e = edges_dev ? edges : reinterpret_cast<emst_edge *>(base + o_edges);
  uint4 *link = out_link ? (link_dev ? out_link : reinterpret_cast<uint4 *>(base + o_link)) : nullptr;
  uint32_t *pout = out_parent ? (par_dev ? out_parent : U(o_pout)) : nullptr;
  Contract A;
  A.e = e;
  A.n = n;
  A.m = m;
  A.counters = U(o_counters);
  A.per_level = U(o_levels);
  A.total = U(o_total);
  A.node = reinterpret_cast<uint2 *>(base + o_node);
  A.uf = U(o_uf);
  A.rest[0] = reinterpret_cast<uint4 *>(base + o_rest0);
  A.rest[1] = reinterpret_cast<uint4 *>(base + o_rest1);
  A.done = reinterpret_cast<uint4 *>(base + o_done);
  A.keys = reinterpret_cast<uint64_t *>(base + o_k0);
  A.vals = U(o_v0);
  A.out_parent = pout;
  A.child = link ? U(o_child) : nullptr;
  uint32_t *status = A.counters + 1;
  // a cooperative grid: what is resident at once, or less for few edges
  static int ctas_per_sm[64] = {0};  // by device, looked up once (every thread finds the same)
  int dev = 0;
  cudaGetDevice(&dev);
  int occ = dev >= 0 && dev < 64 ? ctas_per_sm[dev] : 0;
  bool ok = true;
  if (occ == 0) {
    ok = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dg_contract, kContractThreads, 0) == cudaSuccess &&
         occ >= 1;
    if (ok && dev >= 0 && dev < 64) ctas_per_sm[dev] = occ;
  }
  if (ok) {
    cudaMemsetAsync(base, 0, clear, s);
    cudaMemsetAsync(A.node, 0xff, 8 * (size_t)(2 * n), s);
    if (!edges_dev)
      cudaMemcpyAsync((void *)e, edges, sizeof(emst_edge) * (size_t)m, cudaMemcpyHostToDevice, s);
    k_dg_check<<<grid_for(n, kDgBlock), kDgBlock, 0, s>>>(e, m, n, A.node, A.uf, A.counters);
    int64_t g = (int64_t)sm_count() * occ;
    if (g > (n + kContractThreads - 1) / kContractThreads) g = (n + kContractThreads - 1) / kContractThreads;
    void *args[] = {&A};
    ok = cudaLaunchCooperativeKernel(k_dg_contract, dim3((unsigned)g), dim3(kContractThreads), args, 0, s) ==
         cudaSuccess;
  }
  if (ok) {
    Problem P;  // the sort's buffers
    P.stream = s;
    P.counters = A.counters;
    P.keys[0] = A.keys;
    P.keys[1] = reinterpret_cast<uint64_t *>(base + o_k1);
    P.vals[0] = A.vals;
    P.vals[1] = U(o_v1);
    P.sort_state = U(o_sort);
    // by chain; the edges of one chain stay in rank order (a stable sort)
    const int src = radix_sort_pairs(P, m, 0, (bits_for(n - 1) + 7) / 8, 0, 32);
    uint2 *tile = reinterpret_cast<uint2 *>(base + o_tiles);
    uint32_t *size = link ? P.vals[src ^ 1] : nullptr;  // the sort's other buffer is free again
    launch_next(P, k_dg_tiles, (unsigned)tiles, kDgBlock, 0, P.keys[src], P.vals[src], m, tile, status);
    launch_next(P, k_dg_finish, (unsigned)tiles, kDgBlock, 0, P.keys[src], P.vals[src], m, n, tile, A.node, size,
                                                     A.child, pout, status);
    if (link)
      launch_next(P, k_dg_rows, grid_for(m, kDgBlock), kDgBlock, 0, e, m, size, reinterpret_cast<const uint2 *>(A.child), link, status);
    ok = cudaPeekAtLastError() == cudaSuccess;
    if (out_link && !link_dev)
      cudaMemcpyAsync(out_link, link, 16 * (size_t)m, cudaMemcpyDeviceToHost, s);
    if (out_parent && !par_dev)
      cudaMemcpyAsync(out_parent, pout, 4 * (size_t)(n + m), cudaMemcpyDeviceToHost, s);
    ok = ok && cudaMemcpyAsync(&host_status, status, 4, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
  }
  if (!ok) rc = EMST_ERR_CUDA;
  else rc = status_from_bits(host_status);
  cudaFreeAsync(base, s);
  if (cudaGetLastError() != cudaSuccess && rc == EMST_OK) rc = EMST_ERR_CUDA;
  return rc;
}

}  // namespace emst

extern "C" int emst_dendrogram(const emst_edge *edges, int64_t n, emst_linkage *out_linkage,
                               uint32_t *out_parent, void *stream) {
  static_assert(sizeof(emst_linkage) == 16, "linkage row is 16 bytes");
  return emst::dendrogram_impl(edges, n, reinterpret_cast<uint4 *>(out_linkage), out_parent,
                               (cudaStream_t)stream);
}
