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
// chains, the idea of P. Sao, A. Prokopenko and D. Lebrun-Grandie, "PANDORA: A
// Parallel Dendrogram Construction Algorithm for Single Linkage Clustering on
// GPU" (2024):
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
  uint32_t *counters;  // [1] status, [2] invalid input found before the contraction, [40] barrier,
                       // [41] tiles finished
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
// tile's total since its last chain start (and whether it has one),
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

// and with many tiles, by the last CTA to finish, what the chain that reaches
// into each tile gathered in the tiles before it (in place of the tile's
// total).  Fewer tiles look for it on their own, back to the last chain start,
// which a chain of the usual length ends at once; the scan takes 6 to 10 us of
// the launch's tail (random trees of 5,000 edges 190 -> 196 us a call, of 8M
// 2,273 -> 2,283).  Of all tiles the walks would be quadratic when one chain
// holds most edges (paths of rising weights, walks / scan: 8M edges 1,875 /
// 1,828 us, 100M 30.6 / 16.2 ms), so the line lies where the scan's share is
// below half a percent and the walks' worst below three.
constexpr int64_t kWalkTiles = 4096;  // 8.4M edges
__global__ void __launch_bounds__(kDgBlock) k_dg_tiles(const uint64_t *__restrict__ keys,
                                                       const uint32_t *__restrict__ vals, int64_t m,
                                                       uint2 *tiles, uint32_t *finished,
                                                       const uint32_t *status) {
  wait_for_previous();
  if (*status != 0u) return;
  __shared__ bool s_last;
  uint64_t k[kScanItems + 1];
  uint32_t v[kScanItems], heads;
  const int64_t q0 = (int64_t)blockIdx.x * kScanTile + threadIdx.x * kScanItems;
  Segment before;
  const Segment s = scan_segments(load_items(keys, vals, m, q0, k, v, heads), before);
  if (threadIdx.x == kDgBlock - 1) tiles[blockIdx.x] = make_uint2(s.sum, s.head ? 1u : 0u);
  if (gridDim.x <= kWalkTiles) return;
  if (threadIdx.x == kDgBlock - 1) {
    __threadfence();
    s_last = atomicAdd(finished, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // a run of tiles per thread, read eight at a time (this is the launch's tail)
  constexpr int kAtOnce = 8;
  const int64_t count = gridDim.x;
  const int64_t chunk = ((count + kDgBlock - 1) / kDgBlock + kAtOnce - 1) / kAtOnce * kAtOnce;
  const int64_t lo = (int64_t)threadIdx.x * chunk, hi = lo + chunk < count ? lo + chunk : count;
  auto load = [&](int64_t t, Segment (&x)[kAtOnce]) {
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      const uint2 w = t + u < hi ? __ldcg(tiles + t + u) : make_uint2(0u, 0u);
      x[u] = Segment{w.x, w.y != 0u};
    }
  };
  Segment x[kAtOnce], mine = {0u, false};
  for (int64_t t = lo; t < hi; t += kAtOnce) {
    load(t, x);
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) mine = join(mine, x[u]);
  }
  scan_segments(mine, before);
  for (int64_t t = lo; t < hi; t += kAtOnce) {
    load(t, x);
#pragma unroll
    for (int u = 0; u < kAtOnce; ++u) {
      if (t + u < hi) tiles[t + u].x = before.sum;
      before = join(before, x[u]);
    }
  }
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
  // there already, or in those back to the last one with a chain start
  if (gridDim.x > kWalkTiles) {
    if (threadIdx.x == 0) s_carry = __ldg(&tiles[blockIdx.x].x);
  } else if (threadIdx.x < 32) {
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

// ---------------------------------------------------------------------------
// A tree of at most kOneCtaEdges edges: the same contraction, chains, order and
// totals by one CTA, everything but the edges and the result in shared memory,
// in one launch.  What bounds a small tree is latency: over global memory,
// with a grid barrier per step and a launch per sort pass, the contraction is
// slower here than halving the ranks in shared memory was.  Random trees of
// 300 / 1,000 / 2,000 / 4,096 edges, us a call: halving 114 / 129 / 153 / 182,
// contraction in global memory 112 / 150 / 163 / 180, this 70 / 77 / 89 / 112
// (paths 107 / 120 / 143 / 172, 122 / 168 / 183 / 193, 73 / 76 / 87 / 111).
// It serves every size that fits: at the largest it still takes two thirds of
// the other.
// ---------------------------------------------------------------------------
constexpr int kOneCtaEdges = 4096;  // the largest whose arrays fit (197 KB)
constexpr int kOneCtaThreads = 1024;
constexpr int kOneCtaLevels = 16;   // vertices halve: 13 reach 4,097
constexpr uint32_t kSlotBits = 13;  // slots below 2 * kOneCtaEdges, chains below kOneCtaEdges + 1
constexpr uint32_t kTook16 = 0x8000u;
static_assert(2 * kOneCtaEdges <= 1 << kSlotBits && 2 * (kOneCtaEdges + 1) < (int)kTook16, "ids in 16 bits");

// Where the one-CTA form's arrays lie in shared memory (byte offsets).
struct OneCtaLayout {
  int low, uf, total, done, rest[2], keys, vals, comp, bytes;
  int padded;  // keys are sorted as a power of two
  __host__ __device__ explicit OneCtaLayout(int n) {
    const int m = n - 1;
    padded = 32;
    while (padded < m) padded <<= 1;
    int off = 0;
    auto take = [&](int b) {
      const int at = off;
      off = (off + b + 7) & ~7;
      return at;
    };
    done = take(8 * m);
    rest[0] = take(8 * (m / 2 + 1));  // (with rest[1]: the 2m child entries, 8m bytes, later on)
    rest[1] = take(8 * (m / 2 + 1));
    low = take(4 * 2 * n);
    uf = take(4 * 2 * n);  // (the running totals later on)
    total = take(4 * n);   // (the totals before each chain later on)
    keys = take(4 * padded);
    vals = take(4 * m);
    comp = take(2 * 2 * n);
    bytes = off;
  }
};

// Ascending sort of s[0 .. size), a power of two of at least 32, by the CTA;
// the steps over distances below 32 stay in a warp's registers.
__device__ __forceinline__ void sort_words(uint32_t *s, int size) {
  const int lane = threadIdx.x & 31;
  auto rows = [&](int k0, int k1) {
    __syncthreads();
    for (int e = threadIdx.x; e < size; e += blockDim.x) {
      uint32_t x = s[e];
      for (int k = k0; k <= k1; k <<= 1)
        for (int j = k / 2 < 16 ? k / 2 : 16; j > 0; j >>= 1) {
          const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
          x = ((e & k) == 0) == ((lane & j) == 0) ? min(x, y) : max(x, y);
        }
      s[e] = x;
    }
  };
  rows(2, 32);
  for (int k = 64; k <= size; k <<= 1) {
    for (int j = k >> 1; j >= 32; j >>= 1) {
      __syncthreads();
      for (int t = threadIdx.x; t < size / 2; t += blockDim.x) {
        const int a = ((t & ~(j - 1)) << 1) | (t & (j - 1)), b = a | j;
        const uint32_t x = s[a], y = s[b];
        if ((y < x) == ((a & k) == 0)) {
          s[a] = y;
          s[b] = x;
        }
      }
    }
    rows(k, k);
  }
  __syncthreads();
}

// blockDim: whole warps, at most kOneCtaThreads.  *status: the call's result,
// written in any case.
__global__ void __launch_bounds__(kOneCtaThreads, 1) k_dg_one_cta(const emst_edge *__restrict__ e, int n,
                                                               uint4 *__restrict__ link,
                                                               uint32_t *__restrict__ out_parent,
                                                               uint32_t *status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t c_done[kOneCtaLevels], c_rest[kOneCtaLevels], c_comp[kOneCtaLevels];
  __shared__ uint32_t s_warp[kOneCtaThreads / 32];
  const OneCtaLayout L(n);
  // a row: x = rank, y = the vertices of its sides, 16 bits each, flagged kTook16
  uint2 *done = reinterpret_cast<uint2 *>(smem_raw + L.done);
  uint2 *rest[2] = {reinterpret_cast<uint2 *>(smem_raw + L.rest[0]), reinterpret_cast<uint2 *>(smem_raw + L.rest[1])};
  uint32_t *low = reinterpret_cast<uint32_t *>(smem_raw + L.low);  // a vertex's lowest slot
  uint32_t *uf = reinterpret_cast<uint32_t *>(smem_raw + L.uf);
  uint32_t *total = reinterpret_cast<uint32_t *>(smem_raw + L.total);
  uint32_t *keys = reinterpret_cast<uint32_t *>(smem_raw + L.keys);
  uint32_t *vals = reinterpret_cast<uint32_t *>(smem_raw + L.vals);
  uint16_t *comp = reinterpret_cast<uint16_t *>(smem_raw + L.comp);  // the component that holds a vertex
  const int tid = threadIdx.x, lane = tid & 31, threads = blockDim.x;
  const int m = n - 1;
  const uint32_t lt = (1u << lane) - 1u;
  auto place = [&](bool want, uint32_t *counter) {  // (whole warps call)
    const unsigned b = __ballot_sync(0xffffffffu, want);
    uint32_t at = 0;
    if (lane == 0 && b) at = atomicAdd(counter, (uint32_t)__popc(b));
    return __shfl_sync(0xffffffffu, at, 0) + __popc(b & lt);
  };
  for (int v = tid; v < 2 * n; v += threads) {
    low[v] = kInvalid;
    uf[v] = (uint32_t)v;
  }
  for (int v = tid; v < n; v += threads) total[v] = 0u;
  if (tid < kOneCtaLevels) c_done[tid] = c_rest[tid] = c_comp[tid] = 0u;
  __syncthreads();
  uint32_t err = 0;
  for (int k = tid; k < m; k += threads) {  // (k_dg_check)
    const emst_edge x = e[k];
    if (x.i >= (uint32_t)n || x.j >= (uint32_t)n || x.i == x.j || !(x.w == x.w) || (k + 1 < m && e[k + 1].w < x.w)) {
      err = kErrBadInput;
    } else {
      atomicMin(low + x.i, 2u * (uint32_t)k);
      atomicMin(low + x.j, 2u * (uint32_t)k + 1u);
    }
  }
  int base = 0, nv = n, ne = m, dstart = 0, levels = 0;
  while (!__syncthreads_or(err) && ne > 0 && levels < kOneCtaLevels) {
    const int lv = levels++;
    uint2 *from = rest[lv & 1], *next = rest[(lv + 1) & 1];
    for (int b = 0; b < ne; b += threads) {
      const int t = b + tid;
      bool take = false, keep = false;
      uint32_t rank = 0, u = 0, v = 0;
      if (t < ne) {
        if (lv == 0) {
          rank = (uint32_t)t;
          u = e[t].i;
          v = e[t].j;
        } else {
          const uint2 row = from[t];
          rank = row.x;
          u = row.y & 0xffffu;
          v = row.y >> 16;
        }
        const bool tu = low[u] >> 1 == rank, tv = low[v] >> 1 == rank;
        take = tu || tv;
        keep = !take;
        if (take && !uf_unite(uf, u, v)) err = kErrSpin;
        u |= tu ? kTook16 : 0u;
        v |= tv ? kTook16 : 0u;
      }
      const uint32_t d = place(take, c_done + lv);
      if (take) done[dstart + d] = make_uint2(rank, u | v << 16);
      const uint32_t r = place(keep, c_rest + lv);
      if (keep) {
        if (r <= (uint32_t)m / 2) next[r] = make_uint2(rank, u | v << 16);
        else err = kErrBadInput;  // more edges than half the vertices: not a tree
      }
    }
    __syncthreads();
    for (int b = 0; b < nv; b += threads) {
      const int v = base + b + tid;
      const bool in = b + tid < nv, root = in && uf[v] == (uint32_t)v;
      const int g = base + nv + (int)place(root, c_comp + lv);
      if (in && low[v] == kInvalid) err = kErrBadInput;  // a vertex without an edge: not a tree
      if (root) {
        if (g < 2 * n) comp[v] = (uint16_t)g;
        else err = kErrBadInput;
      }
    }
    if (__syncthreads_or(err)) break;
    const int left = (int)c_rest[lv];
    for (int t = tid; t < nv; t += threads) {
      const uint32_t v = (uint32_t)(base + t), r = uf_find<true>(uf, v);
      if (r != v) comp[v] = comp[r];
    }
    for (int t = tid; t < left; t += threads) {
      const uint2 row = next[t];
      uint32_t u = row.y & 0xffffu, v = row.y >> 16;
      uf_find2<true>(uf, u, v);
      if (u == v) {  // an edge inside a component: it closes a cycle
        err = kErrBadInput;
        continue;
      }
      u = comp[u];
      v = comp[v];
      next[t] = make_uint2(row.x, u | v << 16);
      atomicMin(low + u, 2u * row.x);
      atomicMin(low + v, 2u * row.x + 1u);
    }
    dstart += ne - left;
    base += nv;
    nv = (int)c_comp[lv];
    ne = left;
  }
  if (ne > 0) err |= kErrBadInput;
  if (__syncthreads_or(err)) {
    // (every error is of the input but a spin that ran out)
    const int spin = __syncthreads_or(err & kErrSpin);
    if (tid == 0) *status = spin ? kErrSpin : kErrBadInput;
    return;
  }
  // chains, level by level (totals of lower chains are complete)
  int d0 = 0;
  for (int lv = 0; lv < levels; ++lv) {
    const int d1 = d0 + (int)c_done[lv];
    for (int b = d0; b < d1; b += threads) {
      const int t = b + tid;
      uint32_t c = 0, w = 0;
      if (t < d1) {
        const uint2 row = done[t];
        const bool tu = (row.y & kTook16) != 0u, tv = (row.y >> 16 & kTook16) != 0u;
        const uint32_t u = row.y & (kTook16 - 1u), v = row.y >> 16 & (kTook16 - 1u);
        auto points = [&](uint32_t g) { return g < (uint32_t)n ? 1u : total[g - n]; };
        w = (tu ? points(u) : 0u) + (tv ? points(v) : 0u);
        c = comp[u];
        while (low[c] != kInvalid && low[c] >> 1 < row.x) c = comp[c];
        c -= (uint32_t)n;
        keys[row.x] = c << kSlotBits | (2u * row.x + (tu && !tv ? 1u : 0u));
        vals[row.x] = w;
      }
      warp_add(total, c, w, t < d1);
    }
    d0 = d1;
    __syncthreads();
  }
  for (int q = m + tid; q < L.padded; q += threads) keys[q] = ~0u;
  sort_words(keys, L.padded);
  // running totals over all chains, and what lies before each chain
  uint32_t *run = uf, *before = total, *child = reinterpret_cast<uint32_t *>(smem_raw + L.rest[0]);
  const uint32_t slot_mask = (1u << kSlotBits) - 1u;
  {
    const int per = (m + threads - 1) / threads, q0 = tid * per, q1 = min(q0 + per, m);
    uint32_t sum = 0;
    for (int q = q0; q < q1; ++q) sum += vals[(keys[q] & slot_mask) >> 1];
    uint32_t x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[tid >> 5] = x;
    __syncthreads();
    uint32_t at = x - sum;
    for (int w = 0; w < tid >> 5; ++w) at += s_warp[w];
    for (int q = q0; q < q1; ++q) {
      const uint32_t key = keys[q];
      if (q == 0 || keys[q - 1] >> kSlotBits != key >> kSlotBits) before[key >> kSlotBits] = at;
      at += vals[(key & slot_mask) >> 1];
      run[(key & slot_mask) >> 1] = at;
    }
  }
  __syncthreads();
  // every cluster: its size, and the cluster it merges into (k_dg_finish)
  for (int q = tid; q < m; q += threads) {
    const uint32_t key = keys[q], chain = key >> kSlotBits, rank = (key & slot_mask) >> 1;
    const bool last = q + 1 >= m || keys[q + 1] >> kSlotBits != chain;
    const uint32_t ps = last ? low[n + chain] : keys[q + 1] & slot_mask;
    run[rank] -= before[chain];
    if (out_parent) out_parent[n + rank] = ps == kInvalid ? kInvalid : (uint32_t)n + (ps >> 1);
    if (ps != kInvalid) child[ps] = (uint32_t)n + rank;
  }
  for (int v = tid; v < n; v += threads) {
    if (out_parent) out_parent[v] = (uint32_t)n + (low[v] >> 1);
    child[low[v]] = (uint32_t)v;
  }
  __syncthreads();
  if (link)
    for (int k = tid; k < m; k += threads) {
      const uint32_t a = child[2 * k], b = child[2 * k + 1];
      link[k] = make_uint4(min(a, b), max(a, b), __float_as_uint(e[k].w), run[k]);
    }
  if (tid == 0) *status = 0u;
}

cudaError_t launch_one_cta(const emst_edge *e, int n, uint4 *link, uint32_t *out_parent, uint32_t *status,
                           cudaStream_t s) {
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !attr_set[dev]) {
    const cudaError_t rc = cudaFuncSetAttribute(k_dg_one_cta, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                OneCtaLayout(kOneCtaEdges + 1).bytes);
    if (rc != cudaSuccess) return rc;
    if (dev < 64) attr_set[dev] = true;
  }
  const int threads = n - 1 < kOneCtaThreads ? (n - 1 + 31) & ~31 : kOneCtaThreads;  // one per edge
  k_dg_one_cta<<<1, threads, OneCtaLayout(n).bytes, s>>>(e, n, link, out_parent, status);
  return cudaPeekAtLastError();
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
  const bool one_cta = m <= kOneCtaEdges;  // its arrays are in shared memory
  const int64_t tiles = (m + kScanTile - 1) / kScanTile;
  // counters, per-level counters and totals first: cleared together
  const size_t o_counters = take(256), o_levels = take(4 * kMaxLevels * sizeof(uint32_t));
  auto take_big = [&](size_t bytes) { return take(one_cta ? 0 : bytes); };
  const size_t o_total = take_big(4 * (size_t)n), clear = off;
  const size_t o_node = take_big(8 * (size_t)(2 * n)), o_uf = take_big(4 * (size_t)(2 * n));
  const size_t o_rest0 = take_big(16 * (size_t)(m / 2 + 1)), o_rest1 = take_big(16 * (size_t)(m / 2 + 1));
  const size_t o_done = take_big(16 * (size_t)m);
  const size_t o_k0 = take_big(8 * (size_t)m), o_k1 = take_big(8 * (size_t)m);
  const size_t o_v0 = take_big(4 * (size_t)m), o_v1 = take_big(4 * (size_t)m);
  const size_t o_sort = take_big(4 * (size_t)sort_state_words(m));
  const size_t o_child = take_big(out_link ? 8 * (size_t)m : 0);
  const size_t o_tiles = take_big(8 * (size_t)tiles);
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
  bool ok = true;
  if (!edges_dev)
    ok = cudaMemcpyAsync((void *)e, edges, sizeof(emst_edge) * (size_t)m, cudaMemcpyHostToDevice, s) == cudaSuccess;
  // a cooperative grid: what is resident at once, or less for few edges
  static int ctas_per_sm[64] = {0};  // by device, looked up once (every thread finds the same)
  int dev = 0;
  cudaGetDevice(&dev);
  int occ = dev >= 0 && dev < 64 ? ctas_per_sm[dev] : 0;
  if (one_cta) ok = ok && launch_one_cta(e, (int)n, link, pout, status, s) == cudaSuccess;
  if (occ == 0 && !one_cta) {
    ok = ok && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_dg_contract, kContractThreads, 0) == cudaSuccess &&
         occ >= 1;
    if (ok && dev >= 0 && dev < 64) ctas_per_sm[dev] = occ;
  }
  if (ok && !one_cta) {
    cudaMemsetAsync(base, 0, clear, s);
    cudaMemsetAsync(A.node, 0xff, 8 * (size_t)(2 * n), s);
    k_dg_check<<<grid_for(n, kDgBlock), kDgBlock, 0, s>>>(e, m, n, A.node, A.uf, A.counters);
    int64_t g = (int64_t)stream_sm_count(s) * occ;
    if (g > (n + kContractThreads - 1) / kContractThreads) g = (n + kContractThreads - 1) / kContractThreads;
    void *args[] = {&A};
    auto launch = [&](unsigned ctas) {
      return cudaLaunchCooperativeKernel(k_dg_contract, dim3(ctas), dim3(kContractThreads), args, 0, s);
    };
    ok = launch_cooperative(g, launch) == cudaSuccess;
  }
  if (ok && !one_cta) {
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
    launch_next(P, k_dg_tiles, (unsigned)tiles, kDgBlock, 0, P.keys[src], P.vals[src], m, tile,
                A.counters + 41, status);
    launch_next(P, k_dg_finish, (unsigned)tiles, kDgBlock, 0, P.keys[src], P.vals[src], m, n, tile, A.node, size,
                                                     A.child, pout, status);
    if (link)
      launch_next(P, k_dg_rows, grid_for(m, kDgBlock), kDgBlock, 0, e, m, size, reinterpret_cast<const uint2 *>(A.child), link, status);
    ok = cudaPeekAtLastError() == cudaSuccess;
  }
  if (ok) {
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
