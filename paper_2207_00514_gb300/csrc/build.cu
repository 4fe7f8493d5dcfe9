// build.cu -- the tree build of the method (§2 "ArborX": Z-curve
// linearisation, sort, fully parallel bottom-up hierarchy construction):
//   A1 scene box, A2 Morton codes, A3 (sort.cu), A4 gather + hierarchy + refit.
#include "common.cuh"

namespace emst {

constexpr int kBlock = 256;

// ---------------------------------------------------------------------------
// A1. Scene box: per-dimension min / max of all coordinates, plus a flag for
// any non-finite coordinate.  box[0..2] = ordered min, box[3..5] = ordered max.
// ---------------------------------------------------------------------------
// A CTA's box into the scene box: one atomic per bound (one per warp, all on
// the same few words, made up most of the pass: 200,000 points 20 -> 3.5 us).
template <int DIM>
__device__ __forceinline__ void box_result(const float (&lo)[3], const float (&hi)[3], bool bad,
                                           uint32_t *box, uint32_t *status) {
  __shared__ uint32_t s_part[kBlock / 32][6];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < DIM; ++q) {  // (an empty range, +inf > -inf, is the neutral one)
    const uint32_t l = __reduce_min_sync(0xffffffffu, float_to_ordered(lo[q]));
    const uint32_t h = __reduce_max_sync(0xffffffffu, float_to_ordered(hi[q]));
    if (lane == 0) {
      s_part[warp][q] = l;
      s_part[warp][3 + q] = h;
    }
  }
  const bool any_bad = __syncthreads_or(bad);
  if (threadIdx.x < 2 * DIM) {
    const int q = threadIdx.x % DIM;
    const bool upper = threadIdx.x >= DIM;
    uint32_t v = s_part[0][upper ? 3 + q : q];
    for (int w = 1; w < kBlock / 32; ++w) {
      const uint32_t x = s_part[w][upper ? 3 + q : q];
      v = upper ? max(v, x) : min(v, x);
    }
    // (a CTA without a finite coordinate on this axis leaves the box alone)
    if (upper) {
      if (v != float_to_ordered(-INFINITY)) atomicMax(&box[3 + q], v);
    } else if (v != float_to_ordered(INFINITY)) {
      atomicMin(&box[q], v);
    }
  }
  if (any_bad && threadIdx.x == 0) atomicOr(status, kErrNonFinite);
}

// COPY: the points are read from pinned host memory through its device
// mapping and written to `copy` (device) on the way, so the host-to-device
// transfer of a host input is this pass itself.
template <int DIM, bool COPY>
__global__ void __launch_bounds__(kBlock) k_scene_box(const float *__restrict__ pts, int64_t n,
                                                      uint32_t *__restrict__ box,
                                                      uint32_t *__restrict__ status,
                                                      float *__restrict__ copy) {
  wait_for_previous();
  float lo[3] = {INFINITY, INFINITY, INFINITY};
  float hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  bool bad = false;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  auto take = [&](int64_t k) {
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      const float x = COPY ? pts[k * DIM + q] : __ldg(pts + k * DIM + q);
      if (COPY) copy[k * DIM + q] = x;
      if (!isfinite(x)) { bad = true; continue; }
      lo[q] = fminf(lo[q], x);
      hi[q] = fmaxf(hi[q], x);
    }
  };
  // whole points per thread, four independent ones per step (loads in flight)
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; k + 3 * stride < n; k += 4 * stride) {
    take(k);
    take(k + stride);
    take(k + 2 * stride);
    take(k + 3 * stride);
  }
  for (; k < n; k += stride) take(k);
  box_result<DIM>(lo, hi, bad, box, status);
}

// The COPY form reading 16 bytes per load (the host input through its
// mapping): the flat coordinate array as float4s, element e of dimension
// e % DIM; `tail` (< 4) trailing elements read one by one by thread 0.
// src and copy 16-byte aligned.
template <int DIM>
__global__ void __launch_bounds__(kBlock) k_scene_box_copy4(const float4 *__restrict__ src,
                                                            int64_t nv, int tail,
                                                            uint32_t *__restrict__ box,
                                                            uint32_t *__restrict__ status,
                                                            float4 *__restrict__ copy) {
  wait_for_previous();
  float lo[3] = {INFINITY, INFINITY, INFINITY};
  float hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  bool bad = false;
  auto take = [&](float x, int d) {
    if (!isfinite(x)) { bad = true; return; }
#pragma unroll
    for (int q = 0; q < DIM; ++q) {
      if (q == d) {
        lo[q] = fminf(lo[q], x);
        hi[q] = fmaxf(hi[q], x);
      }
    }
  };
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  auto use = [&](const float4 &a, int64_t v) {
    copy[v] = a;
    const int d0 = (int)((4 * v) % DIM);
    take(a.x, d0);
    take(a.y, (d0 + 1) % DIM);
    take(a.z, (d0 + 2) % DIM);
    take(a.w, (d0 + 3) % DIM);
  };
  // four independent loads in flight per thread (the link's latency is long)
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; v + 3 * stride < nv; v += 4 * stride) {
    const float4 a0 = src[v], a1 = src[v + stride], a2 = src[v + 2 * stride], a3 = src[v + 3 * stride];
    use(a0, v);
    use(a1, v + stride);
    use(a2, v + 2 * stride);
    use(a3, v + 3 * stride);
  }
  for (; v < nv; v += stride) use(src[v], v);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const float *s1 = reinterpret_cast<const float *>(src + nv);
    float *c1 = reinterpret_cast<float *>(copy + nv);
    for (int t = 0; t < tail; ++t) {
      c1[t] = s1[t];
      take(s1[t], (int)((4 * nv + t) % DIM));
    }
  }
  box_result<DIM>(lo, hi, bad, box, status);
}

// All counters to zero, the scene box (4..9) empty: the call's first kernel.
__global__ void k_counters_init(uint32_t *counters) {
  const int t = threadIdx.x;
  counters[t] = t >= 4 && t < 7 ? 0xFFFFFFFFu : 0u;
}

void launch_scene_box(Problem &P) {
  uint32_t *box = P.counters + 4;
  k_counters_init<<<1, 64, 0, P.stream>>>(P.counters);
  int grid = sm_count() * 4;
  int64_t need = (P.n + kBlock - 1) / kBlock;
  if (need < grid) grid = (int)(need < 1 ? 1 : need);
  float *copy = const_cast<float *>(P.points);
  if (P.points_mapped && (reinterpret_cast<uintptr_t>(P.points_mapped) & 15u) == 0 &&
      (reinterpret_cast<uintptr_t>(copy) & 15u) == 0) {
    // read the host input through its mapping 16 bytes at a time, keep a device copy
    const int64_t elems = P.n * P.dim, nv = elems / 4;
    const int tail = (int)(elems - 4 * nv);
    int g4 = sm_count() * 4;
    if ((nv + kBlock - 1) / kBlock < g4) g4 = (int)((nv + kBlock - 1) / kBlock < 1 ? 1 : (nv + kBlock - 1) / kBlock);
    const float4 *src = reinterpret_cast<const float4 *>(P.points_mapped);
    float4 *dst = reinterpret_cast<float4 *>(copy);
    if (P.dim == 3)
      launch_next(P, k_scene_box_copy4<3>, g4, kBlock, 0, src, nv, tail, box, P.counters + 1, dst);
    else
      launch_next(P, k_scene_box_copy4<2>, g4, kBlock, 0, src, nv, tail, box, P.counters + 1, dst);
  } else if (P.points_mapped) {  // read the host input through its mapping, keep a device copy
    if (P.dim == 3)
      launch_next(P, k_scene_box<3, true>, grid, kBlock, 0, P.points_mapped, P.n, box, P.counters + 1, copy);
    else
      launch_next(P, k_scene_box<2, true>, grid, kBlock, 0, P.points_mapped, P.n, box, P.counters + 1, copy);
  } else if (P.dim == 3) {
    launch_next(P, k_scene_box<3, false>, grid, kBlock, 0, P.points, P.n, box, P.counters + 1, nullptr);
  } else {
    launch_next(P, k_scene_box<2, false>, grid, kBlock, 0, P.points, P.n, box, P.counters + 1, nullptr);
  }
  P.launches += 2;
}

// ---------------------------------------------------------------------------
// A2. Morton codes.  Quantisation decided in FP32 exactly as specified (B = 21
// bits per dimension in 3D, 32 in 2D; fewer in the batched form, see
// code_bits):
//   s = 2^B / (hi - lo) (0 for a flat dimension), t = (x - lo) * s,
//   q = t >= 2^B ? 2^B - 1 : trunc(t)
// and the bits interleave x (most significant), y, z.
// ---------------------------------------------------------------------------
// With instances, the instance id goes above the interleaved bits.
template <int DIM>
__global__ void __launch_bounds__(kBlock) k_morton(const float *__restrict__ pts, int64_t n,
                                                   const uint32_t *__restrict__ box,
                                                   const uint32_t *__restrict__ inst_in, int bits,
                                                   uint64_t *__restrict__ keys,
                                                   uint32_t *__restrict__ vals, ClearWords clear) {
  wait_for_previous();
  clear_words(clear);
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const Quantizer Q = make_quantizer(box, DIM, bits);
  uint32_t q[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < DIM; ++d) q[d] = quantize(Q, d, __ldg(pts + k * DIM + d));
  uint64_t code = interleave(q[0], q[1], q[2], DIM);
  if (inst_in) code |= (uint64_t)__ldg(inst_in + k) << (DIM * bits);
  keys[k] = code;
  vals[k] = (uint32_t)k;
}

void launch_morton(Problem &P) {
  const ClearWords clear = {P.sort_state, sort_clear_words(P.n)};
  int g = grid_for(P.n, kBlock);
  const int bits = code_bits(P.dim, P.inst_bits);
  if (P.dim == 3)
    launch_next(P, k_morton<3>, g, kBlock, 0, P.points, P.n, P.counters + 4, P.inst_in, bits,
                                            P.keys[0], P.vals[0], clear);
  else
    launch_next(P, k_morton<2>, g, kBlock, 0, P.points, P.n, P.counters + 4, P.inst_in, bits,
                                            P.keys[0], P.vals[0], clear);
  P.launches += 1;
}

// A2 at the finer grid §4.1 suggests for very dense data (128-bit codes):
// B = 42 bits per dimension in 3D, 64 in 2D, quantised in FP64 so the grid
// resolves FP32 coordinates:
//   s = 2^B / (hi - lo) (0 for a flat dimension), t = (x - lo) * s,
//   q = t >= 2^B ? 2^B - 1 : trunc(t)
// every step rounded explicitly.  The code is the 64-bit interleave of each
// half of the cells: in 3D, with H and L the 63-bit interleaves of the high
// and low 21 bits, code = H << 63 | L; in 2D the halves are the two words.
template <int DIM>
__global__ void __launch_bounds__(kBlock) k_morton128(const float *__restrict__ pts, int64_t n,
                                                      const uint32_t *__restrict__ box,
                                                      uint64_t *__restrict__ code_hi,
                                                      uint64_t *__restrict__ code_lo,
                                                      uint64_t *__restrict__ keys,
                                                      uint32_t *__restrict__ vals, ClearWords clear) {
  wait_for_previous();
  clear_words(clear);
  // the FP64 divisions once per CTA (this GPU has few FP64 units: a division
  // per point and axis took 190 us for 2M points, this 65)
  __shared__ double s_lo[3], s_scale[3];
  constexpr int B = DIM == 3 ? 42 : 64;
  const double twoB = DIM == 3 ? 4398046511104.0 : 18446744073709551616.0;  // 2^B
  const uint64_t qmax = DIM == 3 ? ((1ull << 42) - 1ull) : ~0ull;
  if (threadIdx.x < DIM) {
    const double lo = (double)ordered_to_float(box[threadIdx.x]);
    const double ext = __dsub_rn((double)ordered_to_float(box[3 + threadIdx.x]), lo);
    s_lo[threadIdx.x] = lo;
    s_scale[threadIdx.x] = ext > 0.0 ? __ddiv_rn(twoB, ext) : 0.0;
  }
  __syncthreads();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  uint64_t q[3] = {0, 0, 0};
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const double t = __dmul_rn(__dsub_rn((double)__ldg(pts + k * DIM + d), s_lo[d]), s_scale[d]);
    q[d] = t >= twoB ? qmax : (uint64_t)t;
  }
  uint64_t hi, lo;
  if (DIM == 3) {
    const uint64_t H = interleave((uint32_t)(q[0] >> 21), (uint32_t)(q[1] >> 21), (uint32_t)(q[2] >> 21), 3);
    const uint64_t L = interleave((uint32_t)(q[0] & 0x1fffffu), (uint32_t)(q[1] & 0x1fffffu),
                                  (uint32_t)(q[2] & 0x1fffffu), 3);
    hi = H >> 1;
    lo = L | (H << 63);
  } else {
    hi = interleave((uint32_t)(q[0] >> 32), (uint32_t)(q[1] >> 32), 0u, 2);
    lo = interleave((uint32_t)q[0], (uint32_t)q[1], 0u, 2);
  }
  (void)B;
  code_hi[k] = hi;
  code_lo[k] = lo;
  keys[k] = lo;
  vals[k] = (uint32_t)k;
}

void launch_morton128(Problem &P) {
  const ClearWords clear = {P.sort_state, sort_clear_words(P.n)};
  int g = grid_for(P.n, kBlock);
  if (P.dim == 3)
    launch_next(P, k_morton128<3>, g, kBlock, 0, P.points, P.n, P.counters + 4, P.wide_hi, P.wide_lo,
                                               P.keys[0], P.vals[0], clear);
  else
    launch_next(P, k_morton128<2>, g, kBlock, 0, P.points, P.n, P.counters + 4, P.wide_hi, P.wide_lo,
                                               P.keys[0], P.vals[0], clear);
  P.launches += 1;
}

// out[k] = src[idx[k]] (a 64-bit word carried through a permutation)
__global__ void k_gather_u64(const uint64_t *__restrict__ src, const uint32_t *__restrict__ idx,
                             int64_t n, uint64_t *__restrict__ out) {
  wait_for_previous();
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = __ldg(src + __ldg(idx + k));
}

void launch_gather_u64(Problem &P, const uint64_t *src, const uint32_t *idx, uint64_t *out) {
  launch_next(P, k_gather_u64, grid_for(P.n, kBlock), kBlock, 0, src, idx, P.n, out);
  P.launches += 1;
}

// Instance id of every input row (binary search in the offsets).
__global__ void __launch_bounds__(kBlock) k_instance_ids(const int64_t *__restrict__ offsets,
                                                         int64_t num_inst, int64_t n,
                                                         uint32_t *__restrict__ inst_in) {
  wait_for_previous();
  __shared__ int64_t s_end[2];  // the instances of the CTA's first and last row
  const int64_t first = (int64_t)blockIdx.x * blockDim.x, k = first + threadIdx.x;
  auto find = [&](int64_t row, int64_t lo, int64_t hi) {  // last instance whose start is <= row
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (__ldg(offsets + mid) <= row) lo = mid; else hi = mid - 1;
    }
    return lo;
  };
  if (threadIdx.x < 64 && (threadIdx.x & 31) == 0)
    s_end[threadIdx.x >> 5] =
        find(threadIdx.x == 0 ? first : min(first + (int64_t)blockDim.x, n) - 1, 0, num_inst - 1);
  __syncthreads();
  if (k < n) inst_in[k] = (uint32_t)find(k, s_end[0], s_end[1]);
}

void launch_instance_ids(Problem &P) {
  launch_next(P, k_instance_ids, grid_for(P.n, kBlock), kBlock, 0, P.offsets, P.num_inst, P.n,
                                                                 P.inst_in);
  P.launches += 1;
}

// Root node of each instance's subtree: the node whose chunk range is exactly
// the instance's (one of its two ends is the node's index); kInvalid for an
// instance with fewer than two chunks... of points (nothing to search).
__global__ void __launch_bounds__(kBlock) k_instance_roots(const int64_t *__restrict__ offsets,
                                                           int64_t num_inst, int64_t nc, int leaf,
                                                           const uint2 *__restrict__ range,
                                                           uint32_t *__restrict__ inst_root,
                                                           uint32_t *status) {
  wait_for_previous();
  int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= num_inst) return;
  const int64_t a = __ldg(offsets + I), b = __ldg(offsets + I + 1) - 1;
  if (b <= a) { inst_root[I] = kInvalid; return; }
  const int64_t ca = a / leaf, cb = b / leaf;
  uint32_t root = kInvalid;
  if (ca == cb) {
    root = kInvalid;  // inside one leaf chunk: cannot happen with leaf 1 (a < b)
  } else {
    if (ca < nc - 1) {
      const NodeRange r = unpack_range((uint32_t)ca, __ldg(range + ca));
      if (r.first == (uint32_t)ca && r.last == (uint32_t)cb) root = (uint32_t)ca;
    }
    if (root == kInvalid && cb < nc - 1) {
      const NodeRange r = unpack_range((uint32_t)cb, __ldg(range + cb));
      if (r.first == (uint32_t)ca && r.last == (uint32_t)cb) root = (uint32_t)cb;
    }
  }
  if (root == kInvalid) atomicOr(status, kErrChain);
  inst_root[I] = root;
}

void launch_instance_roots(Problem &P) {
  launch_next(P, k_instance_roots, grid_for(P.num_inst, kBlock), kBlock, 0, P.offsets, P.num_inst, P.nc, P.leaf, P.range, P.inst_root, P.counters + 1);
  P.launches += 1;
}

// ---------------------------------------------------------------------------
// A4 (a). Gather the points into curve order as float4 (x, y, z, original
// index bits) and the first labels (labels(i) = i, Fig. 3), in curve indices.
// ---------------------------------------------------------------------------
// Also counts, over the curve positions whose code equals the previous
// position's: identical points (dup[0]) and distinct points the grid does not
// separate (dup[1]: a cell holding many of them has no spatial order inside,
// so its subtree's boxes all span it); and flags (dup[2] != 0) a run of more
// than 32 equal codes -- the only way a group of identical points can be
// large, which is when the search needs its tie rule.
// code_hi: the codes' high words (128-bit codes), else nullptr.
template <int DIM>
__global__ void __launch_bounds__(kBlock) k_gather(const float *__restrict__ pts,
                                                   const uint32_t *__restrict__ perm, int64_t n,
                                                   float4 *__restrict__ out,
                                                   uint32_t *__restrict__ labels,
                                                   const uint32_t *__restrict__ inst_in,
                                                   uint32_t *__restrict__ inst_of,
                                                   const uint64_t *__restrict__ sorted_codes,
                                                   const uint64_t *__restrict__ code_hi,
                                                   unsigned long long *dup) {
  wait_for_previous();
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  bool same = false, differ = false, run = false, longer = false;
  if (k < n) {
    const uint32_t o = __ldg(perm + k);
    if (inst_of) inst_of[k] = __ldg(inst_in + o);
    const float *p = pts + (int64_t)o * DIM;
    const float x = __ldg(p), y = __ldg(p + 1), z = DIM == 3 ? __ldg(p + 2) : 0.0f;
    out[k] = make_float4(x, y, z, __uint_as_float(o));
    labels[k] = (uint32_t)k;
    auto equal_codes = [&](int64_t j) {
      return __ldg(sorted_codes + k) == __ldg(sorted_codes + j) && (!code_hi || __ldg(code_hi + k) == __ldg(code_hi + j));
    };
    if (k > 0 && equal_codes(k - 1)) {
      const float *q = pts + (int64_t)__ldg(perm + k - 1) * DIM;
      differ = __ldg(q) != x || __ldg(q + 1) != y || (DIM == 3 && __ldg(q + 2) != z);
      same = !differ;
    }
    // sorted codes: equal 32 positions back means all between are equal too
    run = k >= 32 && equal_codes(k - 32);
    // and, two longer than a run of equal keys that the output orders in place
    // (kTieRunMax), for it to choose its sort
    longer = run && k >= kGroupLong && equal_codes(k - kGroupLong);
  }
  // one atomic per CTA and counter (one per warp, all on the same words, made
  // this pass three times as long on dense clusters: 95 -> 32 us for 2M points)
  const int cs = __syncthreads_count(same), cd = __syncthreads_count(differ);
  const int cr = __syncthreads_or(run) ? (__syncthreads_or(longer) ? 3 : 1) : 0;
  if (threadIdx.x == 0) {
    if (cs) atomicAdd(dup, (unsigned long long)cs);
    if (cd) atomicAdd(dup + 1, (unsigned long long)cd);
    if (cr) atomicOr(reinterpret_cast<unsigned int *>(dup + 2), (unsigned int)cr);
  }
}

void launch_gather(Problem &P, const uint32_t *perm) {
  int g = grid_for(P.n, kBlock);
  unsigned long long *dup = reinterpret_cast<unsigned long long *>(P.counters + 28);
  // (zero since the call's first kernel, unless the order is rebuilt)
  if (P.wide) cudaMemsetAsync(dup, 0, 3 * sizeof(unsigned long long), P.stream);
  if (P.dim == 3)
    launch_next(P, k_gather<3>, g, kBlock, 0, P.points, perm, P.n, P.pts, P.labels, P.inst_in,
                                            P.inst_of, P.keys[0], P.code_hi, dup);
  else
    launch_next(P, k_gather<2>, g, kBlock, 0, P.points, perm, P.n, P.pts, P.labels, P.inst_in,
                                            P.inst_of, P.keys[0], P.code_hi, dup);
  P.launches += 1;
}

// ---------------------------------------------------------------------------
// A4 (b, c). Hierarchy and boxes without a climb.
// The hierarchy is Karras's binary radix tree over the leaf chunks (chunks of
// `leaf` consecutive sorted points; leaf = 1: one point per leaf; chunk c's
// key is the code of its first point, augmented by c so equal codes still
// split), numbered as in Fig. 4: internal node i covers a chunk range with
// one end at i, and its split gamma gives the children gamma (left) and
// gamma + 1 (right), leaves when the range ends there.
// With delta(i) the leading bits shared by the keys of chunks i and i + 1,
// the node of split s covers the chunks between the nearest splits p < s < q
// of smaller delta, [p + 1, q] (within any node's range the smallest delta
// occurs once: there the first differing bit goes from 0 to 1).  It hangs on
// the side of the larger of delta(p) and delta(q): under q as its left child
// when delta(q) is larger (its index is then its right end q), else under p
// as its right child (its index is its left end).  So every node follows
// from three range queries: the two nearest smaller deltas, and the boxes of
// its two children -- no arrivals, no walk up the tree.
// k_build_tile: a CTA takes kBuildTile consecutive chunks, tabulates in
// shared memory the boxes of every run of 1, 2, 4, ... chunks and the minima
// of every run of 1, 2, 4, ... deltas, and a thread per split finds p and q
// by descending the tables and each child's box as the union of two runs.  A
// split whose p or q lies outside the CTA stays open; the subtrees between
// the open splits are done and leave as items (box, smallest original id,
// the open split after them and its delta), some 15 of 128 chunks.
// k_build_merge: the same over items instead of chunks, a group of CTAs'
// items per CTA, until one CTA has them all.  A CTA whose group has more
// items than its tables hold takes them in turn, keeping what stays open.
// What bounds it: shared-memory wavefronts and the tables' barriers at 28
// warps per SM.  Measured (us, the climb with one arrival per child that stood
// here before / this): CTA-local part 2,480 / 1,330 at 37M halo points (its
// bytes take 570), 23 / 13 at 200,000; the rest 413 / 219 and 79 / 22 -- a
// climb above the CTAs was a chain of two L2 round trips per level.  256
// chunks per CTA: whole call 35.43 against 35.19 ms at 37M, the same at 1M.
// The child labels are the round-0 ones (a one-point chunk k: label k;
// otherwise several components, kInvalid); a caller with other labels
// rewrites them (A5).
// ---------------------------------------------------------------------------
// kh != nullptr: 128-bit codes, kh their high words (the augmented key is
// then (high, low, position), 160 bits)
__device__ __forceinline__ int prefix_delta(const uint64_t *__restrict__ k,
                                            const uint64_t *__restrict__ kh, int64_t nc, int leaf,
                                            int64_t i, int64_t j) {
  if (j < 0 || j >= nc || i < 0 || i >= nc) return -1;
  int base = 0;
  if (kh) {
    const uint64_t a = __ldg(kh + i * leaf), b = __ldg(kh + j * leaf);
    if (a != b) return __clzll((long long)(a ^ b));
    base = 64;
  }
  uint64_t a = __ldg(k + i * leaf), b = __ldg(k + j * leaf);
  if (a != b) return base + __clzll((long long)(a ^ b));
  return base + 64 + __clz((int)((uint32_t)i ^ (uint32_t)j));
}

#ifndef EMST_BUILD_TILE
#define EMST_BUILD_TILE 128
#endif
constexpr int kBuildTile = EMST_BUILD_TILE;  // leaf chunks per k_build_tile CTA
constexpr int kMergeTile = 256;              // items in a k_build_merge CTA's tables
// The last CTA's: at most 160 splits stay open on either side of what a CTA
// holds (their deltas, below 161, fall towards it), so 512 always leave room.
constexpr int kLastTile = 512;
constexpr int kMaxGroup = 64;                // CTAs whose items one CTA takes

__device__ __forceinline__ void chunk_box(const float4 *__restrict__ pts, int64_t n, int leaf,
                                          int64_t c, float4 &lo, float4 &hi) {
  const int64_t p0 = c * leaf, p1 = p0 + leaf < n ? p0 + leaf : n;
  lo = hi = __ldg(pts + p0);
  for (int64_t m = p0 + 1; m < p1; ++m) {
    const float4 p = __ldg(pts + m);
    lo.x = fminf(lo.x, p.x); lo.y = fminf(lo.y, p.y); lo.z = fminf(lo.z, p.z);
    hi.x = fmaxf(hi.x, p.x); hi.y = fmaxf(hi.y, p.y); hi.z = fmaxf(hi.z, p.z);
    lo.w = __uint_as_float(min(__float_as_uint(lo.w), __float_as_uint(p.w)));
  }
}

// A subtree's box; lo.w: its smallest original id.
struct Subtree {
  float4 lo, hi;
};
__device__ __forceinline__ Subtree unite(const Subtree &a, const Subtree &b) {
  Subtree r;
  r.lo.x = fminf(a.lo.x, b.lo.x); r.lo.y = fminf(a.lo.y, b.lo.y); r.lo.z = fminf(a.lo.z, b.lo.z);
  r.hi.x = fmaxf(a.hi.x, b.hi.x); r.hi.y = fmaxf(a.hi.y, b.hi.y); r.hi.z = fmaxf(a.hi.z, b.hi.z);
  r.lo.w = __uint_as_float(min(__float_as_uint(a.lo.w), __float_as_uint(b.lo.w)));
  r.hi.w = 0.f;
  return r;
}

// Items 0 .. N-1 of a CTA with the splits around them: entry e is the split
// before item e (entry N the one after the last item).
template <int TILE>
struct BuildTables {
  static constexpr int kLevels = TILE == 128 ? 7 : TILE == 256 ? 8 : 9;
  static_assert(TILE == 1 << kLevels, "a power of two");
  float4 lo[kLevels][TILE];                // [k][i]: items i .. i + 2^k - 1
  float4 hi[kLevels][TILE];
  int16_t delta[kLevels + 1][TILE + 2];    // [k][e]: entries e .. e + 2^k - 1
  uint32_t pos[TILE + 1];                  // the splits' chunk positions (k_build_merge)
  uint32_t open[TILE / 32];
  uint32_t before[kMaxGroup + 1];          // k_build_merge: items of the group's CTAs before each
};

struct TreeOut {
  // not null: nothing to build when more than n / 64 codes collide (the host
  // is about to find the same count and starts over with 128-bit codes)
  const unsigned long long *collisions;
  NodeRec *nodes;
  uint2 *nlabels, *range;
  uint32_t *mixed;
  int64_t n, nc;
  int leaf;
};

__device__ __forceinline__ bool abandoned(const TreeOut &T) {
  return T.collisions && __ldcg(T.collisions) * 64ull > (unsigned long long)T.n;
}

// Node `idx` covering chunks [L, R] with split g and children's boxes a, b:
// its record, range and round-0 child labels.
__device__ __forceinline__ void write_node(const TreeOut &T, uint32_t idx, uint32_t L, uint32_t g, uint32_t R,
                                           const Subtree &a, const Subtree &b) {
  const bool lleaf = L == g, rleaf = R == g + 1u;
  NodeRec *rec = T.nodes + idx;
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(rec), "f"(a.lo.x), "f"(a.lo.y),
               "f"(a.lo.z), "f"(a.hi.x), "f"(a.hi.y), "f"(a.hi.z), "f"(b.lo.x), "f"(b.lo.y)
               : "memory");
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                   reinterpret_cast<char *>(rec) + 32),
               "f"(b.lo.z), "f"(b.hi.x), "f"(b.hi.y), "f"(b.hi.z),
               "f"(__uint_as_float(lleaf ? (kLeafBit | g) : g)),
               "f"(__uint_as_float(rleaf ? (kLeafBit | (g + 1u)) : g + 1u)), "f"(a.lo.w), "f"(b.lo.w)
               : "memory");
  T.range[idx] = pack_range(idx, L, g, R);
  // a chunk of exactly one point is its own component in round 0
  auto one_point = [&](int64_t c) { return T.leaf == 1 || T.n - c * T.leaf == 1; };
  T.nlabels[idx] = make_uint2(lleaf && one_point(g) ? (uint32_t)((int64_t)g * T.leaf) : kInvalid,
                              rleaf && one_point(g + 1) ? (uint32_t)((int64_t)(g + 1) * T.leaf) : kInvalid);
}

// One step over the N items in the tables' level 0 (filled by the caller, a
// barrier not yet passed): builds every node whose range ends inside, and
// returns for each thread whether the split after its item is open (the last
// one always counts as open), and then the subtree between the open split
// before and that one, and its rank among them.  LINEAR: item i is chunk
// first + i.  Every thread of the CTA (one per item) calls.
template <int TILE, bool LINEAR>
__device__ __forceinline__ bool build_step(BuildTables<TILE> &S, int N, uint32_t first, const TreeOut &T,
                                           Subtree &item, int &rank, int &count) {
  constexpr int kLevels = BuildTables<TILE>::kLevels;
  const int i = threadIdx.x;
  __syncthreads();
  {
    Subtree me;
    int low = 0;
    if (i < N) { me.lo = S.lo[0][i]; me.hi = S.hi[0][i]; }
    if (i <= N) low = S.delta[0][i];
#pragma unroll
    for (int k = 1; k <= kLevels; ++k) {
      const int h = 1 << (k - 1);
      if (2 * h > N + 1) break;
      if (k < kLevels && i + 2 * h <= N) {
        Subtree o;
        o.lo = S.lo[k - 1][i + h];
        o.hi = S.hi[k - 1][i + h];
        me = unite(me, o);
        S.lo[k][i] = me.lo;
        S.hi[k][i] = me.hi;
      }
      if (i + 2 * h <= N + 1) {
        low = min(low, (int)S.delta[k - 1][i + h]);
        S.delta[k][i] = (int16_t)low;
      }
      __syncthreads();
    }
  }
  auto at = [&](int e) { return LINEAR ? first - 1u + (uint32_t)e : S.pos[e]; };
  // the union of items [a, a + len): two runs that cover it
  auto run = [&](int a, int len) {
    int k = 31 - __clz(len);
    if (k > kLevels - 1) k = kLevels - 1;
    Subtree r;
    r.lo = S.lo[k][a];
    r.hi = S.hi[k][a];
    if (len > (1 << k)) {
      Subtree o;
      o.lo = S.lo[k][a + len - (1 << k)];
      o.hi = S.hi[k][a + len - (1 << k)];
      r = unite(r, o);
    }
    return r;
  };
  bool open = i < N;
  if (i < N - 1) {
    const int e = i + 1;
    const int d = S.delta[0][e];
    int p = e, q = e + 1;  // entries [p, e) and (e, q) lie above d
#pragma unroll
    for (int k = kLevels; k >= 0; --k) {
      if (p >= (1 << k) && S.delta[k][p - (1 << k)] > d) p -= 1 << k;
      if (q + (1 << k) <= N + 1 && S.delta[k][q] > d) q += 1 << k;
    }
    if (p > 0 && q <= N) {
      open = false;
      --p;
      const Subtree a = run(p, e - p), b = run(e, q - e);
      const uint32_t L = at(p) + 1u, R = at(q);
      const int dl = S.delta[0][p], dr = S.delta[0][q];
      // (the root: both outer deltas are -1)
      const uint32_t idx = dr > dl ? R : dl < 0 ? 0u : L;
      write_node(T, idx, L, at(e), R, a, b);
    }
  }
  const unsigned b = __ballot_sync(0xffffffffu, open);
  const int warp = i >> 5;
  if ((i & 31) == 0) S.open[warp] = b;
  __syncthreads();
  rank = 0;
  count = 0;
#pragma unroll
  for (int w = 0; w < TILE / 32; ++w) {
    const int c = __popc(S.open[w]);
    rank += w < warp ? c : 0;
    count += c;
  }
  unsigned m = b & ((1u << (i & 31)) - 1u);
  rank += __popc(m);
  if (open) {
    int w = warp;
    while (m == 0u && w > 0) m = S.open[--w];
    const int prev = m ? w * 32 + 31 - __clz(m) : -1;
    item = run(prev + 1, i - prev);
  }
  return open;
}

// Where the items of a CTA lie: from its first chunk's place on.
struct Items {
  float4 *lo, *hi;  // hi.w: the position of the open split after it
  int *delta;       // of that split
};

template <int TILE>
__global__ void __launch_bounds__(TILE) k_build_tile(const uint64_t *__restrict__ keys,
                                                     const uint64_t *__restrict__ keys_hi,
                                                     const float4 *__restrict__ pts, TreeOut T, Items items,
                                                     uint32_t *__restrict__ counts, uint32_t *status) {
  wait_for_previous();
  if (abandoned(T)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BuildTables<TILE> &S = *reinterpret_cast<BuildTables<TILE> *>(smem_raw);
  const int i = threadIdx.x;
  const int64_t first = (int64_t)blockIdx.x * TILE;
  const int N = (int)(T.nc - first < TILE ? T.nc - first : TILE);
  if (i < N) {
    float4 lo, hi;
    chunk_box(pts, T.n, T.leaf, first + i, lo, hi);
    S.lo[0][i] = lo;
    S.hi[0][i] = hi;
  }
  for (int e = i; e <= N; e += TILE)
    S.delta[0][e] = (int16_t)prefix_delta(keys, keys_hi, T.nc, T.leaf, first - 1 + e, first + e);
  Subtree item;
  int rank, count;
  const bool open = build_step<TILE, true>(S, N, (uint32_t)first, T, item, rank, count);
  // every node still has its child labels to be rewritten (k_node_labels)
  if (i < TILE / 32 && first + i * 32 < T.nc - 1) T.mixed[first / 32 + i] = 0xffffffffu;
  if (gridDim.x == 1) {
    if (i == 0 && count != 1) atomicOr(status, kErrChain);  // cannot happen: both ends are here
    return;
  }
  if (open) {
    items.lo[first + rank] = item.lo;
    items.hi[first + rank] = make_float4(item.hi.x, item.hi.y, item.hi.z, __uint_as_float((uint32_t)(first + i)));
    items.delta[first + rank] = S.delta[0][i + 1];
  }
  if (i == 0) counts[blockIdx.x] = (uint32_t)count;
}

// The items of `group` CTAs of the launch before (each CTA's from place
// span * its index on) reduced to what stays open, in their own first places:
// no more are written than were read, so nothing unread is overwritten.
template <int TILE>
__global__ void __launch_bounds__(TILE) k_build_merge(const uint64_t *__restrict__ keys,
                                                      const uint64_t *__restrict__ keys_hi, TreeOut T, Items items,
                                                      int64_t span, int group, int64_t ctas_in,
                                                      const uint32_t *__restrict__ counts_in,
                                                      uint32_t *__restrict__ counts, uint32_t *status) {
  wait_for_previous();
  if (abandoned(T)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BuildTables<TILE> &S = *reinterpret_cast<BuildTables<TILE> *>(smem_raw);
  const int i = threadIdx.x;
  const int64_t c0 = (int64_t)blockIdx.x * group;
  const int ctas = (int)(ctas_in - c0 < group ? ctas_in - c0 : group);
  const int64_t first = c0 * span;
  const bool last_cta = gridDim.x == 1;
  if (i < kMaxGroup + 1) S.before[i] = i > 0 && i <= ctas ? counts_in[c0 + i - 1] : 0u;
  if (i == TILE - 1) {
    S.pos[0] = (uint32_t)first - 1u;
    S.delta[0][0] = (int16_t)prefix_delta(keys, keys_hi, T.nc, T.leaf, first - 1, first);
  }
  __syncthreads();
  if (i < 32) {  // running totals of two counts per lane
    static_assert(kMaxGroup == 64, "two counts per lane");
    const uint32_t a = S.before[2 * i + 1], b = S.before[2 * i + 2];
    uint32_t x = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
      if (i >= o) x += y;
    }
    S.before[2 * i + 1] = x - b;
    S.before[2 * i + 2] = x;
  }
  __syncthreads();
  const int total = (int)S.before[ctas];
  int have = 0, read = 0;
  int64_t out = first;
  for (;;) {
    const int take = min(total - read, TILE - have);
    if (i < take) {
      const uint32_t f = (uint32_t)(read + i);
      int lo = 0, hi = ctas - 1;  // the last CTA whose items start at or before f
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (S.before[mid] <= f) lo = mid;
        else hi = mid - 1;
      }
      const int64_t at = first + lo * span + (int64_t)(f - S.before[lo]);
      const float4 hi4 = items.hi[at];
      S.lo[0][have + i] = items.lo[at];
      S.hi[0][have + i] = hi4;
      S.pos[have + i + 1] = __float_as_uint(hi4.w);
      S.delta[0][have + i + 1] = (int16_t)items.delta[at];
    }
    read += take;
    have += take;
    Subtree item;
    int rank, count;
    const bool open = build_step<TILE, false>(S, have, 0u, T, item, rank, count);
    const bool more = read < total;
    const uint32_t pos = open ? S.pos[i + 1] : 0u;
    const int16_t delta = open ? S.delta[0][i + 1] : (int16_t)0;
    __syncthreads();
    if (more && (last_cta || count <= TILE / 2)) {  // on with these and the next ones
      if (open) {
        S.lo[0][rank] = item.lo;
        S.hi[0][rank] = item.hi;
        S.pos[rank + 1] = pos;
        S.delta[0][rank + 1] = delta;
      }
      have = count;
      if (have >= TILE) {  // cannot happen (kLastTile)
        if (i == 0) atomicOr(status, kErrChain);
        return;
      }
      continue;
    }
    if (open) {
      items.lo[out + rank] = item.lo;
      items.hi[out + rank] = make_float4(item.hi.x, item.hi.y, item.hi.z, __uint_as_float(pos));
      items.delta[out + rank] = delta;
    }
    out += count;
    if (!more) break;
    if (open && rank == count - 1) {  // a fresh start after the last one
      S.pos[0] = pos;
      S.delta[0][0] = delta;
    }
    have = 0;
  }
  if (i == 0) {
    counts[blockIdx.x] = (uint32_t)(out - first);
    if (last_cta && out - first != 1) atomicOr(status, kErrChain);  // cannot happen: the root is built
  }
}

void launch_build_tree(Problem &P, bool unless_colliding) {
  // The items lie in arrays that the rounds set up later (16, 16 and 4 bytes
  // per point), their counts in list_buf[1] (n words; a count per CTA of each launch).
  const unsigned long long *collisions =
      unless_colliding ? reinterpret_cast<const unsigned long long *>(P.counters + 30) : nullptr;
  const TreeOut T = {collisions, P.nodes, P.nlabels, P.range, P.mixed, P.n, P.nc, P.leaf};
  const Items items = {reinterpret_cast<float4 *>(P.comp_buf[0]), reinterpret_cast<float4 *>(P.comp_buf[1]),
                       reinterpret_cast<int *>(P.root)};
  static bool attr_set[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !attr_set[dev]) {
    cudaFuncSetAttribute(k_build_tile<kBuildTile>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(BuildTables<kBuildTile>));
    cudaFuncSetAttribute(k_build_merge<kMergeTile>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(BuildTables<kMergeTile>));
    cudaFuncSetAttribute(k_build_merge<kLastTile>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)sizeof(BuildTables<kLastTile>));
    if (dev < 64) attr_set[dev] = true;
  }
  int64_t ctas = (P.nc + kBuildTile - 1) / kBuildTile, span = kBuildTile;
  uint32_t *counts = P.list_buf[1];
  launch_next(P, k_build_tile<kBuildTile>, (unsigned)ctas, kBuildTile, sizeof(BuildTables<kBuildTile>), P.keys[0] /*sorted*/, P.code_hi, P.pts, T, items, counts, P.counters + 1);
  P.launches += 1;
  while (ctas > 1) {
    // groups of 16 while that leaves CTAs for the whole GPU, larger ones
    // (tables filled more than once per CTA) beyond that
    const int group = ctas <= kMaxGroup ? (int)ctas : ctas > 16384 ? kMaxGroup : 16;
    const int64_t next = (ctas + group - 1) / group;
    if (next == 1)
      launch_next(P, k_build_merge<kLastTile>, 1, kLastTile, sizeof(BuildTables<kLastTile>), P.keys[0], P.code_hi, T, items, span, group, ctas, counts, counts + ctas, P.counters + 1);
    else
      launch_next(P, k_build_merge<kMergeTile>, (unsigned)next, kMergeTile, sizeof(BuildTables<kMergeTile>), P.keys[0], P.code_hi, T, items, span, group, ctas, counts, counts + ctas, P.counters + 1);
    P.launches += 1;
    counts += ctas;
    ctas = next;
    span *= group;
  }
}

}  // namespace emst
