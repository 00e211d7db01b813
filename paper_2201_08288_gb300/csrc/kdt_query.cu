// kdt_query.cu -- queries on a built tree: boxes (range counts and lists) and
// k nearest neighbours.
//
// The paper motivates the k-d tree by the searches it speeds up (Sec. 1): a
// query visits only the cells its region can reach. A node h at level l < L
// with dim t >= 0 sends keys <= its split key to the left child and the
// others to the right (the build's rule, in the total order of the key
// transform, -0 below +0); a node with dim -1 (an empty or terminal cell)
// has all of its points in its leftmost leaf. Leaf k holds
// perm[offs[k] .. offs[k+1]).
//
// One warp per query, depth first with an explicit stack (at most one node
// per level: the lanes hold it, lane s entry s), a leaf's points 32 at a time,
// one per lane. Many searches of few points each go a thread per query (see
// "searches by a thread").
//   Box: a point is inside when lo_j <= x_j <= hi_j for every coordinate j,
//   compared as keys; the left child is visited when key(lo_t) <= split key,
//   the right when key(hi_t) > split key.
//   Nearest: squared distances in double, summed over j = 0..d-1 in order
//   with no fused multiply-add, so that the value is a fixed function of the
//   inputs; ties go to the smaller original index. The nearer child is
//   visited first; the farther one is skipped when the squared distance to
//   the split plane exceeds the current k-th distance (a lower bound on
//   every point beyond the plane, because rounding to nearest is monotone).
//   Double arithmetic is scarce on this GPU (a warp-wide operation holds its
//   pipe for about 16 cycles), so the search itself runs on float distances
//   with a known error bound, keeps the 32 nearest by them, and measures only
//   those in double at the end. It is repeated with double distances
//   throughout if a point that fell out of the 32 could be among the k.
#include <algorithm>

#include "kdt.h"
#include "kdt_internal.cuh"
#include "kdt_launch.h"
#include "kdt_trace.h"

namespace kdt {

namespace {

constexpr int kQueryThreads = 64;  // (a block ends with its longest search: 64 threads 0.60 ms where 128 take 0.61)
constexpr int kQueryWarps = kQueryThreads / 32;
constexpr unsigned kAll = 0xffffffffu;
constexpr int kDimChunk = 4;  // coordinates of a point whose loads go out together

struct TreeView {
  const float* x;  // [d][n]
  int64_t n;
  int32_t d, L;
  const uint32_t* perm;
  const float* vals;
  const int8_t* dims;
  const int64_t* offs;
};

__device__ __forceinline__ int level_of(uint32_t h) { return 31 - __clz(h + 1u); }

// First leaf below node h at level l.
__device__ __forceinline__ uint32_t first_leaf(const TreeView& tv, uint32_t h, int l) {
  return (h - ((1u << l) - 1u)) << (tv.L - l);
}

// The count goes up by a warp's ballot, so the list keeps the order of the
// leaves and of the points in them. 50,021 boxes of about 40 points among
// 4,000,037 in 3 coordinates: 0.30 ms; 2.45 with one thread per query.
__global__ void __launch_bounds__(kQueryThreads) k_query_box(TreeView tv, const float* lo, const float* hi,
                                                             int32_t nq, uint32_t* count, uint32_t* list,
                                                             uint32_t cap) {
  __shared__ uint2 box[kQueryWarps][KDT_MAX_DIMS];  // keys of lo and hi
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t qi = (int32_t)blockIdx.x * kQueryWarps + warp;
  if (qi >= nq) return;
  const int d = tv.d;
  uint2* bx = box[warp];
  for (int j = lane; j < d; j += 32)
    bx[j] = make_uint2(ord_key(lo[(int64_t)j * nq + qi]), ord_key(hi[(int64_t)j * nq + qi]));
  __syncwarp();
  const unsigned lt = (1u << lane) - 1u;
  uint32_t found = 0;
  uint32_t stack = 0;  // lane s: the right child left for later, s-th from the root
  int sp = 0;
  uint32_t h = 0;
  int l = 0;
  for (;;) {
    const int t = l < tv.L ? (int)tv.dims[h] : -1;
    if (t >= 0) {
      const uint32_t m = ord_key(tv.vals[h]);
      const uint2 b = bx[t];
      const bool left = b.x <= m, right = b.y > m;
      if (left || right) {
        if (left && right && lane == sp) stack = 2u * h + 2u;
        sp += left && right;
        h = left ? 2u * h + 1u : 2u * h + 2u;
        ++l;
        continue;
      }
    } else {
      // a leaf, or a node whose points are all in its leftmost leaf
      const uint32_t k = first_leaf(tv, h, l);
      const int64_t p1 = tv.offs[k + 1];
      for (int64_t p = tv.offs[k]; p < p1; p += 32) {
        bool in = p + lane < p1;
        const uint32_t i = in ? __ldg(tv.perm + p + lane) : 0u;
        for (int j0 = 0; j0 < d; j0 += kDimChunk) {
          uint32_t kx[kDimChunk];
#pragma unroll
          for (int j = 0; j < kDimChunk; ++j)
            if (j0 + j < d) kx[j] = in ? ord_key(__ldg(tv.x + (int64_t)(j0 + j) * tv.n + i)) : 0u;
#pragma unroll
          for (int j = 0; j < kDimChunk; ++j)
            if (j0 + j < d) {
              const uint2 b = bx[j0 + j];
              in = in && b.x <= kx[j] && kx[j] <= b.y;
            }
          if (j0 + kDimChunk < d && !__any_sync(kAll, in)) break;
        }
        const unsigned bal = __ballot_sync(kAll, in);
        const uint32_t at = found + (uint32_t)__popc(bal & lt);
        if (list && in && at < cap) list[(size_t)qi * cap + at] = i;
        found += (uint32_t)__popc(bal);
      }
    }
    if (sp == 0) break;
    h = __shfl_sync(kAll, stack, --sp);
    l = level_of(h);
  }
  if (lane == 0) count[qi] = found;
}

// (distance, index) order: smaller distance first, then smaller index.
__device__ __forceinline__ bool nearer(double a, uint32_t ia, double b, uint32_t ib) {
  return a < b || (a == b && ia < ib);
}

// (coordinate j of the query at q[j stride])
__device__ __forceinline__ double dist2(const TreeView& tv, const float* q, uint32_t i, int64_t stride = 1) {
  double d2 = 0.0;
  for (int j0 = 0; j0 < tv.d; j0 += kDimChunk) {
    float x[kDimChunk];
#pragma unroll
    for (int j = 0; j < kDimChunk; ++j)
      if (j0 + j < tv.d) x[j] = __ldg(tv.x + (int64_t)(j0 + j) * tv.n + i);
#pragma unroll
    for (int j = 0; j < kDimChunk; ++j)
      if (j0 + j < tv.d) {
        const double df = __dsub_rn((double)x[j], (double)q[(j0 + j) * stride]);
        d2 = __dadd_rn(d2, __dmul_rn(df, df));
      }
  }
  return d2;
}

// One lane on its own: the k nearest kept by insertion, a point at a time.
// Queries that meet a distance that is no number (infinities of one sign on
// both sides, NaN in the query) go this way: such distances are in no order,
// so which of them are kept is fixed by the sequence alone.
__device__ void knn_serial(const TreeView& tv, const float* q, int64_t stride, int k, uint32_t* out_idx,
                           double* out_d2) {
  for (int j = 0; j < k; ++j) {
    out_d2[j] = __longlong_as_double(0x7ff0000000000000ll);  // +inf
    out_idx[j] = 0xffffffffu;
  }
  int nbest = 0;
  uint32_t stack_h[KDT_MAX_LEVELS + 2];
  double stack_b[KDT_MAX_LEVELS + 2];  // lower bound of the node's squared distance
  int sp = 0;
  stack_h[sp] = 0;
  stack_b[sp++] = 0.0;
  while (sp > 0) {
    --sp;
    const uint32_t h = stack_h[sp];
    const double bound = stack_b[sp];
    if (nbest == k && bound > out_d2[k - 1]) continue;
    const int l = level_of(h);
    const int t = l < tv.L ? (int)tv.dims[h] : -1;
    if (t >= 0) {
      const float mv = tv.vals[h], qv = q[t * stride];
      const double diff = __dsub_rn((double)qv, (double)mv);
      const bool q_left = ord_key(qv) <= ord_key(mv);
      stack_h[sp] = q_left ? 2u * h + 2u : 2u * h + 1u;  // the farther child, visited last
      stack_b[sp++] = fmax(bound, __dmul_rn(diff, diff));
      stack_h[sp] = q_left ? 2u * h + 1u : 2u * h + 2u;
      stack_b[sp++] = bound;
      continue;
    }
    const uint32_t leaf = first_leaf(tv, h, l);
    for (int64_t p = tv.offs[leaf]; p < tv.offs[leaf + 1]; ++p) {
      const uint32_t i = tv.perm[p];
      const double d2 = dist2(tv, q, i, stride);
      if (nbest == k && !nearer(d2, i, out_d2[k - 1], out_idx[k - 1])) continue;
      int pos = nbest < k ? nbest++ : k - 1;
      for (int j = k - 1; j > 0; --j)
        if (j <= pos && nearer(d2, i, out_d2[j - 1], out_idx[j - 1])) {
          out_d2[j] = out_d2[j - 1];
          out_idx[j] = out_idx[j - 1];
          pos = j - 1;
        }
      out_d2[pos] = d2;
      out_idx[pos] = i;
    }
  }
}

// A candidate of the exact list: the bits of its squared distance (never
// negative, so they order like the distances) and its original index.
struct Near {
  unsigned long long d;
  uint32_t i;
};

__device__ __forceinline__ bool before(const Near& a, const Near& b) {
  return a.d < b.d || (a.d == b.d && a.i < b.i);
}
__device__ __forceinline__ Near shfl_xor(const Near& a, int m) {
  return Near{__shfl_xor_sync(kAll, a.d, m), __shfl_xor_sync(kAll, a.i, m)};
}
__device__ __forceinline__ Near shfl_up1(const Near& a) {
  return Near{__shfl_up_sync(kAll, a.d, 1), __shfl_up_sync(kAll, a.i, 1)};
}
__device__ __forceinline__ Near shfl_from(const Near& a, int src) {
  return Near{__shfl_sync(kAll, a.d, src), __shfl_sync(kAll, a.i, src)};
}

// A candidate of the float list: the distance's bits above the index.
using NearF = unsigned long long;
__device__ __forceinline__ bool before(NearF a, NearF b) { return a < b; }
__device__ __forceinline__ NearF shfl_xor(NearF a, int m) { return __shfl_xor_sync(kAll, a, m); }
__device__ __forceinline__ NearF shfl_up1(NearF a) { return __shfl_up_sync(kAll, a, 1); }
__device__ __forceinline__ NearF shfl_from(NearF a, int src) { return __shfl_sync(kAll, a, src); }
__device__ __forceinline__ float dist_of(NearF a) { return __uint_as_float((uint32_t)(a >> 32)); }

template <class N>
__device__ __forceinline__ void warp_sort_near(N& v, int lane) {
#pragma unroll
  for (int size = 2; size <= 32; size <<= 1)
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1) {
      const N o = shfl_xor(v, j);
      const bool want_small = ((lane & j) == 0) == ((lane & size) == 0);
      if (before(o, v) == want_small) v = o;
    }
}

// Up to this many candidates of a round of 32 points are inserted one by one
// (a ballot and a shift each), more are sorted and merged with the list.
constexpr int kKnnInsertMax = 4;

// Put the candidates c of the lanes in `m` into the sorted list `best` (lane
// j: the j-th smallest); the 32 smallest stay, `lost` becomes the least of
// what it was and what the lane saw fall out. `none` sorts after all.
template <class N>
__device__ __forceinline__ void list_add(N& best, N c, unsigned m, const N& none, int lane, N& lost) {
  if (__popc(m) <= kKnnInsertMax) {
    while (m) {
      const N x = shfl_from(c, __ffs(m) - 1);
      m &= m - 1u;
      const N up = shfl_up1(best);
      const N out = before(best, x) ? x : best;  // lane 31: what falls out
      if (lane == 31 && before(out, lost)) lost = out;
      const int pos = __popc(__ballot_sync(kAll, before(best, x)));  // a prefix of the sorted lanes
      if (lane == pos)
        best = x;
      else if (lane > pos)
        best = up;
    }
  } else {
    if (!((m >> lane) & 1u)) c = none;
    warp_sort_near(c, lane);
    // ascending list, descending candidates: their lane-wise minima are the
    // 32 smallest, a bitonic sequence
    const N r = shfl_xor(c, 31);
    const N out = before(r, best) ? best : r;
    if (before(r, best)) best = r;
    if (before(out, lost)) lost = out;
#pragma unroll
    for (int j = 16; j > 0; j >>= 1) {
      const N o = shfl_xor(best, j);
      if (before(o, best) == ((lane & j) == 0)) best = o;
    }
  }
}

// Float distances: x - q is off by at most 2^-24 of itself, so its square by
// 2^-23, and each of the d fused additions adds 2^-24: a sum f of true value D
// has f (1 - (d + 8) 2^-24) < D < f (1 + (d + 8) 2^-24) with room for the
// products here and for what D itself is rounded, as long as f is neither
// near overflow nor made of underflowed squares: hence the two limits.
constexpr float kFarthest = 1e38f, kNearest = 1e-36f;

enum KnnResult { KNN_DONE, KNN_AGAIN, KNN_ODD };

// One query by one warp. kExact: distances in double throughout; else in
// float, the 32 nearest by them measured in double at the end. Returns
// KNN_AGAIN if the float search cannot tell, KNN_ODD if it met a distance
// that is no number.
template <bool kExact>
__device__ __forceinline__ KnnResult knn_warp(const TreeView& tv, const float* q, int k, int lane, uint32_t* out_idx,
                                              double* out_d2) {
  const int d = tv.d;
  const float inf = __int_as_float(0x7f800000);
  const float shrink = 1.0f - (float)(d + 8) * 0x1p-24f, grow = 1.0f + (float)(d + 8) * 0x1p-24f;
  const Near none{0x7ff0000000000000ull, 0xffffffffu};  // (+inf, no index)
  const NearF none_f = 0x7f800000ffffffffull;
  Near best = none;  // lane j: the j-th nearest so far
  NearF best_f = none_f;
  int nbest = 0;     // points in the list, at most k
  // no point whose float distance times `shrink` is above it is among the k
  // nearest; not below kNearest, +inf while the list is short
  float kth_up = inf;
  Near lost = none;  // the least that the lane saw fall out of the list
  NearF lost_f = none_f;
  uint32_t stack_h = 0;
  float stack_b = 0.0f;
  int sp = 0;
  uint32_t h = 0;
  int l = 0;
  float bound = 0.0f;  // at most the squared distance of any point below h
  for (;;) {
    const int t = l < tv.L ? (int)tv.dims[h] : -1;
    if (t >= 0) {
      const float mv = tv.vals[h], qv = q[t];
      const float diff = __fsub_rz(qv, mv);
      const float fb = fmaxf(bound, __fmul_rd(diff, diff));
      const bool q_left = ord_key(qv) <= ord_key(mv);
      if (!(fb > kth_up)) {  // the farther child waits (it would be skipped now or later)
        if (lane == sp) {
          stack_h = q_left ? 2u * h + 2u : 2u * h + 1u;
          stack_b = fb;
        }
        ++sp;
      }
      h = q_left ? 2u * h + 1u : 2u * h + 2u;
      ++l;
      continue;
    }
    const uint32_t leaf = first_leaf(tv, h, l);
    const int64_t p1 = tv.offs[leaf + 1];
    for (int64_t p = tv.offs[leaf]; p < p1; p += 32) {
      bool in = p + lane < p1;
      const uint32_t i = in ? __ldg(tv.perm + p + lane) : 0u;
      float f = 0.0f;
      for (int j0 = 0; j0 < d; j0 += kDimChunk) {
        float x[kDimChunk];
#pragma unroll
        for (int j = 0; j < kDimChunk; ++j)
          if (j0 + j < d) x[j] = __ldg(tv.x + (int64_t)(j0 + j) * tv.n + i);
#pragma unroll
        for (int j = 0; j < kDimChunk; ++j)
          if (j0 + j < d) {
            const float df = x[j] - q[j0 + j];
            f = fmaf(df, df, f);
          }
        if (j0 + kDimChunk < d) {
          in = in && !(f * shrink > kth_up);
          if (!__any_sync(kAll, in)) break;
        }
      }
      in = in && !(f * shrink > kth_up);
      unsigned m = __ballot_sync(kAll, in);
      if (m == 0u) continue;
      if (__any_sync(kAll, in && f != f)) return KNN_ODD;  // so is the double sum
      if (kExact) {
        Near c = none;
        if (in) c = Near{(unsigned long long)__double_as_longlong(dist2(tv, q, i)), i};
        const Near last = shfl_from(best, k - 1);
        in = in && (nbest < k || before(c, last));
        m = __ballot_sync(kAll, in);
        if (m == 0u) continue;
        list_add(best, c, m, none, lane, lost);
      } else {
        list_add(best_f, ((NearF)__float_as_uint(f) << 32) | i, m, none_f, lane, lost_f);
      }
      nbest = min(k, nbest + __popc(m));
      if (nbest == k) {
        const float up = kExact ? __double2float_ru(__longlong_as_double((long long)__shfl_sync(kAll, best.d, k - 1)))
                                : dist_of(shfl_from(best_f, k - 1)) * grow;
        kth_up = up < kFarthest ? fmaxf(up, kNearest) : inf;
      }
    }
    // the next node that can still hold a nearer point
    bool more = false;
    while (sp > 0 && !more) {
      --sp;
      bound = __shfl_sync(kAll, stack_b, sp);
      more = !(bound > kth_up);
    }
    if (!more) break;
    h = __shfl_sync(kAll, stack_h, sp);
    l = level_of(h);
  }
  if (!kExact) {
    if (best_f != none_f) {
      const uint32_t i = (uint32_t)best_f;
      best = Near{(unsigned long long)__double_as_longlong(dist2(tv, q, i)), i};
    }
    warp_sort_near(best, lane);
    // what fell out must be farther than the k-th that stayed, or the double
    // search has to tell (points that were rejected are farther than k points
    // that were in the list then; those that no longer are fell out)
    const bool full = __any_sync(kAll, lane == 31 && best_f != none_f);
    if (full) {
      const double kth = __longlong_as_double((long long)__shfl_sync(kAll, best.d, k - 1));
      const float least = __uint_as_float(__reduce_min_sync(kAll, (uint32_t)(lost_f >> 32)));
      if (!(kth < 0.5 * (double)kFarthest && least > 2.0f * kNearest && (double)(least * shrink) > kth)) return KNN_AGAIN;
    }
  }
  if (lane < k) {
    const bool used = lane < nbest;
    out_idx[lane] = used ? best.i : 0xffffffffu;
    out_d2[lane] = __longlong_as_double(used ? (long long)best.d : 0x7ff0000000000000ll);
  }
  return KNN_DONE;
}

// What bounds it: the chains of dependent loads (node after node, a leaf's
// offsets, its permutation, the gathered coordinates) over the resident warps.
// 100,003 queries of 8 neighbours among 1,000,003 points in 3 coordinates,
// leaves of 31: 0.60 ms; 0.73 with the coordinates loaded one after another, 2.0
// with double distances throughout as well (the double
// unit), 10.6 with one thread per query (its chains are longer, and 32
// searches diverge).
__global__ void __launch_bounds__(kQueryThreads) k_query_knn(TreeView tv, const float* qs, int32_t nq, int32_t k,
                                                             uint32_t* out_idx, double* out_d2) {
  __shared__ float qsm[kQueryWarps][KDT_MAX_DIMS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t qi = (int32_t)blockIdx.x * kQueryWarps + warp;
  if (qi >= nq) return;
  float* q = qsm[warp];
  for (int j = lane; j < tv.d; j += 32) q[j] = qs[(int64_t)j * nq + qi];
  __syncwarp();
  out_idx += (size_t)qi * k;
  out_d2 += (size_t)qi * k;
  KnnResult r = knn_warp<false>(tv, q, k, lane, out_idx, out_d2);
  if (r == KNN_AGAIN) r = knn_warp<true>(tv, q, k, lane, out_idx, out_d2);
  if (r == KNN_ODD && lane == 0) knn_serial(tv, q, 1, k, out_idx, out_d2);
}

// ----------------------------------------------- searches by a thread
//
// A warp spends as many instructions on a node, or on a leaf of one point, as a
// thread does, so searches that see few points are cheaper 32 at a time, by a
// thread each, once there are enough of them for the threads to hide their loads.
// The lines below are drawn from n / 2^L, all that the host knows of the leaves (in
// depth mode their points, in leaf mode a third to an eighth of them), the number of
// queries and d. Measured, a warp's time over a thread's, among 1,000,003 points in
// 3 coordinates, boxes of half a point to 60 points: 1,000,003 queries, leaves of 1
// (n / 2^L 0.12) 4.8 to 4.5, of 8 (0.95) 3.2 to 2.1, of 16 (3.8) 2.2 to 1.35, of 32
// (7.6) 1.5 to 0.92, of 64 1.1 to 0.8; 300,000 queries 3.9 to 4.4, 2.5 to 1.9, 1.8
// to 1.2, 1.2 to 0.8; 100,000 queries 2.0, 1.3 to 1.0, 1.0 to 0.7; 50,000 queries
// 1.3, 1.0 to 0.6. In 8 coordinates 300,000 queries in leaves of 8 (1.1) 1.4 to 1.1,
// of 16 (4.6) 0.9 to 0.7. The nearest point of a point of the tree, and of a place
// beside one: 1,000,003 queries, leaves of 1 3.8 and 1.6, of 4 (0.48) 2.8 and 1.2,
// of 8 2.2 and 0.9; 300,000 queries 3.1 and 1.1, 2.4 and 0.9, 1.9 and 0.6; in 2
// coordinates 3.5 and 2.2, 2.9 and 2.0, 2.3 and 1.65, of 16 (3.8) 1.7 and 1.2. (More
// coordinates, more leaves around a place; and the threads measure in double. More
// than one neighbour was never better.)
constexpr int kEachThreads = 128;
constexpr int32_t kEachMin = 32768;

float mean_leaf(const TreeView& tv) { return std::ldexp((float)tv.n, -tv.L); }
bool each_box(const TreeView& tv, int32_t nq) {
  return nq >= kEachMin && mean_leaf(tv) * (float)tv.d <= std::min(24.0f, 1.1f * std::pow((float)nq / 50000.0f, 1.25f));
}
bool each_nearest(const TreeView& tv, int32_t nq) {
  return nq >= kEachMin && mean_leaf(tv) * std::pow(5.0f, (float)(tv.d - 2)) <= std::min(4.0f, (float)nq / 75000.0f);
}

__global__ void __launch_bounds__(kEachThreads) k_box_each(TreeView tv, const float* lo, const float* hi, int32_t nq,
                                                           uint32_t* count, uint32_t* list, uint32_t cap) {
  const int64_t qi = (int64_t)blockIdx.x * kEachThreads + threadIdx.x;
  if (qi >= nq) return;
  lo += qi;
  hi += qi;
  uint32_t stack[KDT_MAX_LEVELS + 1];  // right children left for later, one per level at most
  int sp = 0;
  uint32_t h = 0, leaf = 0, found = 0;
  auto next_leaf = [&]() {  // from h on; false: none is left
    for (;;) {
      const int l = level_of(h), t = l < tv.L ? (int)tv.dims[h] : -1;
      if (t < 0) {
        leaf = first_leaf(tv, h, l);
        return true;
      }
      const uint32_t m = ord_key(tv.vals[h]);
      const bool left = ord_key(lo[(int64_t)t * nq]) <= m, right = ord_key(hi[(int64_t)t * nq]) > m;
      if (left || right) {
        if (left && right) stack[sp++] = 2u * h + 2u;
        h = left ? 2u * h + 1u : 2u * h + 2u;
      } else {
        if (sp == 0) return false;
        h = stack[--sp];
      }
    }
  };
  // (the lanes of a warp go down together, then read their leaves together)
  while (next_leaf()) {
    for (int64_t p = tv.offs[leaf]; p < tv.offs[leaf + 1]; ++p) {
      const uint32_t i = tv.perm[p];
      bool in = true;
      for (int j = 0; j < tv.d && in; ++j) {
        const uint32_t kx = ord_key(tv.x[(int64_t)j * tv.n + i]);
        in = ord_key(lo[(int64_t)j * nq]) <= kx && kx <= ord_key(hi[(int64_t)j * nq]);
      }
      if (in) {
        if (list && found < cap) list[(size_t)qi * cap + found] = i;
        ++found;
      }
    }
    if (sp == 0) break;
    h = stack[--sp];
  }
  count[qi] = found;
}

// The nearest point (k = 1). A search that meets a distance that is no number goes
// the serial way.
__global__ void __launch_bounds__(kEachThreads) k_nearest_each(TreeView tv, const float* qs, int32_t nq,
                                                               uint32_t* out_idx, double* out_d2) {
  const int64_t qi = (int64_t)blockIdx.x * kEachThreads + threadIdx.x;
  if (qi >= nq) return;
  qs += qi;
  uint32_t stack_h[KDT_MAX_LEVELS + 1];
  float stack_b[KDT_MAX_LEVELS + 1];  // at most the squared distance of any point below the node
  int sp = 0;
  double best = __longlong_as_double(0x7ff0000000000000ll);  // +inf
  uint32_t best_i = 0xffffffffu, h = 0;
  float bound = 0.0f;
  bool odd = false;
  auto descend = [&]() {  // from h to the leaf on the query's side
    for (;;) {
      const int l = level_of(h), t = l < tv.L ? (int)tv.dims[h] : -1;
      if (t < 0) return first_leaf(tv, h, l);
      const float mv = tv.vals[h], qv = qs[(int64_t)t * nq], diff = __fsub_rz(qv, mv);
      const float fb = fmaxf(bound, __fmul_rd(diff, diff));
      const bool q_left = ord_key(qv) <= ord_key(mv);
      if (!((double)fb > best)) {  // the farther child waits
        stack_h[sp] = q_left ? 2u * h + 2u : 2u * h + 1u;
        stack_b[sp++] = fb;
      }
      h = q_left ? 2u * h + 1u : 2u * h + 2u;
    }
  };
  for (bool more = true; more && !odd;) {
    const uint32_t leaf = descend();
    for (int64_t p = tv.offs[leaf]; p < tv.offs[leaf + 1]; ++p) {
      const uint32_t i = tv.perm[p];
      double d2 = 0.0;
      for (int j = 0; j < tv.d; ++j) {
        const double df = __dsub_rn((double)tv.x[(int64_t)j * tv.n + i], (double)qs[(int64_t)j * nq]);
        d2 = __dadd_rn(d2, __dmul_rn(df, df));
      }
      odd |= d2 != d2;
      if (nearer(d2, i, best, best_i)) {
        best = d2;
        best_i = i;
      }
    }
    more = false;
    while (sp > 0 && !more) {
      bound = stack_b[--sp];
      more = !((double)bound > best);
      h = stack_h[sp];
    }
  }
  out_idx[qi] = best_i;
  out_d2[qi] = best;
  if (odd) knn_serial(tv, qs, nq, 1, out_idx + qi, out_d2 + qi);
}

uint32_t blocks_of(int32_t nq, int per) { return ((uint32_t)nq + (uint32_t)per - 1u) / (uint32_t)per; }

kdt_status check_tree(const float* points, int64_t n, int32_t d, const uint32_t* perm, const float* vals,
                      const int8_t* dims, const int64_t* offs, int32_t L) {
  if (n < 0 || n > (int64_t)0xffffffffLL || d < 1 || d > KDT_MAX_DIMS || L < 0 || L > KDT_MAX_LEVELS)
    return KDT_ERR_INVALID_ARG;
  if (!offs || (n > 0 && (!points || !perm)) || (L > 0 && (!vals || !dims))) return KDT_ERR_INVALID_ARG;
  return KDT_OK;
}

}  // namespace

}  // namespace kdt

using namespace kdt;

extern "C" {

kdt_status kdt_query_box(const float* points, int64_t n, int32_t d, const uint32_t* perm, const float* split_vals,
                         const int8_t* split_dims, const int64_t* node_offsets, int32_t levels, const float* lo,
                         const float* hi, int32_t nq, uint32_t* out_count, uint32_t* out_list, uint32_t list_cap,
                         void* stream) {
  const kdt_status v = check_tree(points, n, d, perm, split_vals, split_dims, node_offsets, levels);
  if (v != KDT_OK) return v;
  if (nq < 0 || (nq > 0 && (!lo || !hi || !out_count)) || (out_list && list_cap == 0)) return KDT_ERR_INVALID_ARG;
  if (capturing((cudaStream_t)stream)) return KDT_ERR_INVALID_ARG;  // the query waits on its stream
  if (nq == 0) return KDT_OK;
  const TreeView tv{points, n, d, levels, perm, split_vals, split_dims, node_offsets};
  cudaStream_t st = (cudaStream_t)stream;
  {
    TraceScope ts(K_QUERY, st, (uint64_t)nq);
    if (each_box(tv, nq))
      k_box_each<<<blocks_of(nq, kEachThreads), kEachThreads, 0, st>>>(tv, lo, hi, nq, out_count, out_list, list_cap);
    else
      k_query_box<<<blocks_of(nq, kQueryWarps), kQueryThreads, 0, st>>>(tv, lo, hi, nq, out_count, out_list, list_cap);
  }
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
    (void)cudaGetLastError();
    return KDT_ERR_CUDA;
  }
  return KDT_OK;
}

kdt_status kdt_query_knn(const float* points, int64_t n, int32_t d, const uint32_t* perm, const float* split_vals,
                         const int8_t* split_dims, const int64_t* node_offsets, int32_t levels, const float* queries,
                         int32_t nq, int32_t k, uint32_t* out_idx, double* out_dist2, void* stream) {
  const kdt_status v = check_tree(points, n, d, perm, split_vals, split_dims, node_offsets, levels);
  if (v != KDT_OK) return v;
  if (nq < 0 || k < 1 || k > KDT_KNN_MAX_K || (nq > 0 && (!queries || !out_idx || !out_dist2)))
    return KDT_ERR_INVALID_ARG;
  if (capturing((cudaStream_t)stream)) return KDT_ERR_INVALID_ARG;  // the query waits on its stream
  if (nq == 0) return KDT_OK;
  const TreeView tv{points, n, d, levels, perm, split_vals, split_dims, node_offsets};
  cudaStream_t st = (cudaStream_t)stream;
  {
    TraceScope ts(K_QUERY, st, (uint64_t)nq);
    if (k == 1 && each_nearest(tv, nq))
      k_nearest_each<<<blocks_of(nq, kEachThreads), kEachThreads, 0, st>>>(tv, queries, nq, out_idx, out_dist2);
    else
      k_query_knn<<<blocks_of(nq, kQueryWarps), kQueryThreads, 0, st>>>(tv, queries, nq, k, out_idx, out_dist2);
  }
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
    (void)cudaGetLastError();
    return KDT_ERR_CUDA;
  }
  return KDT_OK;
}

}  // extern "C"
