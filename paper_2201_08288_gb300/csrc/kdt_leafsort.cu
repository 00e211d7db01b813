// kdt_leafsort.cu -- restore the order of the permutation inside every leaf.
//
// In the sequential definition of the build (paper, Sec. 2: each level
// partitions its cells around their splits) the partition is stable and
// starts from the identity, so inside every terminal cell the permutation is
// ascending original index. The multi-CTA pipeline keeps cells in subset
// order instead (every (cell, subset) segment contiguous), which leaves the
// same set of indices in every leaf in another order. This pass sorts each
// terminal cell's slice of the permutation ascending:
//   - up to kLeafWarpMax points: one warp, bitonic network in registers;
//   - up to kLeafBlockMax points: one CTA, one pass into buckets in shared
//     memory by the leading bits where the leaf's indices differ, then a warp's
//     network per bucket; with a bucket too full for a warp an LSD radix sort
//     (8-bit digits), stable ranks from warp match masks;
//   - up to kBucketPoints: the same buckets, a larger CTA;
//   - larger, or with a bucket too full for a warp: LSD passes over global
//     memory, tiles of kLeafBlockMax points, per-(tile, digit) counts scanned
//     per leaf.
// The last two are host-driven; only shallow trees or cells that stop
// splitting produce such leaves.
// Original indices are distinct, so the result does not depend on stability
// across equal keys; stability is what makes the LSD passes correct.
#include <algorithm>
#include <vector>

#include "kdt_internal.cuh"
#include "kdt_launch.h"
#include "kdt_trace.h"

namespace kdt {

namespace {

constexpr int kLsThreads = 256;
constexpr int kLsWarps = kLsThreads / 32;
constexpr int kLsItems = kLeafBlockMax / kLsThreads;  // 16 keys per thread
constexpr uint32_t kInvalidDigit = 256u;

// Number of 8-bit digits that cover original indices below n.
__host__ __device__ inline int index_digits(uint64_t n) {
  int bits = 0;
  while (bits < 32 && (n - 1) >> bits) ++bits;
  const int digits = (bits + 7) / 8;
  return digits > 1 ? digits : 1;
}

// -------------------------------------------------------- one warp, <= 32K

template <int K>
__device__ void warp_sort_slice(const uint32_t* a, uint32_t* out, uint32_t m) {
  const int lane = threadIdx.x & 31;
  uint32_t v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t e = (uint32_t)(k * 32 + lane);
    v[k] = e < m ? a[e] : 0xffffffffu;
  }
  constexpr int N = 32 * K;
#pragma unroll
  for (int size = 2; size <= N; size <<= 1) {
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1) {
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int e = k * 32 + lane;
        const bool asc = (e & size) == 0;
        if (j >= 32) {
          const int kk = k ^ (j >> 5);
          if (k < kk) {
            const uint32_t lo = min(v[k], v[kk]), hi = max(v[k], v[kk]);
            v[k] = asc ? lo : hi;
            v[kk] = asc ? hi : lo;
          }
        } else {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, v[k], j);
          const bool lower = (lane & j) == 0;
          v[k] = (lower == asc) ? min(v[k], o) : max(v[k], o);
        }
      }
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t e = (uint32_t)(k * 32 + lane);
    if (e < m) out[e] = v[k];
  }
}

// One warp: a[0..m) ascending into out (which may be a), m <= kLeafWarpMax.
__device__ void warp_sort_any(const uint32_t* a, uint32_t* out, uint32_t m) {
  if (m <= 32) warp_sort_slice<1>(a, out, m);
  else if (m <= 64) warp_sort_slice<2>(a, out, m);
  else if (m <= 128) warp_sort_slice<4>(a, out, m);
  else warp_sort_slice<8>(a, out, m);
}

// ------------------------------------------------------ block ranking

// Stable ranks by digit (key >> shift) & 255 of the m <= kLeafBlockMax keys
// src[0..m) (shared memory). Warp w owns positions [w*512, w*512+512) in 16
// rounds of 32 in order; within a round, lanes sharing a digit are ranked by
// their match mask. On return whist[w][b] holds the number of keys with digit
// b in warps before w, dtot[b] the keys with digit b, rank[j] the rank of the
// thread's j-th key among equal digits of its warp, dig[j] its digit.
__device__ void block_rank(const uint32_t* src, uint32_t m, int shift, uint32_t (*whist)[256], uint32_t* dtot,
                           uint32_t (&rank)[kLsItems], uint32_t (&dig)[kLsItems]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  for (int i = threadIdx.x; i < kLsWarps * 256; i += kLsThreads) (&whist[0][0])[i] = 0;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kLsItems; ++j) {
    const uint32_t idx = (uint32_t)(warp * (32 * kLsItems) + j * 32 + lane);
    const uint32_t dgt = idx < m ? (src[idx] >> shift) & 255u : kInvalidDigit;
    const unsigned peers = __match_any_sync(0xffffffffu, dgt);
    const uint32_t base = dgt != kInvalidDigit ? whist[warp][dgt] : 0u;
    __syncwarp();
    if (dgt != kInvalidDigit && (peers & lt) == 0u) whist[warp][dgt] = base + (uint32_t)__popc(peers);
    __syncwarp();
    rank[j] = base + (uint32_t)__popc(peers & lt);
    dig[j] = dgt;
  }
  __syncthreads();
  {
    const int b = threadIdx.x;  // kLsThreads == 256 digits
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < kLsWarps; ++w) {
      const uint32_t v = whist[w][b];
      whist[w][b] = run;
      run += v;
    }
    dtot[b] = run;
  }
  __syncthreads();
}

struct LsShared {
  uint32_t buf[2][kLeafBlockMax];
  uint32_t whist[kLsWarps][256];
  uint32_t dtot[256];
  uint32_t dbase[256];
  uint32_t tmp[33];
};

// One CTA: sort a[0..m) (global) with the keys staged in shared memory.
__device__ __noinline__ void block_sort_slice(uint32_t* a, uint32_t m, int digits, LsShared& S) {
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) S.buf[0][i] = a[i];
  __syncthreads();
  int cur = 0;
  for (int p = 0; p < digits; ++p) {
    uint32_t rank[kLsItems], dig[kLsItems];
    block_rank(S.buf[cur], m, 8 * p, S.whist, S.dtot, rank, dig);
    uint32_t tot;
    const uint32_t ex = block_excl_scan(S.dtot[threadIdx.x], S.tmp, &tot);
    S.dbase[threadIdx.x] = ex;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int j = 0; j < kLsItems; ++j) {
      if (dig[j] == kInvalidDigit) continue;
      const uint32_t idx = (uint32_t)(warp * (32 * kLsItems) + j * 32 + lane);
      S.buf[cur ^ 1][S.dbase[dig[j]] + S.whist[warp][dig[j]] + rank[j]] = S.buf[cur][idx];
    }
    __syncthreads();
    cur ^= 1;
  }
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) a[i] = S.buf[cur][i];
  __syncthreads();
}

// The same by buckets: false (nothing written) if one holds more than a warp
// sorts. A leaf of m keys gets between m / 64 and m / 16 buckets where they are
// spread evenly.
__device__ __noinline__ bool block_bucket_slice(uint32_t* a, uint32_t m, LsShared& S) {
  __shared__ uint32_t lohi[3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* count = &S.whist[0][0];
  count[threadIdx.x] = 0;
  if (threadIdx.x < 3) lohi[threadIdx.x] = threadIdx.x == 0 ? 0xffffffffu : 0u;
  __syncthreads();
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) {
    const uint32_t v = a[i];
    S.buf[0][i] = v;
    lo = min(lo, v);
    hi = max(hi, v);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lane == 0) {
    atomicMin(&lohi[0], lo);
    atomicMax(&lohi[1], hi);
  }
  __syncthreads();
  lo = lohi[0];
  const int bits = min(8, 27 - __clz(m));  // 2^bits <= m / 16
  const int shift = max(0, 32 - __clz(lohi[1] - lo) - bits);
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) atomicAdd(&count[(S.buf[0][i] - lo) >> shift], 1u);
  __syncthreads();
  const uint32_t c = count[threadIdx.x];
  const uint32_t most = __reduce_max_sync(0xffffffffu, c);
  if (lane == 0) atomicMax(&lohi[2], most);
  uint32_t tot;
  const uint32_t ex = block_excl_scan(c, S.tmp, &tot);
  S.dtot[threadIdx.x] = c;
  S.dbase[threadIdx.x] = ex;
  count[threadIdx.x] = ex;
  __syncthreads();
  if (lohi[2] > (uint32_t)kLeafWarpMax) {
    __syncthreads();  // lohi is read by all before the next leaf resets it
    return false;
  }
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) {
    const uint32_t v = S.buf[0][i];
    S.buf[1][atomicAdd(&count[(v - lo) >> shift], 1u)] = v;
  }
  __syncthreads();
  for (int b = warp; b < 256; b += kLsWarps) {
    const uint32_t w = S.dtot[b];
    if (w) warp_sort_any(S.buf[1] + S.dbase[b], a + S.dbase[b], w);
  }
  __syncthreads();
  return true;
}

// A range of CTAs per tree (SlotChunks). Warps sort the small terminal cells, CTAs the middle
// ones; the largest are listed for the global passes. Five CTAs per SM by a
// register bound: the warps' networks, which sort nearly every leaf of a deep
// tree, want the warps; the CTA paths, calls, spill (2^20 leaves of 128 points:
// 0.75 ms; 0.78 with the bucket path inlined).
__global__ void __launch_bounds__(kLsThreads, 5) k_leaf_sort(const TreeDev* trees, SlotChunks sc) {
  chain_wait();
  __shared__ LsShared S;
  uint32_t chunk, chunks;
  const TreeDev& t = trees[pick_chunk(sc, &chunk, &chunks)];
  if (!t.leafsort || *t.status != ST_OK || *t.live > 0) return;
  const uint32_t nrec = min(*t.term_count, t.term_cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t wstride = chunks * kLsWarps;
  uint32_t rec = chunk * kLsWarps + warp;
  TermRec trn = rec < nrec ? t.terms[rec] : TermRec{};
  for (; rec < nrec; rec += wstride) {
    const TermRec tr = trn;  // the next record is read before this cell is sorted
    if (rec + wstride < nrec) trn = t.terms[rec + wstride];
    if (tr.count <= 1u) continue;
    if (tr.count <= (uint32_t)kLeafWarpMax) {
      warp_sort_any(t.out_perm + tr.begin, t.out_perm + tr.begin, tr.count);
    } else if (tr.count > (uint32_t)kLeafBlockMax && lane == 0) {
      const uint32_t k = atomicAdd(t.huge_count, 1u);
      if (k < t.huge_cap) t.huge[k] = rec; else set_status(t, ST_CAPACITY);
    }
  }
  // the middle cells: the CTA reads its share of the records, up to kLsThreads
  // at once, and sorts the ones that need a CTA, one after another. (With
  // kLsThreads records per CTA whatever their number, 1024 leaves of 1950 points
  // had four CTAs at work, sorting by radix: kdt_build of 2,000,003 points in
  // three subsets took 4.9 ms, 1.1 now.)
  __shared__ uint32_t mids[kLsThreads];
  __shared__ uint32_t nmid;
  const int digits = index_digits((uint64_t)t.n);
  const uint32_t share = min((uint32_t)kLsThreads, (nrec + chunks - 1) / chunks);
  for (uint32_t base = chunk * share; base < nrec; base += chunks * share) {
    if (threadIdx.x == 0) nmid = 0;
    __syncthreads();
    const uint32_t rec = base + threadIdx.x;
    const uint32_t cnt = threadIdx.x < share && rec < nrec ? t.terms[rec].count : 0u;
    if (cnt > (uint32_t)kLeafWarpMax && cnt <= (uint32_t)kLeafBlockMax) mids[atomicAdd(&nmid, 1u)] = rec;
    __syncthreads();
    const uint32_t nm = nmid;
    for (uint32_t j = 0; j < nm; ++j) {
      const TermRec tr = t.terms[mids[j]];
      if (!block_bucket_slice(t.out_perm + tr.begin, tr.count, S))
        block_sort_slice(t.out_perm + tr.begin, tr.count, digits, S);
    }
    __syncthreads();  // mids and nmid are reused by the next chunk
  }
}

// ------------------------------------------------- one CTA, buckets (large leaves)

// Leaves of kLeafBlockMax + 1 .. kBucketPoints points, a CTA each: the indices
// are counted by bucket (bits above `shift`, the smallest that leaves at most
// kBuckets of them between the leaf's least and largest index, so 512 to 1024
// when they are spread evenly), moved into shared memory bucket by bucket, and
// each bucket is sorted by a warp in registers straight into the leaf's place.
// A leaf with a bucket above kLeafWarpMax is left as it is and its flag set
// (the caller sorts it by the global passes).
// What bounds it: the shared-memory atomics and the networks; the leaf is read
// three times, twice of them from L2. For 1024 leaves of 48,800 points it took
// 0.42 ms where the four global LSD passes took 2.03.
constexpr int kBucketThreads = 1024;
constexpr int kBuckets = 1024;
constexpr uint32_t kBucketPoints = 54272;
constexpr size_t kBucketSmem = (size_t)kBucketPoints * 4;

__global__ void __launch_bounds__(kBucketThreads) k_leaf_buckets(uint32_t* perm, const uint2* leaves, uint32_t nleaves,
                                                                 uint32_t* failed) {
  extern __shared__ __align__(16) uint32_t keys[];
  __shared__ uint32_t start[kBuckets + 1];
  __shared__ uint32_t cursor[kBuckets];
  __shared__ uint32_t tmp[33];
  __shared__ uint32_t s_lo, s_hi, s_most;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (uint32_t lf = blockIdx.x; lf < nleaves; lf += gridDim.x) {
    const uint32_t m = leaves[lf].y;
    uint32_t* a = perm + leaves[lf].x;
    if (tid == 0) {
      s_lo = 0xffffffffu;
      s_hi = 0u;
      s_most = 0u;
    }
    cursor[tid] = 0;
    __syncthreads();
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll 8
    for (uint32_t i = tid; i < m; i += kBucketThreads) {
      const uint32_t v = a[i];
      lo = min(lo, v);
      hi = max(hi, v);
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      atomicMin(&s_lo, lo);
      atomicMax(&s_hi, hi);
    }
    __syncthreads();
    lo = s_lo;
    const uint32_t span = s_hi - lo;
    const int shift = max(0, 32 - __clz(span) - 10);  // span >> shift < 1024
#pragma unroll 8
    for (uint32_t i = tid; i < m; i += kBucketThreads) atomicAdd(&cursor[(a[i] - lo) >> shift], 1u);
    __syncthreads();
    const uint32_t cnt = cursor[tid];
    const uint32_t most = __reduce_max_sync(0xffffffffu, cnt);
    if (lane == 0) atomicMax(&s_most, most);
    uint32_t tot;
    const uint32_t ex = block_excl_scan(cnt, tmp, &tot);
    start[tid] = ex;
    cursor[tid] = ex;
    if (tid == 0) start[kBuckets] = m;
    __syncthreads();
    if (s_most > (uint32_t)kLeafWarpMax) {
      if (tid == 0) failed[lf] = 1u;
      __syncthreads();  // s_most is read by all before the next leaf resets it
      continue;
    }
#pragma unroll 8
    for (uint32_t i = tid; i < m; i += kBucketThreads) {
      const uint32_t v = a[i];
      keys[atomicAdd(&cursor[(v - lo) >> shift], 1u)] = v;
    }
    __syncthreads();
    for (int b = warp; b < kBuckets; b += kBucketThreads / 32) {
      const uint32_t s0 = start[b], w = start[b + 1] - s0;
      if (w) warp_sort_any(keys + s0, a + s0, w);
    }
    __syncthreads();
  }
}

// --------------------------------------------- global passes (larger leaves)

// Tile of a large leaf: absolute begin of the leaf, its size, the tile's
// offset inside it.
struct LeafTile {
  uint32_t begin, count, off, pad;
};

__global__ void __launch_bounds__(kLsThreads) k_leaf_hist(const uint32_t* src, const LeafTile* tiles, int shift,
                                                          uint32_t* hist) {
  __shared__ uint32_t h[256];
  const LeafTile tl = tiles[blockIdx.x];
  h[threadIdx.x] = 0;
  __syncthreads();
  const uint32_t m = min((uint32_t)kLeafBlockMax, tl.count - tl.off);
  const uint32_t* a = src + tl.begin + tl.off;
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) atomicAdd(&h[(a[i] >> shift) & 255u], 1u);
  __syncthreads();
  hist[(size_t)blockIdx.x * 256 + threadIdx.x] = h[threadIdx.x];
}

// One CTA per large leaf (its tiles are [first, first + ntiles)): turn the
// per-tile digit counts into destinations relative to the leaf (digit-major
// order, tiles in order inside a digit).
__global__ void __launch_bounds__(kLsThreads) k_leaf_scan(const uint32_t* first_tile, const uint32_t* ntiles,
                                                          uint32_t* hist) {
  __shared__ uint32_t tmp[33];
  const uint32_t f = first_tile[blockIdx.x], nt = ntiles[blockIdx.x];
  const uint32_t b = threadIdx.x;
  uint32_t run = 0;
#pragma unroll 8
  for (uint32_t k = 0; k < nt; ++k) {
    uint32_t* h = hist + (size_t)(f + k) * 256 + b;
    const uint32_t v = *h;
    *h = run;
    run += v;
  }
  uint32_t tot;
  const uint32_t base = block_excl_scan(run, tmp, &tot);
#pragma unroll 8
  for (uint32_t k = 0; k < nt; ++k) hist[(size_t)(f + k) * 256 + b] += base;
}

__global__ void __launch_bounds__(kLsThreads) k_leaf_scatter(const uint32_t* src, uint32_t* dst,
                                                             const LeafTile* tiles, int shift,
                                                             const uint32_t* hist) {
  __shared__ uint32_t keys[kLeafBlockMax];
  __shared__ uint32_t whist[kLsWarps][256];
  __shared__ uint32_t dtot[256];
  const LeafTile tl = tiles[blockIdx.x];
  const uint32_t m = min((uint32_t)kLeafBlockMax, tl.count - tl.off);
  const uint32_t* a = src + tl.begin + tl.off;
  for (uint32_t i = threadIdx.x; i < m; i += kLsThreads) keys[i] = a[i];
  __syncthreads();
  uint32_t rank[kLsItems], dig[kLsItems];
  block_rank(keys, m, shift, whist, dtot, rank, dig);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t* hb = hist + (size_t)blockIdx.x * 256;
  uint32_t* out = dst + tl.begin;
#pragma unroll
  for (int j = 0; j < kLsItems; ++j) {
    if (dig[j] == kInvalidDigit) continue;
    const uint32_t idx = (uint32_t)(warp * (32 * kLsItems) + j * 32 + lane);
    const uint32_t pos = hb[dig[j]] + whist[warp][dig[j]] + rank[j];
    if (pos < tl.count) out[pos] = keys[idx];
  }
}

__global__ void k_leaf_copy(const uint32_t* src, uint32_t* dst, const LeafTile* tiles) {
  const LeafTile tl = tiles[blockIdx.x];
  const uint32_t m = min((uint32_t)kLeafBlockMax, tl.count - tl.off);
  for (uint32_t i = threadIdx.x; i < m; i += blockDim.x) dst[tl.begin + tl.off + i] = src[tl.begin + tl.off + i];
}

}  // namespace

void launch_leaf_sort(const TreeDev* trees, const SlotChunks& sc, cudaStream_t st) {
  TraceScope ts(K_LEAF_SORT, st);
  launch_chained(k_leaf_sort, sc.chunks, kLsThreads, 0, st, trees, sc);
}

namespace {

// Leaves of at most kBucketPoints points; those it could not sort go to *rest.
cudaError_t leaf_sort_buckets(const TreeHost& th, const std::vector<uint2>& leaves, std::vector<uint2>* rest,
                              cudaStream_t st) {
  const size_t nl = leaves.size();
  const size_t flags_at = (nl * sizeof(uint2) + 255) & ~(size_t)255;
  if (flags_at + nl * 4 > th.scratch_bytes) {
    rest->insert(rest->end(), leaves.begin(), leaves.end());
    return cudaSuccess;
  }
  uint2* d_leaves = (uint2*)th.scratch;
  uint32_t* d_failed = (uint32_t*)((uint8_t*)th.scratch + flags_at);
  int dev = 0, sms = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(k_leaf_buckets, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBucketSmem)) !=
          cudaSuccess ||
      (e = cudaMemcpyAsync(d_leaves, leaves.data(), nl * sizeof(uint2), cudaMemcpyHostToDevice, st)) != cudaSuccess ||
      (e = cudaMemsetAsync(d_failed, 0, nl * 4, st)) != cudaSuccess)
    return e;
  {
    TraceScope ts(K_LEAF_BUCKETS, st);
    k_leaf_buckets<<<(unsigned)std::min<size_t>(nl, (size_t)sms), kBucketThreads, kBucketSmem, st>>>(
        th.out_perm, d_leaves, (uint32_t)nl, d_failed);
  }
  std::vector<uint32_t> failed(nl);
  if ((e = cudaGetLastError()) != cudaSuccess ||
      (e = cudaMemcpyAsync(failed.data(), d_failed, nl * 4, cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(st)) != cudaSuccess)
    return e;
  for (size_t i = 0; i < nl; ++i)
    if (failed[i]) rest->push_back(leaves[i]);
  return cudaSuccess;
}

}  // namespace

cudaError_t leaf_sort_huge(const TreeHost& th, const std::vector<TermRec>& all, cudaStream_t st) {
  std::vector<uint2> recs, fit;  // begin and count of the leaves
  for (const TermRec& r : all) (r.count <= kBucketPoints ? fit : recs).push_back(make_uint2(r.begin, r.count));
  if (!fit.empty()) {
    const cudaError_t e = leaf_sort_buckets(th, fit, &recs, st);
    if (e != cudaSuccess) return e;
  }
  if (recs.empty()) return cudaSuccess;
  std::vector<LeafTile> tiles;
  std::vector<uint32_t> first, ntiles;
  for (const uint2& r : recs) {
    first.push_back((uint32_t)tiles.size());
    uint32_t k = 0;
    for (uint32_t off = 0; off < r.y; off += kLeafBlockMax, ++k) tiles.push_back(LeafTile{r.x, r.y, off, 0});
    ntiles.push_back(k);
  }
  const size_t nt = tiles.size(), nr = recs.size();
  const size_t need = nt * sizeof(LeafTile) + nt * 256 * 4 + 2 * nr * 4 + 4 * 256;
  if (need > th.scratch_bytes) return cudaErrorMemoryAllocation;
  uint8_t* p = (uint8_t*)th.scratch;
  LeafTile* d_tiles = (LeafTile*)p;
  p += ((nt * sizeof(LeafTile) + 255) & ~(size_t)255);
  uint32_t* d_hist = (uint32_t*)p;
  p += ((nt * 256 * 4 + 255) & ~(size_t)255);
  uint32_t* d_first = (uint32_t*)p;
  uint32_t* d_nt = d_first + nr;
  cudaError_t e;
  if ((e = cudaMemcpyAsync(d_tiles, tiles.data(), nt * sizeof(LeafTile), cudaMemcpyHostToDevice, st)) != cudaSuccess)
    return e;
  if ((e = cudaMemcpyAsync(d_first, first.data(), nr * 4, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
  if ((e = cudaMemcpyAsync(d_nt, ntiles.data(), nr * 4, cudaMemcpyHostToDevice, st)) != cudaSuccess) return e;
  const int digits = index_digits(th.n);
  uint32_t* a = th.out_perm;
  uint32_t* b = th.keys;
  for (int d = 0; d < digits; ++d) {
    { TraceScope ts(K_LEAF_HIST, st); k_leaf_hist<<<(unsigned)nt, kLsThreads, 0, st>>>(a, d_tiles, 8 * d, d_hist); }
    { TraceScope ts(K_LEAF_SCAN, st); k_leaf_scan<<<(unsigned)nr, kLsThreads, 0, st>>>(d_first, d_nt, d_hist); }
    {
      TraceScope ts(K_LEAF_SCATTER, st);
      k_leaf_scatter<<<(unsigned)nt, kLsThreads, 0, st>>>(a, b, d_tiles, 8 * d, d_hist);
    }
    std::swap(a, b);
  }
  if (a != th.out_perm) {
    TraceScope ts(K_LEAF_COPY, st);
    k_leaf_copy<<<(unsigned)nt, kLsThreads, 0, st>>>(a, th.out_perm, d_tiles);
  }
  return cudaGetLastError();
}

}  // namespace kdt
