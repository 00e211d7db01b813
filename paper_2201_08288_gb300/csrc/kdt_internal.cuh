// kdt_internal.cuh -- device-side types and helpers of the CUDA k-d tree build.
//
// The build follows the level structure of the canonical k-d tree (paper,
// Sec. 1 and Sec. 2): level l splits each of its cells along one key
// coordinate, children of heap node h are 2h+1 and 2h+2. Each cell's split is
// combined from per-subset medians (the subsets of Sec. 3.2 / App. C.2); the
// per-subset statistic is the lower median and the combination is the
// count-weighted lower median of those medians.
//
// Layout invariant of the multi-CTA pipeline: inside every cell the points are
// ordered by subset, so each (cell, subset) segment is one contiguous range.
// The root is reordered once by subset (a counting pass; closed form for
// subsets by index mod r; nothing to do for contiguous subsets), and the
// stable two-way partition of every level keeps the order. The medians, the
// splits and the cell sizes do not depend on the order of points inside a
// cell; the one output that does, the order of the permutation inside each
// leaf, is ascending original index in the sequential definition (stable
// partitions of the identity), and a final per-leaf sort restores it.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace kdt {

// ----------------------------------------------------------------- limits

constexpr int kMaxDims = 64;          // d <= 64
constexpr int kMaxSubsets = 4096;     // r <= 4096 on the CUDA path
constexpr int kTile = 2048;           // points per tile of the multi-CTA pipeline
constexpr int kTileRecWords = 2 * kMaxDims + 4;  // words of a tile's record in tile_mm (16-byte aligned)
constexpr int kTileThreads = 256;     // threads of the tile kernels
constexpr int kSelWarpMin = 1024;     // smallest warp_max: sizes the list of CTA-select segments

// status codes (mirror include/kdt.h)
enum : int32_t {
  ST_OK = 0,
  ST_INVALID_ARG = 1,
  ST_NAN_INPUT = 2,
  ST_OOM = 3,
  ST_CUDA = 4,
  ST_CAPACITY = 5,
  ST_TIMEOUT = 6,
  ST_LEVEL_CAP = 7,
  ST_INTERNAL = 9,  // an internal table was inconsistent (reported as a CUDA error)
};

enum : int32_t { KEY_CYCLIC = 0, KEY_WIDEST = 1 };
enum : int32_t { SUB_MOD = 0, SUB_CONTIG = 1, SUB_EXPLICIT = 2 };

// --------------------------------------------------------- data structures

// Everything a kernel needs to know about one tree. Level l reads its points
// from src(l) and the multi-CTA partition writes them to dst(l):
//   src(0) = the root reordered by subset in buf[1] (presorted trees), else
//            the caller's input (perm = identity);
//   src(l>0) = buf[(l-1)&1], dst(l) = buf[l&1].
struct TreeDev {
  int64_t n;
  int32_t d, r, subset_mode, key_rule;
  int32_t depth;       // > 0 depth mode
  int32_t leaf_size;   // leaf mode
  int32_t max_levels;  // leaf mode level cap
  int32_t stall_limit; // d (cyclic) or 1 (widest)
  int32_t sid_bytes;   // explicit mode: 1 or 2
  int32_t small_max;   // cells up to this size finish in the subtree kernel
  int32_t leafsort;    // subsets not in index order: leaves are sorted at the end
  int32_t presorted;   // root reordered by subset into buf[1]; leaves sorted at the end
  uint64_t contig_mul; // contiguous subsets: floor(2^32 r / n)
  const float* x_in;
  const void* sid_in;
  float* xbuf[2];
  uint32_t* pbuf[2];
  uint32_t* root_off;    // [r+1] subset offsets of the root (level 0)
  uint32_t* root_cur;    // [r] subset counts, then fill cursors of the presort
  uint32_t* huge;        // [huge_cap] terminal records too large for one CTA's leaf sort
  uint32_t* huge_count;  // device word
  uint32_t huge_cap;
  int32_t fourier_j;     // > 0: splits by the Fourier-moment estimator with this many harmonics
  int32_t combine_rule;  // 0: count-weighted median of the subset medians; 1: every subset counts once
  int32_t sub_wide;      // small cells run in the subtree kernel's wide shape (else the narrow one)
  uint32_t* out_perm;
  float* out_vals;
  int8_t* out_dims;
  int64_t* out_offs;
  struct TermRec* terms; // terminal cells
  uint32_t term_cap;
  uint32_t pad1;
  uint32_t* term_count;
  int32_t* status;
  int32_t* levels;       // L (max terminal level in leaf mode)
  int32_t* live;         // cells of this tree still waiting to be split (0: the tree is done)
};

constexpr uint32_t kNoRow = 0xffffffffu;

// A cell of the tree: a contiguous position range [begin, begin+count) of its
// tree's current order.
struct alignas(16) Cell {
  uint32_t begin;
  uint32_t count;
  uint32_t heap;
  int32_t tree;
  int8_t level;
  int8_t stall;   // consecutive splits on this path that left the right child empty
  int16_t dim;    // widest-spread key coordinate if already known, else -1
  uint32_t row = kNoRow;  // cells queued for the subtree kernel: row of small_off with the cell's
                          // subset offsets, or kNoRow
  uint32_t tile0 = 0;     // big cells: first of the cell's tiles and segments in the step's tables
  uint32_t seg0 = 0;
};

// A terminal cell (leaf of the real tree); finalize turns these into offsets
// and sentinels below them.
struct TermRec {
  uint32_t begin;
  uint32_t count;
  uint32_t heap;
  int32_t level;
};

// Per-step arrays of the multi-CTA pipeline (one entry per big cell / tile /
// (cell, subset) segment).
struct StepDev {
  const Cell* cells;      // big cells of this step
  uint32_t ncells;              // cells of this step (steps driven by the host)
  const uint32_t* ncells_dev;   // if set: the device word that holds it (steps inside a graph, steps ahead)
  uint32_t ntiles, nseg;        // tiles and segments of this step, or the device words:
  const uint32_t* ntiles_dev;
  const uint32_t* nseg_dev;
  uint32_t bounded;             // the words' values are at most ncells, ntiles and nseg, and seldom much less
  uint32_t tiles_cap, nseg_cap;
  uint2* tiles;           // [ntiles] (cell, offset within cell)
  uint32_t* kdim;         // [ncells] key coordinate
  uint32_t* mkey;         // [ncells] split key
  uint32_t* lcount;       // [ncells] left child size
  uint32_t* tile_mm;      // [ntiles][kTileRecWords] a root's min and max key per coordinate (widest), or a run's sums
  uint32_t* child_mm;     // [ncells][2][kMaxDims][2] per-child min/max keys (widest), reduced
                          // by the scatter with atomics
  uint32_t* seg_w;        // [nseg] points per (cell, subset)
  const uint32_t** seg_key; // [nseg] first key of the segment (raw float bits, key column)
  uint32_t* seg_med;      // [nseg] lower median key
  uint32_t* bigseg;       // [bigseg_cap] segments above warp_max keys
  uint32_t* bigseg_count; // device word
  uint32_t* bigseg_count_next;  // the next step's, cleared by this one
  uint32_t* midseg;       // [midseg_cap] segments of tiny_max+1 .. warp_max keys
  uint32_t* midseg_count; // device word
  uint32_t* midseg_count_next;
  uint32_t few_segs;      // every segment gets a CTA: no lists
  uint32_t wide_segs;     // segments above warp_max get several CTAs (where their cell has room, wide_cell)
  uint32_t* tile_seg;     // [ntiles] first subset offset of the cell at or after the tile's start
  uint32_t* tile_left;    // [ntiles]
  uint32_t* tile_loff;    // [ntiles]
  Cell* next_big;         // children that stay in the multi-CTA pipeline
  unsigned long long* next_big_ctr;   // device: their number (low word) and their segments (high)
  unsigned long long* next_tile_ctr;  // device: their tiles (low) and points (high)
  Cell* small;            // children that finish in the subtree kernel: cells of narrow-shape
                          // trees from the front, of wide-shape trees from the back
  unsigned long long* small_ctr;  // device: cells at the front (low word) and at the back (high:
                                  // small[small_cap - 1 - j])
  uint32_t next_big_cap;
  uint32_t small_cap;
  uint32_t init_small, init_small_w, init_small_points;  // the queue's contents when the step starts
  uint32_t keep_small;        // or what the step before left in it
  uint32_t* small_points;     // points appended to small
  // subset offsets (relative to the cell's begin, r+1 per cell) of this
  // step's cells: rows of off_cur at obase_cur[c]; level-0 cells use their
  // tree's root_off. The scatter fills the rows of the big children.
  const uint32_t* off_cur;
  const uint32_t* obase_cur;  // [ncells]
  uint32_t* off_next;
  uint32_t* obase_next;       // [next_big_cap]
  uint32_t off_cap;
  // subset offsets of cells queued for the subtree kernel (explicit ids, while
  // rows last; other modes follow from the original index, and so does a cell
  // without a row)
  uint32_t* small_off;
  uint32_t* small_off_used;   // device word
  uint32_t small_off_cap;
  uint32_t bigseg_cap;
  // select paths by segment size (kdt_tuning): one thread up to tiny_max keys,
  // a warp's bitonic network up to bitonic_max (at most 128), a warp's brackets up to
  // warp_max, a CTA above
  uint32_t tiny_max, bitonic_max, warp_max;
  uint32_t midseg_cap;
  uint2* crow;                // [ncells][2] (slot, row of off_next) of each big child; (kNoRow, slot in
                              // small) of a child queued for the subtree kernel; else (kNoRow, kNoRow)
  // Sharded build (0 shards: off). The forest's trees 0..shards-1 are the
  // shards of one tree, each owning the subsets s with s % shards == its
  // slot, all at the same level in every step.
  uint32_t shards;
  uint32_t shard_span;        // 2^(levels - 1): entries per shard of shard_idx
  uint32_t* shard_idx;        // [shards][shard_span] step cell of (shard, heap - (2^level - 1)), or kNoRow
  uint32_t* wcount;           // [ncells] points of the cell over all shards (the combine's weight)
  uint32_t* mm_tmp;           // [ncells][2][d][2] children's min / max over all shards
};

// ------------------------------------------------------------- key transform

// Order-preserving map float -> uint32: unsigned comparison of keys equals
// the float order, with -0.0 below +0.0.
__device__ __forceinline__ uint32_t ord_key(float x) {
  uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_float(uint32_t k) {
  uint32_t u = (k & 0x80000000u) ? (k ^ 0x80000000u) : ~k;
  return __uint_as_float(u);
}

__device__ __forceinline__ bool is_nan_bits(float x) {
  return (__float_as_uint(x) & 0x7fffffffu) > 0x7f800000u;
}

// -------------------------------------------------------------- tree views

__device__ __forceinline__ const float* src_cols(const TreeDev& t, int level) {
  return (level == 0 && !t.presorted) ? t.x_in : t.xbuf[(level - 1) & 1];
}
__device__ __forceinline__ const uint32_t* src_perm(const TreeDev& t, int level) {
  return (level == 0 && !t.presorted) ? nullptr : t.pbuf[(level - 1) & 1];
}

__device__ __forceinline__ void set_status(const TreeDev& t, int32_t code) {
  atomicCAS(t.status, ST_OK, code);
}

// Subset of a point from its original index (modes that define it so). For
// contiguous subsets floor(orig r / n) comes from contig_mul = floor(2^32 r /
// n): orig contig_mul / 2^32 falls short of orig r / n by less than 1 (orig <
// 2^32), so its floor is the subset or one below it (a 64-bit division is
// about a hundred instructions here).
__device__ __forceinline__ uint32_t subset_from_orig(const TreeDev& t, uint32_t orig) {
  if (t.subset_mode == SUB_MOD) return orig % (uint32_t)t.r;
  const uint32_t lo = (uint32_t)(((uint64_t)orig * t.contig_mul) >> 32);
  return lo + ((uint64_t)(lo + 1u) * (uint64_t)t.n <= (uint64_t)orig * (uint64_t)t.r ? 1u : 0u);
}

// Subset of the point with original index orig. An explicit id >= r is
// reported as an invalid argument and replaced by 0 so that no table is
// indexed out of range.
__device__ __forceinline__ uint32_t subset_of(const TreeDev& t, uint32_t orig) {
  if (t.subset_mode != SUB_EXPLICIT) return subset_from_orig(t, orig);
  const uint32_t s = t.sid_bytes == 1 ? (uint32_t)__ldg((const uint8_t*)t.sid_in + orig)
                                      : (uint32_t)__ldg((const uint16_t*)t.sid_in + orig);
  if (s >= (uint32_t)t.r) {
    set_status(t, ST_INVALID_ARG);
    return 0;
  }
  return s;
}

// The first statement of a kernel that launch_chained launches: every thread
// waits until the kernel before it in the stream has ended and its writes are
// visible.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// Cells of a step: the host's count, or the device word a graph-driven step
// reads (clamped to the capacity of the cell lists).
__device__ __forceinline__ uint32_t ncells_of(const StepDev& s) {
  return s.ncells_dev ? min(*s.ncells_dev, s.next_big_cap) : s.ncells;
}

__device__ __forceinline__ uint32_t ntiles_of(const StepDev& s) {
  return s.ntiles_dev ? min(*s.ntiles_dev, s.tiles_cap) : s.ntiles;
}
__device__ __forceinline__ uint32_t nseg_of(const StepDev& s) {
  return s.nseg_dev ? min(*s.nseg_dev, s.nseg_cap) : s.nseg;
}
__host__ __device__ __forceinline__ uint32_t tiles_of(uint32_t count) {
  return count / (uint32_t)kTile + (count % (uint32_t)kTile != 0u ? 1u : 0u);
}

// Points of step cell c whose split is being combined: its own count, or in a
// sharded build the cell's count over all shards.
__device__ __forceinline__ uint32_t cell_weight(const StepDev& s, uint32_t c, const Cell& cell) {
  return s.shards ? s.wcount[c] : cell.count;
}

// Terminal test for a cell about to be processed at `level` (reading R8 in
// leaf mode; empty cells and the last level in depth mode).
__device__ __forceinline__ bool is_terminal(const TreeDev& t, uint32_t count, int level, int stall) {
  if (t.depth > 0) return count == 0 || level >= t.depth;
  return count <= (uint32_t)t.leaf_size || stall >= t.stall_limit;
}

__device__ __forceinline__ void record_terminal(const TreeDev& t, uint32_t begin, uint32_t count,
                                                uint32_t heap, int level) {
  uint32_t slot = atomicAdd(t.term_count, 1u);
  if (slot < t.term_cap) {
    t.terms[slot] = TermRec{begin, count, heap, level};
  } else {
    set_status(t, ST_CAPACITY);
  }
  atomicMax(t.levels, level);
}

// ------------------------------------------------------------ warp helpers

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

__device__ __forceinline__ uint32_t warp_sum(uint32_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Given a 256-bin histogram in shared memory (counts or weights) and a
// 0-based target rank, the whole warp finds the digit whose bin holds that
// rank; returns the digit and, in *below, the total of the lower bins.
__device__ __forceinline__ uint32_t warp_find_digit(const uint32_t* hist, uint32_t rank,
                                                    uint32_t* below) {
  const int lane = threadIdx.x & 31;
  uint32_t local[8];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    local[i] = hist[lane * 8 + i];
    s += local[i];
  }
  uint32_t incl = warp_incl_scan(s);
  uint32_t excl = incl - s;
  // the lane whose range [excl, incl) contains rank
  unsigned ballot = __ballot_sync(0xffffffffu, rank >= excl && rank < incl);
  int owner = ballot ? __ffs(ballot) - 1 : 31;
  uint32_t digit = 0, b = 0;
  if (lane == owner) {
    uint32_t acc = excl;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (rank < acc + local[i]) {
        digit = lane * 8 + i;
        b = acc;
        break;
      }
      acc += local[i];
    }
  }
  digit = __shfl_sync(0xffffffffu, digit, owner);
  *below = __shfl_sync(0xffffffffu, b, owner);
  return digit;
}

// Like warp_find_digit for a histogram of nb = 2^bits bins (1 <= bits <= 8).
__device__ __forceinline__ uint32_t warp_find_digit_n(const uint32_t* hist, uint32_t nb, uint32_t rank,
                                                      uint32_t* below) {
  const int lane = threadIdx.x & 31;
  const uint32_t per = nb >= 32u ? nb / 32u : 1u;
  const uint32_t first = lane * per;
  uint32_t local[8];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    local[i] = ((uint32_t)i < per && first + i < nb) ? hist[first + i] : 0u;
    s += local[i];
  }
  const uint32_t incl = warp_incl_scan(s);
  const uint32_t excl = incl - s;
  const unsigned ballot = __ballot_sync(0xffffffffu, rank >= excl && rank < incl);
  const int owner = ballot ? __ffs(ballot) - 1 : 31;
  uint32_t digit = 0, b = 0;
  if (lane == owner) {
    uint32_t acc = excl;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if ((uint32_t)i < per && rank < acc + local[i]) {
        digit = first + i;
        b = acc;
        break;
      }
      acc += local[i];
    }
  }
  digit = __shfl_sync(0xffffffffu, digit, owner);
  *below = __shfl_sync(0xffffffffu, b, owner);
  return digit;
}

// Exact key of 0-based weighted rank `rank` among cnt items (key_of(j),
// w_of(j)), j < cnt, one warp: the smallest key m whose items with key <= m
// weigh more than `rank`. MSD radix select over the bits where the keys
// differ (the common prefix of their min and max is known from the start, so
// no pass is spent on bits every key shares), 8-bit digits, histogram `hist`
// of 256 words owned by the warp.
template <bool kUnit = false, class KeyOf, class WOf, class ValidOf>
__device__ uint32_t warp_weighted_select(uint32_t cnt, uint32_t rank, uint32_t* hist, KeyOf key_of, WOf w_of,
                                         ValidOf valid_of) {
  const int lane = threadIdx.x & 31;
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (uint32_t j = lane; j < cnt; j += 32)
    if (valid_of(j)) {
      const uint32_t k = key_of(j);
      lo = min(lo, k);
      hi = max(hi, k);
    }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  if (lo >= hi) return lo;
  int rem = 32 - __clz(lo ^ hi);  // low bits still unknown
  uint32_t prefix = rem == 32 ? 0u : (lo & ~((1u << rem) - 1u));
  while (rem > 0) {
    const int bits = rem < 8 ? rem : 8;
    const int shift = rem - bits;
    const uint32_t nb = 1u << bits;
    const uint32_t hmask = rem == 32 ? 0u : ~((1u << rem) - 1u);
    for (uint32_t i = lane; i < nb; i += 32) hist[i] = 0;
    __syncwarp();
    for (uint32_t j = lane; j < cnt; j += 32) {
      if (!valid_of(j)) continue;
      const uint32_t k = key_of(j);
      if ((k & hmask) == prefix) atomicAdd(&hist[(k >> shift) & (nb - 1u)], kUnit ? 1u : w_of(j));
    }
    __syncwarp();
    uint32_t below;
    const uint32_t digit = warp_find_digit_n(hist, nb, rank, &below);
    rank -= below;
    prefix |= digit << shift;
    rem = shift;
    __syncwarp();
  }
  return prefix;
}

template <bool kUnit = false, class KeyOf, class WOf>
__device__ uint32_t warp_weighted_select(uint32_t cnt, uint32_t rank, uint32_t* hist, KeyOf key_of, WOf w_of) {
  return warp_weighted_select<kUnit>(cnt, rank, hist, key_of, w_of, [](uint32_t) { return true; });
}

// Lower median of 1 <= w <= 32K keys (key_of(e), e < w) by one warp, element e
// = k * 32 + lane in register k of a lane. The keys are padded to N = 32K with
// the smallest and the largest key so that the median has rank N/2 - 1
// (padding keys equal to a real key would not change the element at that
// rank); the bitonic network runs its stages up to size N/2 only, which
// leaves the first half ascending and the second descending: a bitonic
// sequence whose half-cleaner holds the N/2 smallest keys, the largest of
// which (over the warp) is the median.
template <int K, class KeyOf>
__device__ __forceinline__ uint32_t warp_bitonic_median(KeyOf key_of, uint32_t w) {
  static_assert(K >= 2 && (K & (K - 1)) == 0, "K: a power of two of at least 2");
  const int lane = threadIdx.x & 31;
  constexpr int N = 32 * K;
  const uint32_t zeros_end = w + (uint32_t)(N / 2 - 1) - (w - 1u) / 2u;  // [w, zeros_end) hold 0
  uint32_t v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t e = (uint32_t)(k * 32 + lane);
    v[k] = e < w ? key_of(e) : (e < zeros_end ? 0u : 0xffffffffu);
  }
#pragma unroll
  for (int size = 2; size <= N / 2; size <<= 1) {
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
  uint32_t m = 0u;
#pragma unroll
  for (int k = 0; k < K / 2; ++k) m = max(m, min(v[k], v[k + K / 2]));
  return __reduce_max_sync(0xffffffffu, m);
}

// Block-wide exclusive scan of one value per thread; returns the exclusive
// prefix and writes the block total. `tmp` holds 33 words.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* tmp, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  uint32_t incl = warp_incl_scan(v);
  if (lane == 31) tmp[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nwarps ? tmp[lane] : 0u;
    uint32_t wi = warp_incl_scan(w);
    if (lane < nwarps) tmp[lane] = wi - w;
    if (lane == nwarps - 1) tmp[32] = wi;
  }
  __syncthreads();
  uint32_t r = tmp[warp] + incl - v;
  *total = tmp[32];
  __syncthreads();
  return r;
}

}  // namespace kdt
