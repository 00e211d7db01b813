// kdt_step.cu -- one level of the multi-CTA pipeline for cells too large to
// finish in shared memory.
//
// For every big cell c of the step (paper, Sec. 2: a level splits each of its
// cells along the key coordinate t at a median):
//   0. (roots only) the points are reordered by subset (counting pass, or
//      closed form for subsets by index mod r), so that every (cell, subset)
//      segment is contiguous from then on;
//   1. key coordinate: cyclic (Sec. 1) or widest range (Sec. 1, Friedman
//      rule; computed for the root here, for every other cell by the parent's
//      scatter, which reduces each child's per-coordinate min and max while it
//      moves the columns);
//   2. per (cell, subset) segment (the subsets of Sec. 3.2 / App. C.2): its
//      position range, from the cell's subset offsets;
//   3. per segment: the exact lower median, read in place from the key column
//      (by size: a network, brackets or a radix select);
//   4. per cell: the count-weighted lower median of the segment medians;
//   5. children sizes from per-tile counts and a per-cell scan of them; the
//      children are classified (terminal / small / big) before the move;
//   6. stable partition of all d columns and the permutation around the split
//      (key <= split to the left); the scatter also writes the big children's
//      subset offsets.
// Work is split into tiles of kTile points of one cell; a thread owns kItems
// points of a tile (strided by the block size, so every load is coalesced)
// and issues all of its loads before it uses any of them.
#include <algorithm>

#include "kdt_internal.cuh"
#include "kdt_launch.h"
#include "kdt_ptx.cuh"
#include "kdt_runs.h"
#include "kdt_trace.h"

namespace kdt {

namespace {

constexpr int kItems = kTile / kTileThreads;
constexpr int kWarps = kTileThreads / 32;
constexpr int kPsGroup = 2;                       // tiles per block of the root presort
constexpr int kPsPoints = kPsGroup * kTile;
constexpr int kPsThreads = 512;
constexpr int kPsItems = kPsPoints / kPsThreads;
constexpr uint32_t kPsHole = 0xffffu;             // a place of the sorted group that holds no point
// Places of a group sorted by r subsets (at most one empty place per subset of
// two or more points), and its shared memory (a word and a u16 subset per
// place).
__host__ __device__ constexpr uint32_t ps_places(uint32_t r) { return kPsPoints + (r < kPsPoints / 2u ? r : kPsPoints / 2u); }
constexpr size_t ps_smem_bytes(uint32_t r) { return (size_t)((ps_places(r) + 7u) & ~7u) * 6; }

__device__ __forceinline__ bool tile_of(const StepDev& s, uint32_t tile, uint2* out) {
  if (tile >= ntiles_of(s)) return false;
  *out = s.tiles[tile];
  return true;
}

// ---------------------------------------------------------------- roots

// One warp per cell of a step with roots, before their presort: tile list
// entries (the presort's kernels walk all tiles); zeroed subset counts of a
// presorted root, and (widest spread, coordinate not known yet) the identities
// in its first tile's min / max record, which the presort's groups reduce into.
__device__ __forceinline__ void tiles_cell(const TreeDev* trees, const StepDev& s, uint32_t c) {
  const uint32_t lane = threadIdx.x & 31u;
  const Cell cell = s.cells[c];
  const uint32_t tb = cell.tile0, nt = tiles_of(cell.count);
  for (uint32_t j = lane; j < nt; j += 32u) s.tiles[tb + j] = make_uint2(c, j * (uint32_t)kTile);
  if (cell.level != 0) return;
  const TreeDev& t = trees[cell.tree];
  if (t.presorted) {
    for (uint32_t j = lane; j < (uint32_t)t.r; j += 32u) t.root_cur[j] = 0;
    if (t.key_rule == KEY_WIDEST && cell.dim < 0 && nt > 0u)
      for (uint32_t j = lane; j < 2u * (uint32_t)t.d; j += 32u)
        s.tile_mm[(size_t)tb * kTileRecWords + j] = (j & 1) ? 0u : 0xffffffffu;
  }
}

__global__ void k_tiles(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  const uint32_t wpb = blockDim.x >> 5;
  for (uint32_t c = blockIdx.x * wpb + (threadIdx.x >> 5); c < nc; c += gridDim.x * wpb) tiles_cell(trees, s, c);
}

// ------------------------------------------------------ root presort

__device__ __forceinline__ bool presort_tile(const TreeDev* trees, const StepDev& s, uint32_t tile, uint2* tl,
                                             Cell* cell) {
  if (!tile_of(s, tile, tl)) return false;
  *cell = s.cells[tl->x];
  return cell->level == 0 && trees[cell->tree].presorted;
}

// Points per subset of every presorted root with explicit subset ids. Each
// CTA counts a contiguous range of tiles into a shared histogram and adds it
// to the root's totals (root_cur) when the range moves to another tree and at
// its end.
__global__ void __launch_bounds__(kTileThreads) k_ps_count(const TreeDev* trees, StepDev s) {
  chain_wait();
  __shared__ uint32_t hist[kMaxSubsets];
  const uint32_t ntiles = ntiles_of(s);
  const uint32_t t_begin = (uint32_t)(((uint64_t)blockIdx.x * ntiles) / gridDim.x);
  const uint32_t t_end = (uint32_t)(((uint64_t)(blockIdx.x + 1) * ntiles) / gridDim.x);
  int32_t cur = -1;  // tree whose counts hist holds
  auto flush = [&]() {
    __syncthreads();
    if (cur >= 0) {
      const TreeDev& t = trees[cur];
      for (int j = threadIdx.x; j < t.r; j += blockDim.x)
        if (hist[j]) atomicAdd(&t.root_cur[j], hist[j]);
    }
    __syncthreads();
  };
  for (uint32_t tile = t_begin; tile < t_end; ++tile) {
    const uint2 tl = s.tiles[tile];
    const Cell cell = s.cells[tl.x];
    const TreeDev& t = trees[cell.tree];
    if (cell.level != 0 || !t.presorted || t.subset_mode != SUB_EXPLICIT) continue;
    if (cell.tree != cur) {
      flush();
      for (int j = threadIdx.x; j < t.r; j += blockDim.x) hist[j] = 0;
      cur = cell.tree;
      __syncthreads();
    }
    const uint32_t end = min(tl.y + (uint32_t)kTile, cell.count);
    uint32_t sub[kItems];
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
      const uint32_t i = tl.y + threadIdx.x + q * kTileThreads;
      sub[q] = i < end ? subset_of(t, i) : 0xffffffffu;
    }
#pragma unroll
    for (int q = 0; q < kItems; ++q)
      if (sub[q] != 0xffffffffu) atomic_add_shared(&hist[sub[q]], 1u);
  }
  flush();
}

// One CTA per root cell: its subset offsets (r + 1 entries). Explicit ids:
// exclusive scan of the counts (which also become the fill cursors); subsets
// by index mod r: r_j = floor(n/r) + [j < n mod r] points each; contiguous
// subsets (already in order): subset j starts at ceil(j n / r).
__device__ __forceinline__ void ps_offsets_cell(const TreeDev* trees, const StepDev& s, uint32_t c) {
  __shared__ uint32_t tmp[33];
  const Cell cell = s.cells[c];
  if (cell.level != 0) return;
  const TreeDev& t = trees[cell.tree];
  const uint32_t r = (uint32_t)t.r, n = cell.count;
  if (t.subset_mode == SUB_EXPLICIT) {
    uint32_t run = 0;
    for (uint32_t j0 = 0; j0 < r; j0 += blockDim.x) {
      const uint32_t j = j0 + threadIdx.x;
      const uint32_t v = j < r ? t.root_cur[j] : 0u;
      uint32_t tot;
      const uint32_t ex = block_excl_scan(v, tmp, &tot);
      if (j < r) {
        t.root_off[j] = run + ex;
        t.root_cur[j] = run + ex;
      }
      run += tot;
    }
    if (threadIdx.x == 0) {
      t.root_off[r] = run;
      if (run != n) set_status(t, ST_INTERNAL);
    }
  } else if (t.subset_mode == SUB_MOD) {
    const uint32_t q = n / r, rem = n % r;
    for (uint32_t j = threadIdx.x; j <= r; j += blockDim.x) t.root_off[j] = j * q + min(j, rem);
  } else {
    for (uint32_t j = threadIdx.x; j <= r; j += blockDim.x)
      t.root_off[j] = (uint32_t)(((uint64_t)j * n + r - 1) / r);
  }
}

__global__ void k_ps_offsets(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    ps_offsets_cell(trees, s, c);
    __syncthreads();  // the cell's shared memory is free for the next one
  }
}

// Per group of kPsGroup consecutive tiles of a presorted root (kPsPoints
// points): every point gets a rank inside its subset within the group
// (shared-memory counter; order inside a subset is immaterial, see
// kdt_internal.cuh), each subset of the group reserves a run of its place in
// subset order (explicit ids: from the fill cursors; index mod r: closed
// form), and every column passes through shared memory in subset order so
// that the stores are contiguous runs of about kPsPoints / r points. With
// subsets by index mod r a warp's 32 points go to 32 consecutive subsets, and
// at an even distance of kPsPoints / r places they share banks (64 subsets:
// all 32 in one), so there a subset takes an odd number of places (one is left
// empty where its count is even): 50,000,021 points in 3 coordinates, 64
// subsets, 0.50 ms against 1.16. Explicit ids spread over the banks by
// themselves; the empty places only cost (2^27 points in 8: 3.25 ms against
// 2.91).
__global__ void __launch_bounds__(kPsThreads) k_ps_move(const TreeDev* trees, StepDev s) {
  chain_wait();
  uint2 tl;
  Cell cell;
  if (!presort_tile(trees, s, blockIdx.x, &tl, &cell)) return;
  const TreeDev& t = trees[cell.tree];
  // widest spread: the group's min / max key per coordinate go by atomics into
  // the record of the root's first tile, the other tiles' records hold the
  // identities
  const bool want_mm = t.key_rule == KEY_WIDEST && cell.dim < 0;
  if ((tl.y / (uint32_t)kTile) % (uint32_t)kPsGroup != 0u) {  // the group's first tile runs it
    if (want_mm)
      for (int j = threadIdx.x; j < 2 * t.d; j += blockDim.x)
        s.tile_mm[(size_t)blockIdx.x * kTileRecWords + j] = (j & 1) ? 0u : 0xffffffffu;
    return;
  }
  extern __shared__ __align__(16) uint32_t ps_buf[];  // a word per place, then a u16 subset per place
  uint16_t* lsub = (uint16_t*)(ps_buf + ((ps_places((uint32_t)t.r) + 7u) & ~7u));
  __shared__ uint32_t loff[kMaxSubsets];   // counts, then local offsets
  __shared__ uint32_t gbase[kMaxSubsets];  // global start of each subset's run
  __shared__ uint32_t tmp[33];
  __shared__ uint32_t gmm[kMaxDims][2];
  const uint32_t r = (uint32_t)t.r, i0 = tl.y, end = min(i0 + (uint32_t)kPsPoints, cell.count);
  const bool expl = t.subset_mode == SUB_EXPLICIT;
  for (uint32_t j = threadIdx.x; j < r; j += kPsThreads) loff[j] = 0;
  for (int j = threadIdx.x; j < 2 * t.d; j += kPsThreads) gmm[j / 2][j & 1] = (j & 1) ? 0u : 0xffffffffu;
  __syncthreads();
  uint32_t sub[kPsItems], lp[kPsItems];
#pragma unroll
  for (int q = 0; q < kPsItems; ++q) {
    const uint32_t i = i0 + threadIdx.x + q * kPsThreads;
    sub[q] = i < end ? subset_of(t, i) : 0xffffffffu;
  }
#pragma unroll
  for (int q = 0; q < kPsItems; ++q) lp[q] = sub[q] != 0xffffffffu ? atomic_add_shared(&loff[sub[q]], 1u) : 0u;
  __syncthreads();
  uint32_t run = 0;
  for (uint32_t j0 = 0; j0 < r; j0 += kPsThreads) {
    const uint32_t j = j0 + threadIdx.x;
    const uint32_t c = j < r ? loff[j] : 0u;
    if (j < r) {
      if (expl)
        gbase[j] = c ? atomicAdd(&t.root_cur[j], c) : 0u;
      else  // indices below i0 in subset j: floor(i0 / r) + [j < i0 mod r]
        gbase[j] = t.root_off[j] + i0 / r + (j < i0 % r ? 1u : 0u);
    }
    uint32_t tot;
    const uint32_t odd = c + (!expl && c != 0u && (c & 1u) == 0u ? 1u : 0u);
    const uint32_t ex = block_excl_scan(odd, tmp, &tot);
    if (j < r) {
      loff[j] = run + ex;
      if (odd != c) lsub[run + ex + c] = (uint16_t)kPsHole;
    }
    run += tot;
  }
  const uint32_t m = run;  // places in use
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kPsItems; ++q)
    if (sub[q] != 0xffffffffu) {
      lp[q] += loff[sub[q]];
      lsub[lp[q]] = (uint16_t)sub[q];
    }
  __syncthreads();
  // place a value per point in subset order, then store the runs
  auto pass = [&](auto value_of, auto store) {
#pragma unroll
    for (int q = 0; q < kPsItems; ++q)
      if (sub[q] != 0xffffffffu) ps_buf[lp[q]] = value_of(q);
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < m; j += kPsThreads) {
      const uint32_t sj = lsub[j];
      if (sj == kPsHole) continue;
      const uint32_t dst = gbase[sj] + (j - loff[sj]);
      if (dst < cell.count) store(dst, ps_buf[j]); else set_status(t, ST_INTERNAL);
    }
    __syncthreads();
  };
  const int64_t n = t.n;
  // each column's loads are issued before the previous column's passes
  uint32_t x[kPsItems], xn[kPsItems];
  auto load = [&](int l, uint32_t (&v)[kPsItems]) {
    const uint32_t* X = (const uint32_t*)(t.x_in + (int64_t)l * n);
#pragma unroll
    for (int q = 0; q < kPsItems; ++q) {
      const uint32_t i = i0 + threadIdx.x + q * kPsThreads;
      v[q] = i < end ? __ldg(X + i) : 0u;
    }
  };
  // the input's NaN check (the scatter of a presorted root skips it): a NaN
  // key lies above +inf's or below -inf's
  bool nan = false;
  load(0, x);
  for (int l = 0; l < t.d; ++l) {
    if (l + 1 < t.d) load(l + 1, xn);
    if (want_mm) {
      uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
      for (int q = 0; q < kPsItems; ++q)
        if (sub[q] != 0xffffffffu) {
          const uint32_t k = ord_key(__uint_as_float(x[q]));
          lo = min(lo, k);
          hi = max(hi, k);
        }
      nan |= hi > 0xff800000u || lo < 0x007fffffu;
      lo = __reduce_min_sync(0xffffffffu, lo);
      hi = __reduce_max_sync(0xffffffffu, hi);
      if ((threadIdx.x & 31) == 0) {
        atomic_min_shared(&gmm[l][0], lo);
        atomic_max_shared(&gmm[l][1], hi);
      }
    } else {
#pragma unroll
      for (int q = 0; q < kPsItems; ++q) nan |= sub[q] != 0xffffffffu && is_nan_bits(__uint_as_float(x[q]));
    }
    uint32_t* out = (uint32_t*)(t.xbuf[1] + (int64_t)l * n);
    pass([&](int q) { return x[q]; }, [&](uint32_t dst, uint32_t v) { out[dst] = v; });
#pragma unroll
    for (int q = 0; q < kPsItems; ++q) x[q] = xn[q];
  }
  if (nan) set_status(t, ST_NAN_INPUT);
  if (want_mm) {  // the passes' barriers order the shared-memory reductions before this
    // into the root's first tile record (identities set by k_tiles); this
    // tile's own record, if another, holds the identities
    const uint32_t tb = cell.tile0;
    for (int j = threadIdx.x; j < 2 * t.d; j += kPsThreads) {
      uint32_t* acc = &s.tile_mm[(size_t)tb * kTileRecWords + j];
      if (j & 1) atomicMax(acc, gmm[j / 2][1]); else atomicMin(acc, gmm[j / 2][0]);
      if (blockIdx.x != tb)
        s.tile_mm[(size_t)blockIdx.x * kTileRecWords + j] = (j & 1) ? 0u : 0xffffffffu;
    }
  }
  pass([&](int q) { return i0 + threadIdx.x + q * kPsThreads; },
       [&](uint32_t dst, uint32_t v) { t.pbuf[1][dst] = v; });
}

// ------------------------------------------------------- widest spread

// Per tile and coordinate of a cell whose key coordinate is not known yet
// (the root): min and max key, reduced per cell by k_pick_dim.
__global__ void __launch_bounds__(kTileThreads) k_minmax(const TreeDev* trees, StepDev s) {
  chain_wait();
  uint2 tl;
  if (!tile_of(s, blockIdx.x, &tl)) return;
  const Cell cell = s.cells[tl.x];
  const TreeDev& t = trees[cell.tree];
  if (t.key_rule != KEY_WIDEST || cell.dim >= 0 || t.presorted) return;  // presorted: from k_ps_move
  __shared__ uint32_t red[2][kWarps];
  const float* X = src_cols(t, cell.level) + cell.begin;
  const int64_t n = t.n;
  const uint32_t end = min(tl.y + (uint32_t)kTile, cell.count);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool nan = false;
  for (int l = 0; l < t.d; ++l) {
    float x[kItems];
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
      const uint32_t i = tl.y + threadIdx.x + q * kTileThreads;
      x[q] = i < end ? X[(int64_t)l * n + i] : 0.0f;
    }
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
      const uint32_t i = tl.y + threadIdx.x + q * kTileThreads;
      if (i < end) {
        nan |= is_nan_bits(x[q]);
        const uint32_t k = ord_key(x[q]);
        lo = min(lo, k);
        hi = max(hi, k);
      }
    }
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane == 0) {
      red[0][warp] = lo;
      red[1][warp] = hi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < kWarps; ++w) {
        lo = min(lo, red[0][w]);
        hi = max(hi, red[1][w]);
      }
      s.tile_mm[(size_t)blockIdx.x * kTileRecWords + 2 * l + 0] = lo;
      s.tile_mm[(size_t)blockIdx.x * kTileRecWords + 2 * l + 1] = hi;
    }
    __syncthreads();
  }
  if (nan) set_status(t, ST_NAN_INPUT);
}

// Range of a coordinate from its min and max keys: (double)max - (double)min,
// 0 when both are the same key.
__device__ __forceinline__ double key_range(uint32_t lo, uint32_t hi) {
  return (lo == hi) ? 0.0 : (double)key_float(hi) - (double)key_float(lo);
}

// One CTA per cell with an unknown widest coordinate: reduce the tile
// partials and pick the coordinate of largest range (lowest on ties). Every
// thread walks its own tiles, eight coordinates at a time (four 16-byte loads
// per tile: a tile's record holds min, max of each coordinate in turn).
__device__ __forceinline__ void pick_dim_cell(const TreeDev* trees, const StepDev& s, uint32_t c) {
  const Cell cell = s.cells[c];
  const TreeDev& t = trees[cell.tree];
  if (t.key_rule != KEY_WIDEST || cell.dim >= 0) return;
  __shared__ uint32_t slo[kMaxDims], shi[kMaxDims];
  for (int l = threadIdx.x; l < t.d; l += blockDim.x) {
    slo[l] = 0xffffffffu;
    shi[l] = 0u;
  }
  __syncthreads();
  // the roots of a sharded build's shards are parts of one root: every one
  // of them reduces the tiles of all
  const uint32_t tb = s.shards ? 0u : cell.tile0;
  // a presorted root's presort gathered its min / max in its first tile's
  // record; other roots' are spread over their tiles
  const uint32_t te = s.shards ? ntiles_of(s) : tb + (t.presorted ? 1u : tiles_of(cell.count));
  const int lane = threadIdx.x & 31;
  for (int c0 = 0; c0 < t.d; c0 += 8) {
    const int nc = min(8, t.d - c0);
    uint32_t lo[8], hi[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      lo[q] = 0xffffffffu;
      hi[q] = 0u;
    }
    for (uint32_t j = tb + threadIdx.x; j < te; j += blockDim.x) {
      // 16-byte aligned: a record is a multiple of 4 words, c0 of 8
      const uint4* p = (const uint4*)(s.tile_mm + (size_t)j * kTileRecWords + 2 * c0);
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (2 * h >= nc) break;
        const uint4 v = p[h];
        lo[2 * h] = min(lo[2 * h], v.x);
        hi[2 * h] = max(hi[2 * h], v.y);
        lo[2 * h + 1] = min(lo[2 * h + 1], v.z);
        hi[2 * h + 1] = max(hi[2 * h + 1], v.w);
      }
    }
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (q < nc) {
        const uint32_t l2 = __reduce_min_sync(0xffffffffu, lo[q]);
        const uint32_t h2 = __reduce_max_sync(0xffffffffu, hi[q]);
        if (lane == 0) {
          atomic_min_shared(&slo[c0 + q], l2);
          atomic_max_shared(&shi[c0 + q], h2);
        }
      }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int best = 0;
    double best_range = -1.0;
    for (int l = 0; l < t.d; ++l) {
      const double range = key_range(slo[l], shi[l]);
      if (range > best_range) {
        best_range = range;
        best = l;
      }
    }
    s.kdim[c] = (uint32_t)best;
  }
}

__global__ void __launch_bounds__(1024) k_pick_dim(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    pick_dim_cell(trees, s, c);
    __syncthreads();  // the cell's shared memory is free for the next one
  }
}

// ------------------------------------------------------------ segments

// Key column of a cell (raw float bits; ord_key is applied on every load).
__device__ __forceinline__ const uint32_t* key_column(const TreeDev& t, const Cell& cell, uint32_t dim) {
  return (const uint32_t*)(src_cols(t, cell.level) + (int64_t)dim * t.n);
}

__device__ __forceinline__ uint32_t kload(const uint32_t* p) { return ord_key(__uint_as_float(__ldg(p))); }


// Words that a segment of several CTAs keeps while its median is sought: a
// histogram, then its state (key bits found, rank left, CTAs that are done).
// They lie in the part of the next level's first column that the cell's
// scatter will overwrite, so a cell has room for them or takes one CTA per
// segment.
constexpr uint32_t kWideBins = 2048, kWideWords = kWideBins + 4;
__device__ __forceinline__ bool wide_cell(const TreeDev& t, const Cell& cell) {
  return (uint64_t)t.r * kWideWords <= (uint64_t)cell.count;
}
__device__ __forceinline__ uint32_t* wide_words(const TreeDev& t, const Cell& cell, uint32_t j) {
  return (uint32_t*)t.xbuf[cell.level & 1] + cell.begin + (size_t)j * kWideWords;
}

// A group of `gt` threads per cell (after a root's presort and key
// coordinate): the cell's tile list entries and key coordinate; size and first
// key of every (cell, subset) segment from the cell's subset offsets, and the
// lists of segments for the warp and CTA selects; for each of the cell's
// tiles, the first segment start in it (the scatter turns the starts in a tile
// into the children's). Offsets are clamped to the cell, so a damaged table
// cannot send a later kernel outside it (it is reported instead). Where a
// cell's tiles and segments start in the step's tables was settled when its
// parent was classified, so no scan over the cells is needed.
__device__ __forceinline__ void open_cell(const TreeDev* trees, const StepDev& s, uint32_t c, uint32_t tid,
                                          uint32_t gt) {
  const Cell cell = s.cells[c];
  const TreeDev& t = trees[cell.tree];
  const uint32_t tb = cell.tile0, nt = tiles_of(cell.count);
  for (uint32_t k = tid; k < nt; k += gt) s.tiles[tb + k] = make_uint2(c, k * (uint32_t)kTile);
  uint32_t dim;
  if (t.key_rule == KEY_CYCLIC)
    dim = (uint32_t)(cell.level % t.d);
  else
    dim = cell.dim >= 0 ? (uint32_t)cell.dim : s.kdim[c];  // (a widest root's was picked before)
  if (tid == 0) s.kdim[c] = dim;
  if (t.fourier_j) return;  // no segments
  const uint32_t r = (uint32_t)t.r;
  const uint32_t* off = cell.level == 0 ? t.root_off : s.off_cur + s.obase_cur[c];
  const uint32_t g0 = cell.seg0;
  const uint32_t* kc = key_column(t, cell, dim) + cell.begin;
  if (tid == 0 && (off[0] != 0u || off[r] != cell.count)) set_status(t, ST_INTERNAL);
  // tiles that start in (off[j], off[j + 1]] have start j + 1 as their first
  // (the first tile, at 0, has start 0); with fewer subsets than threads
  // several threads share a segment's tiles
  if (tid == 0 && nt > 0u) s.tile_seg[tb] = 0;
  if (nt > 1u) {
    const uint32_t per = max(1u, gt / r);
    for (uint32_t q = tid; q < r * per; q += gt) {
      const uint32_t j = q / per, a = min(off[j], cell.count), b = min(off[j + 1], cell.count);
      for (uint32_t k = a / (uint32_t)kTile + 1u + q % per; k < nt && k * (uint32_t)kTile <= b; k += per)
        s.tile_seg[tb + k] = j + 1u;
    }
  }
  const bool wide = s.wide_segs && wide_cell(t, cell);
  for (uint32_t j = tid; j < r; j += gt) {
    const uint32_t a = min(off[j], cell.count), b = min(off[j + 1], cell.count);
    if (b < a) set_status(t, ST_INTERNAL);
    const uint32_t w = b >= a ? b - a : 0u;
    s.seg_key[g0 + j] = kc + a;
    s.seg_w[g0 + j] = w;
    if (s.few_segs || (wide && w > s.warp_max)) continue;
    if (w > s.warp_max) {
      const uint32_t k = atomicAdd(s.bigseg_count, 1u);
      if (k < s.bigseg_cap) s.bigseg[k] = g0 + j; else set_status(t, ST_INTERNAL);
    } else if (w > s.tiny_max) {
      const uint32_t k = atomicAdd(s.midseg_count, 1u);
      if (k < s.midseg_cap) s.midseg[k] = g0 + j; else set_status(t, ST_INTERNAL);
    }
  }
}

// The first kernel over a step's cells; `gt` divides the CTA. It also sets the
// counters that the step's later kernels, and the next step's first, append to.
// (Scanning the cells' tiles and segments first took two more launches, one of
// them a single CTA: 135 us for the six steps of a build of 65,536 points, 50
// now.)
__global__ void __launch_bounds__(256) k_cells(const TreeDev* trees, StepDev s, uint32_t gt) {
  chain_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *s.next_big_ctr = 0ull;
    *s.next_tile_ctr = 0ull;
    if (!s.keep_small) {
      *s.small_ctr = (unsigned long long)s.init_small | ((unsigned long long)s.init_small_w << 32);
      *s.small_points = s.init_small_points;
      *s.small_off_used = 0;
    }
    *s.bigseg_count_next = 0;
    *s.midseg_count_next = 0;
  }
  const uint32_t nc = ncells_of(s);
  const uint32_t per = blockDim.x / gt, sub = threadIdx.x / gt, tid = threadIdx.x % gt;
  for (uint32_t c = blockIdx.x * per + sub; c < nc; c += gridDim.x * per) open_cell(trees, s, c, tid, gt);
}

// ------------------------------------------------------------ selection

// Batcher's odd-even merge sort of v[0, M) ascending, M a power of two. In
// the round of merge width 2p and distance k, position x is compared with
// x + k when x lies in an even block of k positions counted from k mod p and
// both lie in one block of 2p; every comparator is fixed at compile time.
template <int M>
__device__ __forceinline__ void oddeven_sort(uint32_t (&v)[M]) {
#pragma unroll
  for (int p = 1; p < M; p <<= 1)
#pragma unroll
    for (int k = p; k >= 1; k >>= 1)
#pragma unroll
      for (int x = 0; x < M; ++x) {
        const int j0 = k % p;
        if (x >= j0 && ((x - j0) / k) % 2 == 0 && x + k < M && x / (2 * p) == (x + k) / (2 * p)) {
          const uint32_t a = v[x], b = v[x + k];
          v[x] = min(a, b);
          v[x + k] = max(a, b);
        }
      }
}

// Lower median (rank (w-1)/2) of a segment of 1 <= w <= 2M keys by one
// thread. The keys are padded to 2M: M - 1 - (w-1)/2 copies of the smallest
// key 0, the rest the largest key ~0, so that the median has rank M - 1 among
// the 2M (padding keys equal to a real key would not change the element at
// that rank). Both halves are sorted; A ascending followed by B reversed is
// bitonic, so min(A[i], B[M-1-i]) over i are the M smallest of the 2M, and
// the largest of them is the element of rank M - 1.
template <int M>
__device__ __forceinline__ uint32_t thread_lower_median(const uint32_t* keys, uint32_t w) {
  const uint32_t zeros_end = w + (uint32_t)(M - 1) - (w - 1u) / 2u;  // [w, zeros_end) hold 0
  uint32_t a[M], b[M];
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const uint32_t e = (uint32_t)i, f = (uint32_t)(i + M);
    a[i] = e < w ? kload(keys + e) : (e < zeros_end ? 0u : 0xffffffffu);
    b[i] = f < w ? kload(keys + f) : (f < zeros_end ? 0u : 0xffffffffu);
  }
  oddeven_sort<M>(a);
  oddeven_sort<M>(b);
  uint32_t med = 0u;
#pragma unroll
  for (int i = 0; i < M; ++i) med = max(med, min(a[i], b[M - 1 - i]));
  return med;
}

// One thread per segment of at most tiny_max <= 64 points (the
// threads stride over the segments of the step). The network's size is
// chosen per warp, by the warp's largest segment, so a warp never runs two.
// Five CTAs per SM by a register bound (48 registers): the path waits on its
// loads, and the extra warps hide that better than keeping the larger
// networks in registers does (they spill about 300 bytes per thread to local
// memory; measured faster than four or six CTAs per SM).
__global__ void __launch_bounds__(256, 5) k_select_tiny(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nseg = nseg_of(s);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t g0 = blockIdx.x * blockDim.x + (threadIdx.x & ~31u); g0 < nseg; g0 += stride) {
    const uint32_t g = g0 + lane;
    uint32_t w = g < nseg ? s.seg_w[g] : 0u;
    if (w > s.tiny_max) w = 0u;
    const uint32_t wmax = __reduce_max_sync(0xffffffffu, w);
    if (wmax == 0u) continue;
    const uint32_t* keys = w ? s.seg_key[g] : nullptr;
    uint32_t med;
    if (wmax <= 8u)
      med = thread_lower_median<4>(keys, w);
    else if (wmax <= 16u)
      med = thread_lower_median<8>(keys, w);
    else if (wmax <= 32u)
      med = thread_lower_median<16>(keys, w);
    else
      med = thread_lower_median<32>(keys, w);
    if (w) s.seg_med[g] = med;
  }
}

// State of a warp's radix select: the key bits found so far (`prefix`, all
// bits above `rem`) and the rank still sought below them.
struct RadixState {
  uint32_t prefix, rank;
  int rem;
};

__device__ __forceinline__ bool radix_start(uint32_t lo, uint32_t hi, uint32_t rank, RadixState* st) {
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  st->rank = rank;
  if (lo >= hi) {
    st->prefix = lo;
    st->rem = 0;
    return false;
  }
  st->rem = 32 - __clz(lo ^ hi);
  st->prefix = st->rem == 32 ? 0u : (lo & ~((1u << st->rem) - 1u));
  return true;
}

// The key of the given rank among w by one warp: MSD radix select with
// 8-bit digits over the bits where the keys differ (histogram of 256 words
// owned by the warp), the keys read on every pass from global memory (raw
// float bits, turned into order keys), 8 loads per lane issued together, or
// from a shared-memory copy (order keys already).
template <bool kGlobal>
__device__ uint32_t warp_select_stream(const uint32_t* keys, uint32_t w, uint32_t rank, uint32_t* hist) {
  constexpr int U = 8;
  const int lane = threadIdx.x & 31;
  auto load = [&](uint32_t i) -> uint32_t { return kGlobal ? kload(keys + i) : keys[i]; };
  uint32_t lo = 0xffffffffu, hi = 0u;
  for (uint32_t b0 = 0; b0 < w; b0 += 32 * U) {
    uint32_t x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t i = b0 + (uint32_t)(u * 32 + lane);
      x[u] = i < w ? load(i) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (b0 + (uint32_t)(u * 32 + lane) < w) {
        lo = min(lo, x[u]);
        hi = max(hi, x[u]);
      }
  }
  RadixState st;
  if (!radix_start(lo, hi, rank, &st)) return st.prefix;
  while (st.rem > 0) {
    const int bits = st.rem < 8 ? st.rem : 8, shift = st.rem - bits;
    const uint32_t nb = 1u << bits, hmask = st.rem == 32 ? 0u : ~((1u << st.rem) - 1u);
    for (uint32_t i = lane; i < nb; i += 32) hist[i] = 0;
    __syncwarp();
    for (uint32_t b0 = 0; b0 < w; b0 += 32 * U) {
      uint32_t x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t i = b0 + (uint32_t)(u * 32 + lane);
        x[u] = i < w ? load(i) : 0u;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (b0 + (uint32_t)(u * 32 + lane) < w && (x[u] & hmask) == st.prefix)
          atomicAdd(&hist[(x[u] >> shift) & (nb - 1u)], 1u);
    }
    __syncwarp();
    uint32_t below;
    const uint32_t digit = warp_find_digit_n(hist, nb, st.rank, &below);
    st.rank -= below;
    st.prefix |= digit << shift;
    st.rem = shift;
    __syncwarp();
  }
  return st.prefix;
}

// Ascending sort of 32 K keys, element k * 32 + lane in register k of a lane:
// the bitonic network of warp_bitonic_median with its last stages.
template <int K>
__device__ __forceinline__ void warp_sort(uint32_t (&v)[K]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32 * K; size <<= 1)
#pragma unroll
    for (int j = size >> 1; j > 0; j >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const bool asc = ((k * 32 + lane) & size) == 0;
        if (j >= 32) {
          const int kk = k ^ (j >> 5);
          if (k < kk) {
            const uint32_t lo = min(v[k], v[kk]), hi = max(v[k], v[kk]);
            v[k] = asc ? lo : hi;
            v[kk] = asc ? hi : lo;
          }
        } else {
          const uint32_t o = __shfl_xor_sync(0xffffffffu, v[k], j);
          v[k] = (((lane & j) == 0) == asc) ? min(v[k], o) : max(v[k], o);
        }
      }
}

// Keys between which the one of rank m of c is expected: those `under` below
// and `over` above its place in a sorted sample of 32 K, taken at even distances.
template <int K, class Get>
__device__ __forceinline__ void warp_bracket(Get get, uint32_t c, uint32_t m, int under, int over, uint32_t* a,
                                             uint32_t* b) {
  const int lane = threadIdx.x & 31;
  uint32_t v[K];
#pragma unroll
  for (int k = 0; k < K; ++k) v[k] = get(((uint32_t)(k * 32 + lane) * c) / (32u * K));
  warp_sort<K>(v);
  const int at = (int)((m * 32u * K) / c), i = at - under, j = at + over;
  uint32_t x = 0u, y = 0xffffffffu;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t p = __shfl_sync(0xffffffffu, v[k], i & 31), q = __shfl_sync(0xffffffffu, v[k], j & 31);
    if (i >= 0 && (i >> 5) == k) x = p;
    if ((j >> 5) == k) y = q;
  }
  *a = x;
  *b = y;
}

// One pass over c keys, U rows of 32 loaded together: how many lie below a, how
// many in [a, b], and those (up to cap of them, in their order) to dst.
template <int U, class Get>
__device__ __forceinline__ void warp_bracket_pass(Get get, uint32_t c, uint32_t a, uint32_t b, uint32_t* dst,
                                                  uint32_t cap, uint32_t* below, uint32_t* inside) {
  const uint32_t lane = threadIdx.x & 31u, width = b - a;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t l = 0, n = 0;
  for (uint32_t b0 = 0; b0 < c; b0 += 32 * U) {
    uint32_t x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t i = b0 + (uint32_t)(u * 32) + lane;
      x[u] = i < c ? get(i) : 0u;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool real = b0 + (uint32_t)(u * 32) + lane < c, in = real && x[u] - a <= width;
      l += real && x[u] < a ? 1u : 0u;
      const unsigned who = __ballot_sync(0xffffffffu, in);
      const uint32_t pos = n + (uint32_t)__popc(who & lt);
      if (in && pos < cap) dst[pos] = x[u];
      n += (uint32_t)__popc(who);
    }
  }
  *below = __reduce_add_sync(0xffffffffu, l);
  *inside = n;
  __syncwarp();
}

// A pass for the key of rank m, and where the sample misled (about one time in
// fifty) another over the side that holds it. On return [a, b] holds it, at
// rank m among the *inside keys there.
template <int U, class Get>
__device__ __forceinline__ void warp_bracket_narrow(Get get, uint32_t c, uint32_t* m, uint32_t* a, uint32_t* b,
                                                    uint32_t* dst, uint32_t cap, uint32_t* inside) {
  uint32_t below;
  warp_bracket_pass<U>(get, c, *a, *b, dst, cap, &below, inside);
  if (*m < below || *m - below >= *inside) {
    if (*m < below) {
      *b = *a - 1u;
      *a = 0u;
    } else {
      *a = *b + 1u;
      *b = 0xffffffffu;
    }
    warp_bracket_pass<U>(get, c, *a, *b, dst, cap, &below, inside);
  }
  *m -= below;
}

// Lower median of w > 32 keys by one warp: a small sorted sample gives two keys
// that the median lies between, and one pass keeps what does (two fifths for a
// sample of 32, a fifth for 128); again among those, until a sort of 32 ends it.
// Many equal keys may not thin out: what is left then goes to the radix select,
// as does what finds no room. (The radix select, for all segments above 256 keys,
// took up to four passes with a shared-memory atomic per key, 92 instructions per
// 32 keys of 1024 against 71 here; the bitonic network of 256 keys, for those
// above 128, 28 rounds of shuffles of 8 registers. 2^27 points, 256 subsets: the
// small selects of a build 3.75 -> 2.82 ms; 2^24 points, 64 subsets: 590 -> 497
// us; 50,000,021 points, 64 subsets: 428 -> 284. Columns per lane instead of a
// dense list, or a first pass that compares floats, took 519 and 530 us where
// this takes 497. A CTA's select by brackets lost to its radix select, whose
// later passes hit L1 and L2: 56 against 41 us for 2^24 keys in segments of 8192.)
constexpr uint32_t kBracketA = 1024, kBracketB = 512;  // room after odd and after even passes
template <class Get>
__device__ uint32_t warp_bracket_median(const uint32_t* keys, Get get, uint32_t w, uint32_t* buf) {
  const uint32_t lane = threadIdx.x & 31u;
  uint32_t a, b, c, m = (w - 1u) / 2u;
  if (w > 1024u)
    warp_bracket<4>(get, w, m, 12, 13, &a, &b);
  else
    warp_bracket<1>(get, w, m, 6, 7, &a, &b);
  warp_bracket_narrow<8>(get, w, &m, &a, &b, buf, kBracketA, &c);
  if (a == b) return a;
  if (c > kBracketA) return warp_select_stream<true>(keys, w, (w - 1u) / 2u, buf);
  uint32_t *src = buf, *dst = buf + kBracketA, cap = kBracketB;
  while (c > 32u) {
    auto kept = [&](uint32_t i) { return src[i]; };
    warp_bracket<1>(kept, c, m, 6, 7, &a, &b);
    const uint32_t m0 = m;
    uint32_t n;
    warp_bracket_narrow<4>(kept, c, &m, &a, &b, dst, cap, &n);
    if (a == b) return a;
    if (n > cap || 8u * n > 7u * c) return warp_select_stream<false>(src, c, m0, dst);
    c = n;
    uint32_t* const t = src;
    src = dst;
    dst = t;
    cap = kBracketB;
  }
  uint32_t v[1] = {lane < c ? src[lane] : 0xffffffffu};
  warp_sort<1>(v);
  return __shfl_sync(0xffffffffu, v[0], (int)m);
}

// One warp per listed segment of tiny_max+1 .. warp_max points: up to
// bitonic_max keys sorted in registers, larger ones by brackets.
__global__ void __launch_bounds__(256) k_select_small(const TreeDev* trees, StepDev s) {
  chain_wait();
  __shared__ uint32_t buf[8][kBracketA + kBracketB];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cnt = min(*s.midseg_count, s.midseg_cap);
  for (uint32_t j = blockIdx.x * 8u + (uint32_t)warp; j < cnt; j += gridDim.x * 8u) {
    const uint32_t g = s.midseg[j];
    const uint32_t w = s.seg_w[g];
    const uint32_t* keys = s.seg_key[g];
    auto key_of = [&](uint32_t e) { return kload(keys + e); };
    uint32_t med;
    if (w <= s.bitonic_max && w <= 64u)
      med = warp_bitonic_median<2>(key_of, w);
    else if (w <= s.bitonic_max && w <= 128u)
      med = warp_bitonic_median<4>(key_of, w);
    else
      med = warp_bracket_median(keys, key_of, w, buf[warp]);
    if (lane == 0) s.seg_med[g] = med;
    __syncwarp();
  }
}

// add(raw bits) for each of w keys by a CTA: 16 bytes at a time, four loads of
// a thread in flight (the unaligned head and tail by single words).
template <int kThreads, class Add>
__device__ __forceinline__ void cta_for_keys(const uint32_t* keys, uint32_t w, Add add) {
  const uint32_t head = min(w, (4u - (uint32_t)(((uintptr_t)keys >> 2) & 3u)) & 3u);
  const uint4* kv = (const uint4*)(keys + head);  // 16-byte aligned
  const uint32_t nv = (w - head) >> 2, tail0 = head + nv * 4u;
  uint32_t v = threadIdx.x;
  for (; v + 3 * kThreads < nv; v += 4 * kThreads) {
    uint4 q[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) q[u] = __ldg(kv + v + u * kThreads);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      add(q[u].x);
      add(q[u].y);
      add(q[u].z);
      add(q[u].w);
    }
  }
  for (; v < nv; v += kThreads) {
    const uint4 q = __ldg(kv + v);
    add(q.x);
    add(q.y);
    add(q.z);
    add(q.w);
  }
  if (threadIdx.x < head) add(__ldg(keys + threadIdx.x));
  if (threadIdx.x < w - tail0) add(__ldg(keys + tail0 + threadIdx.x));
}

// Lower median of w >= 1 keys by a CTA of kThreads: MSD radix select with
// kBits-bit digits (8: four passes, one histogram
// per warp, which suits the few bins that the top digits of clustered data
// fall into; 11: three passes over a CTA-wide 2048-bin histogram), keys read
// from global memory 16 bytes at a time (the unaligned head and tail of the
// segment by single words).
template <int kThreads, int kBits>
__device__ __forceinline__ uint32_t cta_lower_median(const uint32_t* keys, uint32_t w) {
  constexpr int kW = kThreads / 32;
  constexpr bool kWarpHist = kBits == 8;
  constexpr int kBins = 1 << kBits;
  constexpr int kHist = kWarpHist ? kW * kBins : kBins;
  constexpr int kPer = kBins >= kThreads ? kBins / kThreads : 1;  // bins per thread in the digit search
  __shared__ uint32_t hist[kHist];
  __shared__ uint32_t tot_w[kWarpHist ? kBins : 1];
  __shared__ uint32_t tmp[33];
  __shared__ uint32_t bcast[2];
  const int warp = threadIdx.x >> 5;
  uint32_t* tot = kWarpHist ? tot_w : hist;
  uint32_t rank = (w - 1) / 2, prefix = 0;
  for (int top = 32; top > 0;) {  // bits [top, 32) are known
    const int bits = top < kBits ? top : kBits, shift = top - bits;
    const uint32_t mask = top == 32 ? 0u : ~((1u << top) - 1u), nb = 1u << bits;
    for (int i = threadIdx.x; i < kHist; i += kThreads) hist[i] = 0;
    __syncthreads();
    uint32_t* wh = kWarpHist ? hist + warp * kBins : hist;
    auto add = [&](uint32_t u) {
      const uint32_t k = ord_key(__uint_as_float(u));
      if ((k & mask) == prefix) atomicAdd(&wh[(k >> shift) & (nb - 1u)], 1u);
    };
    cta_for_keys<kThreads>(keys, w, add);
    __syncthreads();
    if (kWarpHist) {
      for (int b = threadIdx.x; b < kBins; b += kThreads) {
        uint32_t sum = 0;
#pragma unroll
        for (int q = 0; q < kW; ++q) sum += hist[q * kBins + b];
        tot[b] = sum;
      }
      __syncthreads();
    }
    // the bin holding `rank`: each thread scans kPer consecutive bins
    const uint32_t first = (uint32_t)threadIdx.x * kPer;
    uint32_t loc[kPer], sum = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      loc[q] = first + q < nb ? tot[first + q] : 0u;
      sum += loc[q];
    }
    uint32_t all;
    const uint32_t ex = block_excl_scan(sum, tmp, &all);
    if (rank >= ex && rank < ex + sum) {
      uint32_t acc = ex;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        if (rank < acc + loc[q]) {
          bcast[0] = first + q;
          bcast[1] = acc;
          break;
        }
        acc += loc[q];
      }
    }
    __syncthreads();
    rank -= bcast[1];
    prefix |= bcast[0] << shift;
    top = shift;
    __syncthreads();
  }
  return prefix;
}

// CTAs stride over the listed segments above the warp-select size.
template <int kThreads, int kBits>
__global__ void __launch_bounds__(kThreads) k_select_big(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t cnt = min(*s.bigseg_count, s.bigseg_cap);
  for (uint32_t jb = blockIdx.x; jb < cnt; jb += gridDim.x) {
    const uint32_t g = s.bigseg[jb];
    const uint32_t med = cta_lower_median<kThreads, kBits>(s.seg_key[g], s.seg_w[g]);
    if (threadIdx.x == 0) s.seg_med[g] = med;
  }
}

// Steps of few segments: a CTA for every one of them, whatever its size, in
// one launch instead of three.
__global__ void __launch_bounds__(256) k_select_all(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nseg = nseg_of(s);
  for (uint32_t g = blockIdx.x; g < nseg; g += gridDim.x) {
    const uint32_t w = s.seg_w[g];
    if (w == 0u) continue;
    const uint32_t med = cta_lower_median<256, 11>(s.seg_key[g], w);
    if (threadIdx.x == 0) s.seg_med[g] = med;
  }
}

// Steps of few, large segments (the first levels, and every tree of few
// subsets): a segment's keys are spread over gridDim.x CTAs. Three launches,
// 11 key bits each (10 in the last): every CTA counts the digits of its part
// in shared memory and adds them to the segment's histogram; the last one to
// finish finds the digit that holds the rank and clears the histogram for the
// next launch. One segment of 20,000,003 keys (a tree of one subset, depth 10):
// kdt_build 18.6 -> 2.7 ms, where one CTA had read it three times.
constexpr int kWideThreads = 512;

__device__ __forceinline__ bool wide_segment(const TreeDev* trees, const StepDev& s, uint32_t* g, uint32_t* w,
                                             uint32_t** words) {
  if (blockIdx.z >= ncells_of(s)) return false;  // a step ahead: fewer cells than its launches allow for
  const Cell cell = s.cells[blockIdx.z];
  const TreeDev& t = trees[cell.tree];
  if (blockIdx.y >= (uint32_t)t.r || !wide_cell(t, cell)) return false;
  *g = cell.seg0 + blockIdx.y;
  *w = s.seg_w[*g];
  *words = wide_words(t, cell, blockIdx.y);
  return *w > s.warp_max;
}

__global__ void __launch_bounds__(kWideThreads) k_wide_clear(const TreeDev* trees, StepDev s) {
  chain_wait();
  uint32_t g, w, *H;
  if (!wide_segment(trees, s, &g, &w, &H)) return;
  for (uint32_t i = threadIdx.x; i < kWideWords; i += kWideThreads) H[i] = i == kWideBins + 1u ? (w - 1u) / 2u : 0u;
}

__global__ void __launch_bounds__(kWideThreads) k_wide_pass(const TreeDev* trees, StepDev s, int top) {
  chain_wait();
  __shared__ uint32_t hist[kWideBins];
  __shared__ uint32_t tmp[33];
  __shared__ bool last;
  constexpr int kPer = kWideBins / kWideThreads;
  uint32_t g, w, *H;
  if (!wide_segment(trees, s, &g, &w, &H)) return;
  uint32_t* state = H + kWideBins;
  const int bits = min(top, 11), shift = top - bits;
  const uint32_t mask = top == 32 ? 0u : ~((1u << top) - 1u), nb = 1u << bits;
  const uint32_t prefix = state[0];
  for (int i = threadIdx.x; i < (int)kWideBins; i += kWideThreads) hist[i] = 0;
  __syncthreads();
  const uint32_t a = (uint32_t)(((uint64_t)w * blockIdx.x) / gridDim.x);
  const uint32_t b = (uint32_t)(((uint64_t)w * (blockIdx.x + 1u)) / gridDim.x);
  cta_for_keys<kWideThreads>(s.seg_key[g] + a, b - a, [&](uint32_t u) {
    const uint32_t k = ord_key(__uint_as_float(u));
    if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & (nb - 1u)], 1u);
  });
  __syncthreads();
  for (int i = threadIdx.x; i < (int)kWideBins; i += kWideThreads)
    if (hist[i]) atomicAdd(&H[i], hist[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&state[2], 1u) == gridDim.x - 1u;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const uint32_t rank = state[1];  // written before this launch
  uint32_t loc[kPer], sum = 0;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const uint32_t i = threadIdx.x * kPer + q;
    loc[q] = __ldcg(H + i);
    H[i] = 0u;
    sum += loc[q];
  }
  uint32_t all;
  uint32_t acc = block_excl_scan(sum, tmp, &all);
  if (rank >= acc && rank < acc + sum) {  // one thread
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if (rank < acc + loc[q]) {
        const uint32_t key = prefix | ((threadIdx.x * kPer + q) << shift);
        state[0] = key;
        state[1] = rank - acc;
        if (shift == 0) s.seg_med[g] = key;
        break;
      }
      acc += loc[q];
    }
  }
  if (threadIdx.x == 0) state[2] = 0u;
}

// One CTA per cell: count-weighted lower median of the segment medians: the
// smallest median m whose segments with median <= m hold at least
// ceil(W/2) of the W points (weighted 8-bit MSD radix select).
__device__ __forceinline__ void combine_cell(const TreeDev* trees, const StepDev& s, uint32_t c) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t bcast[2];
  const Cell cell = s.cells[c];
  const TreeDev& t = trees[cell.tree];
  const int r = t.r;
  const uint32_t g0 = cell.seg0;
  const bool unit = t.combine_rule == 1;  // every non-empty subset counts once
  uint32_t rank = (cell_weight(s, c, cell) - 1) / 2, prefix = 0, mask = 0;
  if (unit) {  // rank (m - 1) / 2 among the m non-empty segments
    if (threadIdx.x == 0) bcast[0] = 0;
    __syncthreads();
    uint32_t m = 0;
    for (int j = threadIdx.x; j < r; j += blockDim.x) m += s.seg_w[g0 + j] != 0u;
    m = warp_sum(m);
    if ((threadIdx.x & 31) == 0) atomicAdd(&bcast[0], m);
    __syncthreads();
    rank = (bcast[0] - 1u) / 2u;
    __syncthreads();
  }
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    for (int j = threadIdx.x; j < r; j += blockDim.x) {
      const uint32_t w = s.seg_w[g0 + j];
      if (!w) continue;
      const uint32_t k = s.seg_med[g0 + j];
      if ((k & mask) == prefix) atomicAdd(&hist[(k >> shift) & 255u], unit ? 1u : w);
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      uint32_t below;
      const uint32_t digit = warp_find_digit(hist, rank, &below);
      if (threadIdx.x == 0) {
        bcast[0] = digit;
        bcast[1] = below;
      }
    }
    __syncthreads();
    rank -= bcast[1];
    prefix |= bcast[0] << shift;
    mask |= 255u << shift;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    s.mkey[c] = prefix;
    t.out_vals[cell.heap] = key_float(prefix);
    t.out_dims[cell.heap] = (int8_t)s.kdim[c];
  }
}

__global__ void __launch_bounds__(256) k_combine(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    combine_cell(trees, s, c);
    __syncthreads();  // the cell's shared memory is free for the next one
  }
}

// One warp per cell (steps with many cells): the same weighted lower median
// by the warp radix select, which starts at the first bit where the cell's
// segment medians differ.
__device__ __forceinline__ void combine_warp_cell(const TreeDev* trees, const StepDev& s, uint32_t c) {
  __shared__ uint32_t hist[8][256];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Cell cell = s.cells[c];
  const TreeDev& t = trees[cell.tree];
  const uint32_t g0 = cell.seg0;
  const uint32_t* med = s.seg_med + g0;
  const uint32_t* wt = s.seg_w + g0;
  const bool unit = t.combine_rule == 1;  // every non-empty subset counts once
  uint32_t rank = (cell_weight(s, c, cell) - 1) / 2;
  if (unit) {
    uint32_t nz = 0;
    for (uint32_t j = lane; j < (uint32_t)t.r; j += 32) nz += wt[j] != 0u;
    rank = (warp_sum(nz) - 1u) / 2u;
  }
  const uint32_t m = warp_weighted_select(
      (uint32_t)t.r, rank, hist[warp], [&](uint32_t j) { return med[j]; },
      [&](uint32_t j) { return unit ? 1u : wt[j]; }, [&](uint32_t j) { return wt[j] != 0u; });
  if (lane == 0) {
    s.mkey[c] = m;
    t.out_vals[cell.heap] = key_float(m);
    t.out_dims[cell.heap] = (int8_t)s.kdim[c];
  }
}

__global__ void __launch_bounds__(256, 1) k_combine_warp(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x * 8u + (threadIdx.x >> 5); c < nc; c += gridDim.x * 8u) combine_warp_cell(trees, s, c);
}

// ------------------------------------------- the paper's estimator (Sec. 3)

constexpr int kFourierTerms = 2 * KDT_FOURIER_MAX_J + 1;
static_assert(kFourierTerms * 2 <= kTileRecWords, "a tile's sums fit its record");

// The sums over a cell's points of the basis terms of Lemma 1 on its key
// coordinate, c_0 = 1, c_{2j-1} = cos((2j-1)x), c_{2j} = sin((2j-1)x) for
// j = 1..J (the additive statistics of Sec. 3.2). The kernel is persistent: CTA k
// takes the runs (kdt_runs.h) that start among the tiles [k T / G, (k+1) T / G) of
// the step (T tiles, G CTAs). Each thread holds 8 points of a tile and runs the odd
// harmonics for all of them at once (h(k+2) = 2 cos(2x) h(k) - h(k-2), from one
// sincosf per point), adding each harmonic's terms in float, then over the warp by
// a shuffle tree in float (double arithmetic is scarce on this GPU); the CTA adds
// the warps' sums in double in a fixed order into a running total per term,
// written to the record of the run's first tile when the run ends. The split
// kernel adds a cell's run records in an order that their number fixes, so the
// result does not depend on scheduling. A coordinate outside (0,1) is reported.
__global__ void __launch_bounds__(256, 2) k_fourier_moments(const TreeDev* trees, StepDev s) {
  chain_wait();
  constexpr int kPer = kTile / 256;
  __shared__ float red[8][kFourierTerms];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t ntiles = ntiles_of(s);
  auto start_from = [&](uint32_t tile) {
    if (tile >= ntiles) return ntiles;
    const uint2 tl = s.tiles[tile];
    const Cell cell = s.cells[tl.x];
    return run_start(tile, tl.y / (uint32_t)kTile, tiles_of(cell.count), run_tiles(tiles_of((uint32_t)trees[cell.tree].n)));
  };
  const uint32_t t_begin = start_from((uint32_t)(((uint64_t)blockIdx.x * ntiles) / gridDim.x));
  const uint32_t t_end = start_from((uint32_t)(((uint64_t)(blockIdx.x + 1) * ntiles) / gridDim.x));
  // a tile's record, cell and this thread's points (loaded one tile ahead)
  struct Ahead {
    uint2 tl;
    int32_t tree;
    uint32_t end, run;
    float x[kPer];
  };
  auto fetch = [&](uint32_t tile, Ahead& a) {
    a.tl = s.tiles[tile];
    const Cell cell = s.cells[a.tl.x];
    const TreeDev& t = trees[cell.tree];
    const float* X = (const float*)key_column(t, cell, s.kdim[a.tl.x]) + cell.begin;
    a.tree = cell.tree;
    a.run = run_tiles(tiles_of((uint32_t)t.n));
    a.end = min(a.tl.y + (uint32_t)kTile, cell.count);
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const uint32_t i = a.tl.y + threadIdx.x + 256u * q;
      a.x[q] = i < a.end ? __ldg(X + i) : 0.5f;
    }
  };
  double run = 0.0;  // thread j: term j of the current run
  uint32_t run_first = t_begin;
  Ahead cur, nxt;
  if (t_begin < t_end) fetch(t_begin, cur);
  for (uint32_t tile = t_begin; tile < t_end; ++tile) {
    if (tile + 1 < t_end) fetch(tile + 1, nxt);  // in flight while this tile is summed
    const TreeDev& t = trees[cur.tree];
    const int J = t.fourier_j;
    float c2[kPer], cp[kPer], sp[kPer], cc[kPer], sc[kPer];
    bool outside = false, nan = false;
    uint32_t cnt = 0;
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const uint32_t i = cur.tl.y + threadIdx.x + 256u * q;
      const bool ok = i < cur.end;
      const float x = cur.x[q];
      nan |= ok && x != x;
      outside |= ok && !(x > 0.f && x < 1.f);
      float sx, cx;
      sincosf(x, &sx, &cx);
      const float w = ok ? 1.f : 0.f;  // a missing point adds nothing
      c2[q] = 2.f * (cx * cx - sx * sx);
      cp[q] = w * cx;  // harmonic -1
      sp[q] = -w * sx;
      cc[q] = w * cx;  // harmonic 1
      sc[q] = w * sx;
      cnt += ok ? 1u : 0u;
    }
    if (outside) set_status(t, nan ? ST_NAN_INPUT : ST_INVALID_ARG);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) red[warp][0] = (float)cnt;
    for (int k = 1; k <= J; ++k) {
      float ac = 0.f, as = 0.f;
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        ac += cc[q];
        as += sc[q];
        const float cn = fmaf(c2[q], cc[q], -cp[q]), sn = fmaf(c2[q], sc[q], -sp[q]);
        cp[q] = cc[q];
        sp[q] = sc[q];
        cc[q] = cn;
        sc[q] = sn;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        ac += __shfl_down_sync(0xffffffffu, ac, o);
        as += __shfl_down_sync(0xffffffffu, as, o);
      }
      if (lane == 0) {
        red[warp][2 * k - 1] = ac;
        red[warp][2 * k] = as;
      }
    }
    __syncthreads();
    if ((int)threadIdx.x <= 2 * J) {
      double v = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) v += (double)red[w][threadIdx.x];
      run += v;
    }
    // the run ends here: write its record
    if (tile + 1 == t_end || nxt.tl.x != cur.tl.x ||
        (cur.tl.y / (uint32_t)kTile + 1u) % cur.run == 0u) {
      if ((int)threadIdx.x <= 2 * J) ((double*)(s.tile_mm + (size_t)run_first * kTileRecWords))[threadIdx.x] = run;
      run = 0.0;
      run_first = tile + 1;
    }
    __syncthreads();
    cur = nxt;
  }
}

// Per cell, one CTA: the cell's sums C_j (its run records, every G-th by one of G
// threads per term, then the G partial sums in order), its bounds (a, b) on its key coordinate (the splits of its
// ancestors on that coordinate, (0,1) at the root), and the root of Eq.
// (kd:eq:b) by 60 bisection steps in double on (a, b) of F(m) = 1_J(a, m) -
// 1_J(m, b) = sum_j C_j (g_j(a, m) - g_j(m, b)), with g_j of Lemma 1: the term
// of j = 0 is (1(b<1) - 1(a>0)) / 2, of j = 2k-1 q (2 sin(Km) - 1(a>0) sin(Ka)
// - 1(b<1) sin(Kb)) and of j = 2k q (1(a>0) cos(Ka) + 1(b<1) cos(Kb) - 2
// cos(Km)), K = 2k-1, q = 2 / (pi K). The lower end moves up while F < 0; the
// split is the last midpoint rounded to float, and a point goes left when its
// coordinate is <= it. The harmonics of the midpoint are evaluated in float
// (their error moves the root by about 1e-7 of the cell's width), the sums in
// double.
// Double arithmetic bounds this: an SM's quarter finishes one warp-wide double
// operation in 64 cycles and starts the next after about as many (conversions
// to and from double too), and a step is a chain of a product, two sums per
// term, a tree of five sums and a midpoint. A warp per cell that took the 60
// steps one by one, each lane with its own terms and its own conversions, was
// 165 us per level whatever the cells. So the CTA takes three steps at once:
//   the seven midpoints that the three can meet (candidate w stands for the
//     path that w's bits below its highest one spell, 0 where F >= 0) were
//     formed during the round before, for each of its eight outcomes, by warps
//     without terms of their own;
//   a thread per candidate and harmonic evaluates both of its terms; what can
//     be had exactly from integers (K m rounded to float, the waves widened to
//     double) is;
//   half a warp per candidate adds its terms, in the order and tree of the
//     one-warp form, so the splits are the same bits; the signs are the round's
//     outcome.
// The records are loaded eight at a time per thread, so that a root's thousands
// wait for few round trips; their sums are split over as many threads as there are,
// since a double addition occupies a quarter of an SM for 64 cycles. 4,000,037
// points, J = 16, ten levels: 0.50 ms per build; 0.58 with the records staged 32 at
// a time and one thread per term, 1.86 with a warp per cell.
constexpr int kFsSteps = 3, kFsCand = 1 << kFsSteps;  // candidates 1 .. kFsCand - 1
constexpr int kFsThreads = 256;
constexpr int kFsParts = 8;  // partial sums of a term at most
static_assert((kFsCand - 1) * KDT_FOURIER_MAX_J <= kFsThreads, "a thread per candidate and harmonic");
static_assert((kFsCand - 1) * 16 <= kFsThreads && 4 * KDT_FOURIER_MAX_J <= kFsThreads, "threads for the other parts");

// (float)(k * x) for 0 < x < 4 and an odd k below 64, k * x rounded to double
// first: the product of x's 53 bits and k's 6 in 64, rounded to nearest even
// twice.
__device__ __forceinline__ float product_float(uint32_t k, double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)(u >> 52);
  if (ex < 1023 - 96) return (float)((double)k * x);  // (zero, or near the float's smallest numbers)
  unsigned long long p = ((u & 0xfffffffffffffull) | 0x10000000000000ull) * k;  // below 2^59
  auto round_off = [&](int n) {  // p / 2^n to nearest even, n >= 1
    const unsigned long long half = 1ull << (n - 1), rest = p & ((1ull << n) - 1ull);
    p >>= n;
    p += rest > half || (rest == half && (p & 1ull)) ? 1ull : 0ull;
  };
  int e = ex - 1075;  // the value is p 2^e
  const int over = 64 - __clzll((long long)p) - 53;
  if (over > 0) {
    round_off(over);
    e += over;
  }
  const int more = 64 - __clzll((long long)p) - 24;  // p has 53 or 54 bits
  round_off(more);
  e += more;
  return __int2float_rn((int)p) * __int_as_float((e + 127) << 23);  // both exact: at most 25 bits, a power of two
}

// (double)x from its bits where x is a normal float.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x), e = (u >> 23) & 255u;
  if (e == 0u || e == 255u) return (double)x;
  return __hiloint2double((int)((u & 0x80000000u) | ((e + 896u) << 20) | ((u >> 3) & 0xfffffu)), (int)(u << 29));
}

__global__ void __launch_bounds__(kFsThreads) k_fourier_split(const TreeDev* trees, StepDev s) {
  chain_wait();
  __shared__ double s_part[kFsParts][kFourierTerms];
  __shared__ double s_base[kFourierTerms], s_slope[kFourierTerms];
  __shared__ double s_wave[4][KDT_FOURIER_MAX_J];  // sin K a, sin K b, cos K a, cos K b
  __shared__ double s_mid[2][kFsCand][kFsCand];  // by round's parity, outcome of the round before, candidate
  __shared__ double s_end[2][kFsCand][2];        // and each outcome's (lo, hi)
  __shared__ double s_term[kFsCand][96];
  __shared__ uint32_t s_neg[2];  // by round's parity; bit w: F < 0 at candidate w's midpoint
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t nc = ncells_of(s);
  for (int i = tid; i < kFsCand * 96; i += kFsThreads) (&s_term[0][0])[i] = 0.0;  // terms that no tree here has
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    const Cell cell = s.cells[c];
    const TreeDev& t = trees[cell.tree];
    const int J = t.fourier_j, nt = 2 * J + 1;
    // thread (part, term): the sum of every parts-th run record
    const uint32_t len = run_tiles(tiles_of((uint32_t)t.n)), nrun = (tiles_of(cell.count) + len - 1u) / len;
    const int parts = min(kFsParts, kFsThreads / nt), part = tid / nt;
    if (part < parts) {
      const int j = tid % nt;
      const double* first = (const double*)(s.tile_mm + (size_t)cell.tile0 * kTileRecWords) + j;
      const size_t step = (size_t)len * (kTileRecWords / 2);
      double sum = 0.0;
      for (uint32_t m0 = (uint32_t)part; m0 < nrun; m0 += 8u * (uint32_t)parts) {
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const uint32_t m = m0 + (uint32_t)(u * parts);
          v[u] = m < nrun ? first[m * step] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (m0 + (uint32_t)(u * parts) < nrun) sum += v[u];
      }
      s_part[part][j] = sum;
    }
    __syncthreads();
    double C = 0.0;  // thread j: the sum of term j
    if (tid < nt)
      for (uint32_t p = 0; p < min((uint32_t)parts, nrun); ++p) C += s_part[p][tid];
    // bounds: lane i of every warp takes the i-th ancestor (splits are in
    // [0, 1], where floats order like their bits)
    const uint32_t dim = s.kdim[c];
    uint32_t ba = 0u, bb = __float_as_uint(1.0f);
    if (lane < (int)cell.level) {
      const uint32_t par = ((cell.heap + 1u) >> (lane + 1)) - 1u;
      const uint32_t child = ((cell.heap + 1u) >> lane) - 1u;
      if (((uint32_t)cell.level - 1u - (uint32_t)lane) % (uint32_t)t.d == dim) {
        const uint32_t v = __float_as_uint(t.out_vals[par]);
        if (child == 2u * par + 1u) bb = v; else ba = v;
      }
    }
    const double a = (double)__uint_as_float(__reduce_max_sync(0xffffffffu, ba));
    const double b = (double)__uint_as_float(min(__reduce_min_sync(0xffffffffu, bb), __float_as_uint(1.0f)));
    // the bounds' waves, a thread each (a bound at the interval's end has
    // weight 0: its waves are not needed)
    {
      const int which = tid / KDT_FOURIER_MAX_J, j = tid % KDT_FOURIER_MAX_J;
      if (which < 4 && j < J) {
        const double x = (double)(2 * j + 1) * ((which & 1) ? b : a);
        const bool needed = (which & 1) ? b < 1.0 : a > 0.0;
        s_wave[which][j] = !needed ? 0.0 : which < 2 ? sin(x) : cos(x);
      }
    }
    __syncthreads();
    // per term: F_j(m) = base + slope * (sin or cos)(K m)
    const double ia = a > 0.0 ? 1.0 : 0.0, ib = b < 1.0 ? 1.0 : 0.0;
    if (tid < nt) {
      double base, slope = 0.0;
      if (tid == 0) {
        base = C * 0.5 * (ib - ia);
      } else {
        const int j = (tid - 1) / 2;
        const double qk = 2.0 / (3.14159265358979323846 * (double)(2 * j + 1));
        if (tid & 1) {
          base = -C * qk * (ia * s_wave[0][j] + ib * s_wave[1][j]);
          slope = 2.0 * C * qk;
        } else {
          base = C * qk * (ia * s_wave[2][j] + ib * s_wave[3][j]);
          slope = -2.0 * C * qk;
        }
      }
      s_base[tid] = base;
      s_slope[tid] = slope;
    }
    __syncthreads();
    // this thread's candidate and harmonic, and the half warp's candidate
    const int cand = 1 + tid / J, k = 1 + tid % J;
    const bool waves = cand < kFsCand;
    const double base_s = waves ? s_base[2 * k - 1] : 0.0, slope_s = waves ? s_slope[2 * k - 1] : 0.0;
    const double base_c = waves ? s_base[2 * k] : 0.0, slope_c = waves ? s_slope[2 * k] : 0.0;
    const int sum_cand = 1 + tid / 16, l = tid & 15;
    const bool sums = sum_cand < kFsCand;
    if (tid < kFsCand) s_term[tid][0] = s_base[0];
    const bool wave_s = slope_s != 0.0, wave_c = slope_c != 0.0;
    // half of a sum of bounds: its exponent less one (0 only for the cell [0, 0])
    auto half = [](double x) {
      const int h = __double2hiint(x), g = __double2loint(x);
      return (h | g) == 0 ? 0.0 : __hiloint2double(h - 0x00100000, g);
    };
    // thread (outcome, candidate): the midpoint of the candidate after that
    // outcome of a round whose midpoints are `mids`, its bounds to `end`
    auto form = [&](int i, double x, double y, const double* mids, double (*next)[kFsCand], double (*end)[2]) {
      const int out = i / kFsCand, cnd = i % kFsCand, top = 31 - __clz(cnd);
      if (mids) {
        uint32_t w = 1;
#pragma unroll
        for (int st = 0; st < kFsSteps; ++st) {
          const uint32_t up = ((uint32_t)out >> (kFsSteps - 1 - st)) & 1u;
          if (up) x = mids[w]; else y = mids[w];
          w = 2u * w + up;
        }
      }
      if (cnd == 0) {
        end[out][0] = x;
        end[out][1] = y;
        return;
      }
      double mid = half(x + y);
#pragma unroll
      for (int st = 0; st < kFsSteps - 1; ++st)
        if (top > st) {
          if ((cnd >> (top - 1 - st)) & 1) x = mid; else y = mid;
          mid = half(x + y);
        }
      next[out][cnd] = mid;
    };
    if (tid < kFsCand) form(tid, a, b, nullptr, s_mid[0], s_end[0]);  // the first round: outcome 0 of none
    if (tid == 0) s_neg[0] = 0u;
    uint32_t out = 0;
    __syncthreads();
    for (int it = 0; it < 60 / kFsSteps; ++it) {
      const double* mids = s_mid[it & 1][out];
      if (waves) {
        const float arg = product_float((uint32_t)(2 * k - 1), mids[cand]);
        float sn, cs;
        sincosf(arg, &sn, &cs);
        s_term[cand][2 * k - 1] = wave_s ? __dadd_rn(base_s, __dmul_rn(slope_s, widen(sn))) : base_s;
        s_term[cand][2 * k] = wave_c ? __dadd_rn(base_c, __dmul_rn(slope_c, widen(cs))) : base_c;
      }
      if (tid >= kFsThreads - kFsCand * kFsCand)  // the last two warps (with terms of their own only for J > 27)
        form(tid - (kFsThreads - kFsCand * kFsCand), s_end[it & 1][out][0], s_end[it & 1][out][1], mids,
             s_mid[(it + 1) & 1], s_end[(it + 1) & 1]);
      __syncthreads();
      if (tid == 0) s_neg[(it + 1) & 1] = 0u;  // (read by all before this barrier, written after the next)
      {
        double f = 0.0;
        if (sums) {
          const double* p = s_term[sum_cand];
          double u = p[l], v = p[l + 16];
          if (l + 32 < nt) u = __dadd_rn(u, p[l + 32]);
          if (l + 48 < nt) v = __dadd_rn(v, p[l + 48]);
          if (l + 64 < nt) u = __dadd_rn(u, p[l + 64]);
          f = __dadd_rn(u, v);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) f += __shfl_down_sync(0xffffffffu, f, o, 16);
        // F < 0: the sign, unless it is zero
        const int h = __double2hiint(f);
        if (sums && l == 0 && h < 0 && (((uint32_t)h << 1) | (uint32_t)__double2loint(f)) != 0u)
          atomicOr(&s_neg[it & 1], 1u << sum_cand);
      }
      __syncthreads();
      const uint32_t neg = s_neg[it & 1];
      uint32_t w = 1;
#pragma unroll
      for (int st = 0; st < kFsSteps; ++st) w = 2u * w + ((neg >> w) & 1u);
      out = w - (uint32_t)kFsCand;
    }
    const double lo = s_end[0][out][0], hi = s_end[0][out][1];
    if (tid == 0) {
      const float m32 = (float)(0.5 * (lo + hi));
      s.mkey[c] = ord_key(m32);
      t.out_vals[cell.heap] = m32;
      t.out_dims[cell.heap] = (int8_t)dim;
    }
    __syncthreads();  // shared memory is free for the next cell
    if (c + gridDim.x < nc)  // (another tree may have fewer terms)
      for (int i = tid; i < kFsCand * 96; i += kFsThreads) (&s_term[0][0])[i] = 0.0;
  }
}

// ------------------------------------------------------------ partition

// Per tile: number of points with key <= split. One warp per tile: the
// tile's key range is read 16 bytes at a time with all of a lane's loads in
// flight together (its unaligned head and tail by single words).
__device__ __forceinline__ void part_count_tile(const TreeDev* trees, const StepDev& s, uint32_t tile, uint2 tl) {
  constexpr int kV = kTile / 4 / 32;  // 16-byte vectors per lane of a full tile
  const int lane = threadIdx.x & 31;
  const Cell cell = s.cells[tl.x];
  const TreeDev& t = trees[cell.tree];
  const float* X = src_cols(t, cell.level) + (int64_t)s.kdim[tl.x] * t.n + cell.begin + tl.y;
  const uint32_t m = s.mkey[tl.x];
  const uint32_t cnt_pts = min((uint32_t)kTile, cell.count - tl.y);
  const uint32_t head = min(cnt_pts, (4u - (uint32_t)(((uintptr_t)X >> 2) & 3u)) & 3u);
  const uint32_t nv = (cnt_pts - head) >> 2, tail0 = head + nv * 4u;
  const float4* xv = (const float4*)(X + head);  // 16-byte aligned
  float4 v[kV];
#pragma unroll
  for (int q = 0; q < kV; ++q) {
    const uint32_t i = (uint32_t)(lane + q * 32);
    v[q] = i < nv ? __ldg(xv + i) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  uint32_t cnt = 0;
#pragma unroll
  for (int q = 0; q < kV; ++q)
    if ((uint32_t)(lane + q * 32) < nv)
      cnt += (ord_key(v[q].x) <= m) + (ord_key(v[q].y) <= m) + (ord_key(v[q].z) <= m) + (ord_key(v[q].w) <= m);
  if ((uint32_t)lane < head) cnt += ord_key(__ldg(X + lane)) <= m;
  if ((uint32_t)lane < cnt_pts - tail0) cnt += ord_key(__ldg(X + tail0 + lane)) <= m;
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if (lane == 0) s.tile_left[tile] = cnt;
}

// Warps stride over the tiles; three CTAs per SM by a register bound (80
// registers: a lane's sixteen 16-byte loads still fit, with a few words of
// spill).
__global__ void __launch_bounds__(256, 3) k_part_count(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t ntiles = ntiles_of(s);
  for (uint32_t tile = blockIdx.x * 8u + (threadIdx.x >> 5); tile < ntiles; tile += gridDim.x * 8u)
    part_count_tile(trees, s, tile, s.tiles[tile]);
}

// One CTA per cell: exclusive scan of its tiles' left counts.
__device__ __forceinline__ void part_scan_cell(const StepDev& s, uint32_t c, const Cell& cell) {
  __shared__ uint32_t tmp[33];
  const uint32_t tb = cell.tile0, te = tb + tiles_of(cell.count);
  uint32_t run = 0;
  for (uint32_t j0 = tb; j0 < te; j0 += blockDim.x) {
    const uint32_t j = j0 + threadIdx.x;
    const uint32_t v = j < te ? s.tile_left[j] : 0u;
    uint32_t tot;
    const uint32_t ex = block_excl_scan(v, tmp, &tot);
    if (j < te) s.tile_loff[j] = run + ex;
    run += tot;
  }
  if (threadIdx.x == 0) s.lcount[c] = run;
}

__global__ void k_part_scan(StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    part_scan_cell(s, c, s.cells[c]);
    __syncthreads();  // the cell's shared memory is free for the next one
  }
}

// One warp per cell (widest spread): the key coordinate of each big child,
// and of each child queued for the subtree kernel (its first level), from its
// min and max key per coordinate (reduced by the scatter): the
// largest range (double)max - (double)min, 0 for equal keys, lowest
// coordinate on ties. A range is never negative, so the bit patterns of two
// ranges order like the ranges as unsigned integers: the argmax runs on the
// high word, then the low word, then the lowest coordinate, by integer warp
// reductions (double arithmetic, slow on this part, only for the one
// subtraction per range).
__device__ __forceinline__ void child_dims_cell(const TreeDev* trees, const StepDev& s, uint32_t c) {
  const int lane = threadIdx.x & 31;
  const Cell cell = s.cells[c];
  const TreeDev& t = trees[cell.tree];
  if (t.key_rule != KEY_WIDEST) return;
  const int d = t.d;
  for (int side = 0; side < 2; ++side) {
    const uint2 cr = s.crow[2 * c + side];
    if (cr.x == kNoRow && cr.y == kNoRow) continue;  // terminal
    uint64_t rb = 0ull;
    uint32_t ib = 0xffffffffu;
    for (int l = lane; l < d; l += 32) {  // l ascending: the first of equal ranges is kept
      const uint2 mm = *(const uint2*)&s.child_mm[(((size_t)c * 2 + side) * kMaxDims + l) * 2];
      const uint64_t range = (uint64_t)__double_as_longlong(key_range(mm.x, mm.y));
      if (ib == 0xffffffffu || range > rb) {
        rb = range;
        ib = (uint32_t)l;
      }
    }
    const uint32_t rh = (uint32_t)(rb >> 32), rl = (uint32_t)rb;
    const uint32_t mh = __reduce_max_sync(0xffffffffu, ib != 0xffffffffu ? rh : 0u);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, (ib != 0xffffffffu && rh == mh) ? rl : 0u);
    ib = __reduce_min_sync(0xffffffffu, (ib != 0xffffffffu && rh == mh && rl == ml) ? ib : 0xffffffffu);
    if (lane == 0) {
      if (cr.x != kNoRow)
        s.next_big[cr.x].dim = (int16_t)ib;
      else
        s.small[cr.y].dim = (int16_t)ib;  // the subtree kernel's first level
    }
  }
}

__global__ void __launch_bounds__(256, 1) k_child_dims(const TreeDev* trees, StepDev s) {
  chain_wait();
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x * 8u + (threadIdx.x >> 5); c < nc; c += gridDim.x * 8u) child_dims_cell(trees, s, c);
}

// ------------------------------------------------------------- children

// Exclusive prefix of v over the warp's lanes; *total for all.
__device__ __forceinline__ uint32_t warp_excl(uint32_t v, uint32_t* total) {
  const uint32_t inc = warp_incl_scan(v);
  *total = __shfl_sync(0xffffffffu, inc, 31);
  return inc - v;
}

// The cells of a warp's active lanes, one each, after the children's sizes are
// known and before the move: terminal children are recorded, small ones queued
// for the subtree kernel, big ones get a slot of the next step, their tiles,
// their segments and a row of subset offsets (which the scatter fills). The
// warp's children reserve together, an atomic per counter (each counter is one
// address for all cells of a step); every row of offsets is one word longer
// than the child's segments, so the big children's slots and segments, counted
// in one 64-bit word, give its place too.
__device__ __forceinline__ void classify_lanes(const TreeDev* trees, const StepDev& s, uint32_t c, bool active) {
  const int lane = threadIdx.x & 31;
  Cell cell{};
  uint32_t L = 0;
  if (active) {
    cell = s.cells[c];
    L = s.lcount[c];
  }
  const TreeDev& t = trees[cell.tree];
  const uint32_t R = cell.count - L;
  const int level = cell.level + 1;
  const int stall = (R == 0) ? cell.stall + 1 : 0;
  const uint32_t cb[2] = {cell.begin, cell.begin + L};
  const uint32_t cc[2] = {L, R};
  int live_delta = -1;  // this cell is done; each child that still needs splitting adds one
  bool big[2] = {false, false}, small[2] = {false, false};
  uint32_t row_words[2] = {0u, 0u};
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    if (!active) continue;
    if (is_terminal(t, cc[side], level, stall)) {
      record_terminal(t, cb[side], cc[side], 2u * cell.heap + 1u + (uint32_t)side, level);
    } else if (t.depth == 0 && level >= t.max_levels) {
      set_status(t, ST_LEVEL_CAP);
    } else {
      ++live_delta;
      small[side] = cc[side] <= (uint32_t)t.small_max;
      big[side] = !small[side];
      // explicit ids: a row of subset offsets where it is shorter than the cell
      if (small[side] && t.subset_mode == SUB_EXPLICIT && (uint32_t)t.r < cc[side])
        row_words[side] = (uint32_t)t.r + 1u;
    }
  }
  const uint32_t nb = (uint32_t)big[0] + (uint32_t)big[1], ns = (uint32_t)small[0] + (uint32_t)small[1];
  const bool wide = active && t.sub_wide != 0;
  const uint32_t tl[2] = {big[0] ? tiles_of(cc[0]) : 0u, big[1] ? tiles_of(cc[1]) : 0u};
  const uint32_t segs = active ? nb * (uint32_t)t.r : 0u;
  uint32_t nb_all, segs_all, tl_all, bp_all, nn_all, nw_all, sp_all, rw_all;
  const uint32_t nb_ex = warp_excl(nb, &nb_all);
  const uint32_t segs_ex = warp_excl(segs, &segs_all);
  const uint32_t tl_ex = warp_excl(tl[0] + tl[1], &tl_all);
  const uint32_t nn_ex = warp_excl(wide ? 0u : ns, &nn_all);
  const uint32_t nw_ex = warp_excl(wide ? ns : 0u, &nw_all);
  const uint32_t rw_ex = warp_excl(row_words[0] + row_words[1], &rw_all);
  bp_all = warp_sum((big[0] ? cc[0] : 0u) + (big[1] ? cc[1] : 0u));
  sp_all = warp_sum((small[0] ? cc[0] : 0u) + (small[1] ? cc[1] : 0u));
  unsigned long long b0 = 0, t0 = 0, s0 = 0;
  uint32_t w0 = 0;
  if (lane == 0) {
    if (nb_all) {
      b0 = atomicAdd(s.next_big_ctr, (unsigned long long)nb_all | ((unsigned long long)segs_all << 32));
      t0 = atomicAdd(s.next_tile_ctr, (unsigned long long)tl_all | ((unsigned long long)bp_all << 32));
    }
    if (nn_all | nw_all) {
      s0 = atomicAdd(s.small_ctr, (unsigned long long)nn_all | ((unsigned long long)nw_all << 32));
      atomicAdd(s.small_points, sp_all);
    }
    if (rw_all) w0 = atomicAdd(s.small_off_used, rw_all);
  }
  b0 = __shfl_sync(0xffffffffu, b0, 0);
  t0 = __shfl_sync(0xffffffffu, t0, 0);
  s0 = __shfl_sync(0xffffffffu, s0, 0);
  w0 = __shfl_sync(0xffffffffu, w0, 0);
  if (!active) return;
  // the two ends of the queue never meet while their counts sum to small_cap at most
  const bool room = (uint64_t)(uint32_t)s0 + (uint32_t)(s0 >> 32) + nn_all + nw_all <= (uint64_t)s.small_cap;
  uint32_t slot_b = (uint32_t)b0 + nb_ex, seg = (uint32_t)(b0 >> 32) + segs_ex, tile = (uint32_t)t0 + tl_ex;
  uint32_t slot_n = (uint32_t)s0 + nn_ex, slot_w = (uint32_t)(s0 >> 32) + nw_ex, rw = w0 + rw_ex;
#pragma unroll
  for (int side = 0; side < 2; ++side) {
    uint2 cr = make_uint2(kNoRow, kNoRow);
    Cell child{cb[side], cc[side], 2u * cell.heap + 1u + (uint32_t)side, cell.tree, (int8_t)level, (int8_t)stall,
               (int16_t)-1};
    if (small[side]) {
      if (room) {
        const uint32_t slot = wide ? s.small_cap - 1u - slot_w++ : slot_n++;
        const uint32_t words = row_words[side];
        if (words && rw < s.small_off_cap && words <= s.small_off_cap - rw) child.row = rw;
        rw += words;
        s.small[slot] = child;
        cr = make_uint2(kNoRow, slot);  // its widest coordinate is picked with the big children's
      } else {
        set_status(t, ST_CAPACITY);
      }
    } else if (big[side]) {
      const uint32_t r = (uint32_t)t.r, row = seg + slot_b;
      if (slot_b < s.next_big_cap && row <= s.off_cap - (r + 1u) && seg + r <= s.nseg_cap &&
          tile + tl[side] <= s.tiles_cap) {
        child.tile0 = tile;
        child.seg0 = seg;
        s.next_big[slot_b] = child;
        s.obase_next[slot_b] = row;
        cr = make_uint2(slot_b, row);
      } else {
        set_status(t, ST_CAPACITY);
      }
      ++slot_b;
      seg += r;
      tile += tl[side];
    }
    s.crow[2 * c + side] = cr;
  }
  if (live_delta) atomicAdd(t.live, live_delta);
}

// Identities for the scatter's min / max reductions of the cell's children.
__device__ __forceinline__ void clear_child_mm(const TreeDev* trees, const StepDev& s, uint32_t c, uint32_t tid,
                                               uint32_t threads) {
  const TreeDev& t = trees[s.cells[c].tree];
  if (t.key_rule != KEY_WIDEST) return;
  for (uint32_t j = tid; j < 4u * (uint32_t)t.d; j += threads) {
    const uint32_t side = j / (2u * (uint32_t)t.d), l = (j / 2u) % (uint32_t)t.d, which = j & 1u;
    s.child_mm[(((size_t)c * 2 + side) * kMaxDims + l) * 2 + which] = which ? 0u : 0xffffffffu;
  }
}

// 32 cells per CTA: the left counts of each cell's tiles are scanned by a warp
// (unless k_part_scan did), then one warp classifies the 32 together.
__global__ void __launch_bounds__(256) k_classify(const TreeDev* trees, StepDev s, bool scanned) {
  chain_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nc = ncells_of(s);
  for (uint32_t c0 = blockIdx.x * 32u; c0 < nc; c0 += gridDim.x * 32u) {
    for (uint32_t c = c0 + warp; c < min(c0 + 32u, nc); c += 8u) {
      clear_child_mm(trees, s, c, lane, 32u);
      if (scanned) continue;
      const Cell cell = s.cells[c];
      const uint32_t tb = cell.tile0, te = tb + tiles_of(cell.count);
      uint32_t run = 0;
      for (uint32_t j0 = tb; j0 < te; j0 += 32) {
        const uint32_t j = j0 + (uint32_t)lane;
        const uint32_t v = j < te ? s.tile_left[j] : 0u;
        const uint32_t inc = warp_incl_scan(v);
        if (j < te) s.tile_loff[j] = run + inc - v;
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (lane == 0) s.lcount[c] = run;
    }
    __syncthreads();
    if (warp == 0) classify_lanes(trees, s, c0 + lane, c0 + lane < nc);
    __syncthreads();
  }
}

// Steps of few cells of few tiles: one CTA per cell does what k_combine,
// k_part_count, k_part_scan and k_classify do in four launches (65,536 points, 8
// subsets: 75 us for the six steps of a build, 183 in four launches each).
constexpr int kSplitThreads = 512;
__global__ void __launch_bounds__(kSplitThreads) k_split(const TreeDev* trees, StepDev s) {
  chain_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t nc = ncells_of(s);
  for (uint32_t c = blockIdx.x; c < nc; c += gridDim.x) {
    const Cell cell = s.cells[c];
    clear_child_mm(trees, s, c, threadIdx.x, kSplitThreads);
    combine_cell(trees, s, c);
    __syncthreads();  // the split key is written
    const uint32_t nt = tiles_of(cell.count);
    for (uint32_t k = warp; k < nt; k += kSplitThreads / 32)
      part_count_tile(trees, s, cell.tile0 + k, make_uint2(c, k * (uint32_t)kTile));
    __syncthreads();
    part_scan_cell(s, c, cell);
    __syncthreads();
    if (warp == 0) classify_lanes(trees, s, c, lane == 0);
    __syncthreads();  // shared memory is free for the next cell
  }
}

}  // namespace

// ------------------------------------------------------------ launcher

// From here on a warp per cell in combine (a line of 256, 1024 and 4096 cells: 1,000,003
// points, 4096 subsets 1097, 1098 and 1091 us, 3,000,017, 1000 subsets 1.90, 1.90 and
// 1.87 ms, trees of fewer subsets the same).
constexpr uint32_t kManyCells = 1024;

// Steps whose launches weigh more than their work: while all segments fit the
// SMs at once (8 CTAs of 256 threads each) and are of at most 8192 keys on
// average, every one gets such a CTA, in one launch (65,536 points, 8 subsets:
// 68 us for the six steps of a build, 229 in three launches a step). Larger ones
// get the 512 threads of the listed path (64 segments of 780,000 keys and the
// four levels below them: 1.33 ms here, 0.84 there).
bool step_selects_all(uint32_t nseg, uint64_t points, uint32_t sms) {
  return nseg <= 8u * sms && points <= 8192ull * nseg;
}

// Few, large segments: several CTAs each. A CTA takes about 0.2 ns a key, the
// four launches 40 us and 4 ps a key of the step. Builds of one level: 32
// segments of 262,144 keys 209 us here and 208 with a CTA each, of 524,288 keys
// 276 and 303; 8 of 262,144 keys 156 and 173; 64 of 262,144 keys take a CTA each
// 57 us and would take 108 here.
bool step_selects_wide(uint32_t nseg, uint64_t points) { return nseg <= 32u && points >= 262144ull * nseg; }

// One CTA per cell combines, counts, scans and classifies: in steps of at most two
// cells per SM, of at most 64 tiles on average (a warp reads 4). (kdt_build of
// 1,000,003 and 3,000,017 points in 3 coordinates, 16 subsets, and of 2^24, 64: up
// to four cells per SM 680, 1354 and 3490 us, two 660, 1339 and 3467, one 668, 1342
// and 3459, half of one 669, 1342 and 3468; with 16 tiles 684, 1362 and 3480, with
// 256 708, 1366 and 3496, at four cells per SM. In a step ahead both are bounds: a
// cell with most of the points has one CTA all the same. 16,000,057 points, 95% of
// them at one place: 20.6 ms, 22.5 with four launches and a wait per step.)
static bool step_splits(const StepDev& s, uint32_t sms2) {
  return (!s.ncells_dev || s.bounded) && s.ncells <= sms2 && s.ntiles <= 64u * s.ncells;
}

// The selects by segment size: one thread, one warp, one CTA per segment.
static void launch_listed_selects(const TreeDev* trees, const StepDev& s, uint32_t nseg, uint32_t max_r,
                                  uint32_t max_bigseg, const SelectTuning& tune, uint64_t points, uint32_t sms,
                                  cudaStream_t st) {
  {
    TraceScope ts(K_SELECT_TINY, st, points);
    launch_chained(k_select_tiny, std::max<uint32_t>(1, std::min<uint32_t>((nseg + 255) / 256, sms * 16u)), 256, 0, st,
                   trees, s);
  }
  {
    TraceScope ts(K_SELECT_SMALL, st, points);
    launch_chained(k_select_small, std::max<uint32_t>(1, std::min<uint32_t>((nseg + 7) / 8, sms * 8u)), 256, 0, st,
                   trees, s);
  }
  if (max_bigseg == 0) return;
  if (s.wide_segs) {
    // CTAs per segment: four per SM in all, of at least 8192 keys each
    const uint32_t x = std::max<uint32_t>(
        1, (uint32_t)std::min<uint64_t>(2u * sms / std::max(1u, nseg), points / std::max(1u, nseg) / 8192u));
    const uint32_t y = std::min(max_r, nseg - std::min(nseg, s.ncells) + 1u);  // every cell has a segment
    {
      TraceScope ts(K_SELECT_WIDE, st);
      launch_chained(k_wide_clear, dim3(1, y, s.ncells), kWideThreads, 0, st, trees, s);
    }
    for (int top = 32; top > 0; top -= 11) {
      TraceScope ts(K_SELECT_WIDE, st, points);
      launch_chained(k_wide_pass, dim3(x, y, s.ncells), kWideThreads, 0, st, trees, s, top);
    }
  }
  TraceScope ts(K_SELECT_BIG, st);
  // nseg bounds the big segments too; with few of them (the first levels
  // of a large tree) a CTA's loads in flight set the rate, so they take
  // 512 threads whatever the tuning, and 1024 while two CTAs per SM take them
  // all (64 segments of 780,000 keys: 322 us with 512 threads, 188 with 1024;
  // 300 of 100,000: 71 and 64; a build of 50,000,021 points 5.64 -> 5.42 ms)
  const uint32_t grid = std::max<uint32_t>(1, std::min<uint32_t>(std::min(max_bigseg, nseg), sms * 4u));
  if (nseg <= sms) {
    if (tune.digit_bits == 8)
      launch_chained(k_select_big<1024, 8>, grid, 1024, 0, st, trees, s);
    else
      launch_chained(k_select_big<1024, 11>, grid, 1024, 0, st, trees, s);
  } else if (tune.cta_threads == 512 || nseg <= sms * 4u) {
    if (tune.digit_bits == 8)
      launch_chained(k_select_big<512, 8>, grid, 512, 0, st, trees, s);
    else
      launch_chained(k_select_big<512, 11>, grid, 512, 0, st, trees, s);
  } else {
    if (tune.digit_bits == 8)
      launch_chained(k_select_big<256, 8>, grid, 256, 0, st, trees, s);
    else
      launch_chained(k_select_big<256, 11>, grid, 256, 0, st, trees, s);
  }
}

namespace {

// Trees that join the engine, a CTA each: their records, cleared words, the
// root's cell in its list, or (a root that is terminal) its terminal record
// and, up to kAdmitIota points, the identity permutation.
__device__ __forceinline__ void admit_tree(const AdmitRec& a, TreeDev* trees) {
  const TreeDev& t = a.tree;
  if (a.terminal && t.n <= (int64_t)kAdmitIota)
    for (uint32_t i = threadIdx.x; i < (uint32_t)t.n; i += blockDim.x) t.out_perm[i] = i;
  if (threadIdx.x != 0) return;
  trees[a.slot] = t;
  *t.status = ST_OK;
  *t.levels = 0;
  *t.huge_count = 0;
  *t.term_count = a.terminal ? 1u : 0u;
  *t.live = a.terminal ? 0 : 1;
  if (a.terminal)
    t.terms[0] = TermRec{0u, (uint32_t)t.n, 0u, 0};
  else
    *a.root_dst = Cell{0u, (uint32_t)t.n, 0u, (int32_t)a.slot, 0, 0, -1, kNoRow, a.tile0, a.seg0};
}

__global__ void __launch_bounds__(256) k_admit(const AdmitRec* recs, TreeDev* trees) {
  chain_wait();
  admit_tree(recs[blockIdx.x], trees);
}

// The same with the records among the launch's parameters (no copy before it).
__global__ void __launch_bounds__(256) k_admit_few(const __grid_constant__ AdmitFew few, TreeDev* trees) {
  chain_wait();
  admit_tree(few.rec[blockIdx.x], trees);
}

}  // namespace

cudaError_t launch_admit(const std::vector<AdmitRec>& recs, AdmitRec* staging, TreeDev* trees, cudaStream_t st) {
  if (recs.empty()) return cudaSuccess;
  if (recs.size() <= (size_t)kAdmitFew) {
    AdmitFew few{};
    std::copy(recs.begin(), recs.end(), few.rec);
    TraceScope ts(K_ADMIT, st);
    launch_chained(k_admit_few, (unsigned)recs.size(), 256, 0, st, few, trees);
  } else {
    const cudaError_t e =
        cudaMemcpyAsync(staging, recs.data(), recs.size() * sizeof(AdmitRec), cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    TraceScope ts(K_ADMIT, st);
    launch_chained(k_admit, (unsigned)recs.size(), 256, 0, st, staging, trees);
  }
  for (const AdmitRec& a : recs)
    if (a.terminal && a.tree.n > (int64_t)kAdmitIota) launch_iota(a.tree.out_perm, (uint32_t)a.tree.n, st);
  return cudaGetLastError();
}

cudaError_t prepare_step_kernels() {
  return cudaFuncSetAttribute(k_ps_move, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)ps_smem_bytes(kMaxSubsets));
}

void launch_big_step(const TreeDev* trees, const StepDev& s, uint32_t max_tiles, uint32_t nseg,
                     uint32_t max_bigseg, bool has_roots, bool need_root_dims, bool any_widest, int max_r, int uniform_d,
                     const SelectTuning& tune, uint64_t points, uint32_t sms, cudaStream_t st, bool fourier) {
  // s.ncells: the step's cells, or at most so many (s.bounded), or (a step inside
  // a graph) their capacity; per-cell kernels stride over the cells, so their
  // grids cover the cells exactly in the first two and are capped in the last
  const uint32_t nc = s.ncells;
  if (nc == 0) return;
  const bool dev = s.ncells_dev != nullptr && !s.bounded;
  auto cells_grid = [&](uint32_t per_block, uint32_t cap) {
    const uint32_t g = (nc + per_block - 1) / per_block;
    return std::max<uint32_t>(1, dev ? std::min(g, cap) : g);
  };
  if (s.shards) launch_shard_index(s, nc, st);
  if (has_roots) {
    { TraceScope ts(K_TILES, st); launch_chained(k_tiles, cells_grid(8, sms * 8u), 256, 0, st, trees, s); }
    {
      TraceScope ts(K_PS_COUNT, st, points);
      launch_chained(k_ps_count, std::max<uint32_t>(1, std::min(max_tiles, sms * 4u)), kTileThreads, 0, st, trees, s);
    }
    { TraceScope ts(K_PS_OFFSETS, st); launch_chained(k_ps_offsets, nc, 1024, 0, st, trees, s); }
    {
      TraceScope ts(K_PS_MOVE, st, points);
      launch_chained(k_ps_move, max_tiles, kPsThreads, ps_smem_bytes((uint32_t)max_r), st, trees, s);
    }
  }
  if (need_root_dims) {
    { TraceScope ts(K_MINMAX, st, points); launch_chained(k_minmax, max_tiles, kTileThreads, 0, st, trees, s); }
    { TraceScope ts(K_PICK_DIM, st); launch_chained(k_pick_dim, nc, 1024, 0, st, trees, s); }
  }
  {
    // threads per cell: enough for its segments
    uint32_t gt = 32;
    while (gt < 256u && gt < (uint32_t)max_r) gt *= 2;
    if (!dev && nc < sms) gt = 256;  // few cells: their tiles count
    TraceScope ts(K_CELLS, st);
    launch_chained(k_cells, cells_grid(256u / gt, sms * 8u), 256, 0, st, trees, s, gt);
  }
  // a CTA per cell while cells are few (large subset counts, deep scans),
  // a warp per cell once they are many (and in a graph, where the count is
  // not known when the launch is recorded)
  const bool many = dev || nc >= kManyCells;
  const bool split = step_splits(s, sms) && !fourier;
  if (fourier) {  // the paper's estimator: per-run sums, then the root per cell
    const uint32_t mgrid = std::max<uint32_t>(1, std::min(max_tiles, sms * 2u));
    {
      TraceScope ts(K_FOURIER_MOMENTS, st, points);
      launch_chained(k_fourier_moments, mgrid, 256, 0, st, trees, s);
    }
    {
      TraceScope ts(K_FOURIER_SPLIT, st);
      launch_chained(k_fourier_split, cells_grid(1, sms * 4u), kFsThreads, 0, st, trees, s);
    }
  } else {
    if (s.few_segs) {
      TraceScope ts(K_SELECT_ALL, st, points);
      launch_chained(k_select_all, std::max<uint32_t>(1, nseg), 256, 0, st, trees, s);
    } else {
      launch_listed_selects(trees, s, nseg, (uint32_t)max_r, max_bigseg, tune, points, sms, st);
    }
    if (s.shards) launch_shard_medians(trees, s, nc, st);  // the all-gather of the segment statistics
    if (!split) {
      TraceScope ts(K_COMBINE, st);
      if (many)
        launch_chained(k_combine_warp, cells_grid(8, sms * 8u), 256, 0, st, trees, s);
      else
        launch_chained(k_combine, nc, 256, 0, st, trees, s);
    }
  }
  if (split) {
    TraceScope ts(K_SPLIT, st, points);
    launch_chained(k_split, nc, kSplitThreads, 0, st, trees, s);
  } else {
    {
      TraceScope ts(K_PART_COUNT, st, points);
      launch_chained(k_part_count, std::max<uint32_t>(1, std::min((max_tiles + 7) / 8, sms * 16u)), 256, 0, st, trees,
                     s);
    }
    // a cell of very many tiles: a CTA scans them, not a warp
    const bool scanned = !dev && max_tiles / nc > 64u;
    if (scanned) {
      TraceScope ts(K_PART_SCAN, st);
      launch_chained(k_part_scan, nc, 1024, 0, st, s);
    }
    {
      TraceScope ts(K_CLASSIFY, st);
      launch_chained(k_classify, cells_grid(32, sms * 4u), 256, 0, st, trees, s, scanned);
    }
  }
  launch_scatter(trees, s, max_tiles, sms / 2, points, uniform_d, any_widest, st);
  if (any_widest && s.shards) launch_shard_minmax(trees, s, nc, st);
  if (any_widest) {
    TraceScope ts(K_CHILD_DIMS, st);
    launch_chained(k_child_dims, cells_grid(8, sms * 8u), 256, 0, st, trees, s);
  }
}

namespace {

// Last node of a graph's loop body: count the iteration and keep looping
// while the next step has cells (at most `limit` iterations).
__global__ void k_loop_cond(cudaGraphConditionalHandle h, const uint32_t* ncells_next, uint32_t* iters,
                            uint32_t limit) {
  const uint32_t it = *iters + 1u;
  *iters = it;
  cudaGraphSetConditional(h, (*ncells_next > 0u && it < limit) ? 1u : 0u);
}

}  // namespace

void launch_loop_cond(cudaGraphConditionalHandle h, const uint32_t* ncells_next, uint32_t* iters, uint32_t limit,
                      cudaStream_t st) {
  k_loop_cond<<<1, 1, 0, st>>>(h, ncells_next, iters, limit);
}

}  // namespace kdt
