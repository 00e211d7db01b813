// kdt_launch.h -- host-side declarations shared by the CUDA translation units.
#pragma once
#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

#include "kdt_internal.cuh"

namespace kdt {

// Per-level local cell of the subtree kernel (shared memory while a level's
// live cells fit the shape's table, else a per-CTA slice of global memory).
struct LCell {
  uint32_t heap;
  uint32_t mkey;    // split key
  uint16_t begin;   // local position
  uint16_t count;
  uint16_t lcount;  // left child size
  uint8_t dim;      // key coordinate
  uint8_t stall;    // consecutive splits that left the right child empty
};
static_assert(sizeof(LCell) == 16, "LCell is 16 bytes");

// A launch that may be prepared while the kernel before it in the stream
// drains; the kernel begins with chain_wait(). The levels of a build are chains
// of short kernels, and what lies between two of them is 2 to 4 us less this
// way (65,536 points, 24 launches: 329 to 286 us; 300,007 points, 46: 553 to
// 450; 3,000,017 points, 111: 2139 to 1894). Blocks that come to the SMs as soon
// as those before them have started, and wait there, cost the running ones more
// than that saves (511 us for the 300,007 points). Steps recorded into a graph
// keep plain edges.
template <class... P, class... A>
inline void launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = st;
  c.attrs = at;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  c.numAttrs = cudaStreamIsCapturing(st, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, P(args)...);
}

// The subtree kernel comes in three shapes:
//   narrow (d <= kSubtreeNarrowMaxD): 256 threads of at most 5 positions (1280
//     points), three CTAs per SM in 74 KB of dynamic shared memory each, cell
//     tables of 128 cells;
//   wide (larger d): 256 threads of at most 8 positions (2048 points), two CTAs
//     per SM in 112 KB each, cell tables of 256 cells;
//   tall (trees built alone whose cells of that size are no more than the SMs):
//     1024 threads of at most 5 positions (5120 points), one CTA per SM in 220
//     KB, cell tables of 256 cells.
// In the first two several CTAs share an SM, each finishing its own cell, so
// that one CTA's barriers and copies overlap the others' work: that is best
// while there are more cells than CTAs. With fewer, what a build waits for is
// the levels above, a chain of launches each (about 25 us a level), so the tall
// shape takes cells two levels larger. (kdt_build, the shape by d and the tall one:
// 65,536 points, d = 3 291 and 282 us; 150,001, d = 8 488 and 369; 300,007, d = 16,
// its 128 cells the most that the rule allows, 528 and 450; 250,001, d = 8, widest
// spread 467 and 479.)
struct SubtreeShape {
  int threads;
  int q;        // positions per thread
  int ctas;     // CTAs per SM
  size_t smem;  // dynamic shared memory per CTA
  int cells;    // cells of one level's table in shared memory
  int bigs;     // segments above the rank-counting size (32): points / 33 at most
};
constexpr SubtreeShape kSubNarrow{256, 5, 3, 74 * 1024, 128, 64};
constexpr SubtreeShape kSubWide{256, 8, 2, 112 * 1024, 256, 64};
constexpr SubtreeShape kSubTall{1024, 5, 1, 220 * 1024, 256, 160};
constexpr int kSubtreeNarrowMaxD = 8;
constexpr int kSubtreeHists = 8;                       // warps that may use a radix histogram at a time
constexpr int kSubtreeHistWords = kSubtreeHists * 256;  // their histograms; also the root's subset counts
__host__ __device__ constexpr size_t subtree_fixed_bytes(const SubtreeShape& sh) {
  return (size_t)kSubtreeHistWords * 4 + (size_t)sh.bigs * 2 + 2 * (size_t)sh.cells * sizeof(LCell);
}
inline const SubtreeShape& subtree_shape(int d) { return d <= kSubtreeNarrowMaxD ? kSubNarrow : kSubWide; }

// Column stride (elements) of a cell of N points in shared memory: room for
// the 16-byte alignment phase of the bulk copies.
__host__ __device__ inline uint32_t subtree_stride(uint32_t N) { return (N + 8 + 3) & ~3u; }

// Bytes of shared memory a cell of N points with d coordinates needs beyond
// the fixed part: d key columns at the padded stride, the keys in local order
// and the segment medians (4 bytes each), the subset ids, two orders, cell
// ids, a scan and the segment starts (2 bytes each).
__host__ __device__ inline size_t subtree_point_bytes(uint32_t N, int d) {
  const size_t stride = subtree_stride(N);
  return (size_t)d * stride * 4 + 2 * (((size_t)N * 4 + 15) & ~(size_t)15) +
         6 * ((((size_t)N + 1) * 2 + 15) & ~(size_t)15);
}

// Largest cell (points) that a shape of the subtree kernel holds for d
// coordinates.
inline int subtree_capacity(int d, const SubtreeShape& sh) {
  if (d < 1) return 0;
  const size_t fixed = subtree_fixed_bytes(sh);
  int lo = 32, hi = 8192;
  if (fixed + subtree_point_bytes(lo, d) > sh.smem) return 0;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (fixed + subtree_point_bytes(mid, d) <= sh.smem) lo = mid; else hi = mid - 1;
  }
  return std::min(lo & ~31, sh.q * sh.threads);
}
inline int subtree_capacity(int d) { return subtree_capacity(d, subtree_shape(d)); }

// Subset counts of a small root (put in subset order by the subtree kernel)
// live in the warp histograms: trees with more subsets presort their root in
// the multi-CTA pipeline instead.
inline bool subtree_sorts_root(int r) { return r <= kSubtreeHistWords; }

// The tuning of the select paths (kdt_tuning, validated) in force when a level
// step starts.
struct SelectTuning {
  uint32_t tiny_max, bitonic_max, warp_max;
  int cta_threads, digit_bits;
};
SelectTuning current_tuning();

// A tree that joins the engine: what a kernel writes into its tables.
struct AdmitRec {
  TreeDev tree;
  uint32_t slot;
  uint32_t terminal;  // the root is a leaf
  Cell* root_dst;     // else: its entry of a cell list
  uint32_t tile0, seg0;  // and where a big root's tiles and segments start
};
constexpr uint32_t kAdmitIota = 65536;  // larger terminal roots get their identity permutation from a launch of their own
constexpr int kAdmitFew = 8;            // records that travel as launch parameters (below 4 KB)
struct AdmitFew {
  AdmitRec rec[kAdmitFew];
};
static_assert(sizeof(AdmitFew) <= 4000, "launch parameters");
// staging: device memory for recs.size() records (more than kAdmitFew only)
cudaError_t launch_admit(const std::vector<AdmitRec>& recs, AdmitRec* staging, TreeDev* trees, cudaStream_t st);

cudaError_t prepare_step_kernels();
// Whether a step of nseg segments of so many points gets a CTA for each (StepDev::few_segs).
bool step_selects_all(uint32_t nseg, uint64_t points, uint32_t sms);
// ... or several CTAs for its large segments (StepDev::wide_segs).
bool step_selects_wide(uint32_t nseg, uint64_t points);
// One thread: the loop condition of a graph whose body is a pair of level
// steps (keep going while ncells_next > 0, at most `limit` iterations; the
// count of iterations is kept in *iters).
void launch_loop_cond(cudaGraphConditionalHandle h, const uint32_t* ncells_next, uint32_t* iters, uint32_t limit,
                      cudaStream_t st);
void launch_big_step(const TreeDev* trees, const StepDev& s, uint32_t max_tiles, uint32_t nseg,
                     uint32_t max_bigseg, bool has_roots, bool need_root_dims, bool any_widest, int max_r, int uniform_d,
                     const SelectTuning& tune, uint64_t points, uint32_t sms, cudaStream_t st, bool fourier = false);

// Most dynamic shared memory of the staged scatter: three CTAs per SM with
// their static part and the kilobyte that each one reserves.
constexpr uint32_t kScatterSmemBytes = 74240;
constexpr uint32_t kScatterLargeSmemBytes = 112640;  // and two CTAs per SM
cudaError_t prepare_scatter_kernel(int uniform_d, bool any_widest);
// uniform_d: the coordinate count of every tree of the step, 0 if they differ
// (a kernel compiled for that d is used where there is one)
void launch_scatter(const TreeDev* trees, const StepDev& s, uint32_t max_tiles, uint32_t sms, uint64_t points,
                    int uniform_d, bool any_widest, cudaStream_t st);

// Sharded build (kdt_shard.cu): the per-level exchanges among the shards of
// a step whose StepDev has shards > 0 (ncells_cap bounds the step's cells).
void launch_shard_index(const StepDev& s, uint32_t ncells_cap, cudaStream_t st);
void launch_shard_medians(const TreeDev* trees, const StepDev& s, uint32_t ncells_cap, cudaStream_t st);
void launch_shard_minmax(const TreeDev* trees, const StepDev& s, uint32_t ncells_cap, cudaStream_t st);

cudaError_t prepare_subtree_kernel();
// One launch of the subtree kernel in the given shape over a queue of small
// cells. count_dev: if set, the device word holding the queue's length
// (count is then its cap). reversed: the queue is filled from the end of the
// list (item j at list[count_cap - 1 - j], count_cap = count). small_off: the
// cells' rows of subset offsets.
void launch_subtree(const SubtreeShape& sh, const TreeDev* trees, const Cell* list, uint32_t count,
                    const uint32_t* count_dev, bool reversed, const uint32_t* small_off, uint32_t* head,
                    LCell* slices, uint32_t slice_cells, uint32_t grid, uint64_t points, cudaStream_t st);

void launch_iota(uint32_t* out, uint32_t n, cudaStream_t st);

// CTAs of the kernels that walk the terminal records of several trees. One
// tree (slots null: slot 0) has all of them; else slots[0, n) are the trees
// and CTAs [first[i], first[i + 1]) work on the i-th, first = slots + n.
constexpr uint32_t kChunkRecords = 32;  // records per CTA that the counts aim at
struct SlotChunks {
  const uint32_t* slots;
  uint32_t nslots, chunks;
};
__device__ __forceinline__ uint32_t pick_chunk(const SlotChunks& sc, uint32_t* chunk, uint32_t* chunks) {
  if (!sc.slots) {
    *chunk = blockIdx.x;
    *chunks = gridDim.x;
    return 0;
  }
  const uint32_t* first = sc.slots + sc.nslots;
  uint32_t lo = 0, hi = sc.nslots;
  while (hi - lo > 1u) {
    const uint32_t mid = (lo + hi) / 2u;
    if (first[mid] <= blockIdx.x) lo = mid; else hi = mid;
  }
  *chunk = blockIdx.x - first[lo];
  *chunks = first[lo + 1u] - first[lo];
  return sc.slots[lo];
}

// Leaf sort (kdt_leafsort.cu): terminal cells up to kLeafWarpMax points are
// sorted by one warp, up to kLeafBlockMax by one CTA; larger ones are listed
// in the tree's `huge` table and sorted by leaf_sort_huge.
constexpr int kLeafWarpMax = 256;
constexpr int kLeafBlockMax = 4096;
void launch_leaf_sort(const TreeDev* trees, const SlotChunks& sc, cudaStream_t st);
// Host view of a finished tree for the global leaf-sort passes: the
// permutation, a ping-pong buffer of n words and scratch for tile tables
// (the tree's working buffers, free once its build is done).
struct TreeHost {
  uint64_t n = 0;
  uint32_t* out_perm = nullptr;
  uint32_t* keys = nullptr;
  void* scratch = nullptr;
  size_t scratch_bytes = 0;
  const uint32_t* huge = nullptr;   // device: the records listed for the global passes
  uint32_t huge_cap = 0;
  const TermRec* terms = nullptr;   // device
  uint32_t term_cap = 0;
};
cudaError_t leaf_sort_huge(const TreeHost& th, const std::vector<TermRec>& recs, cudaStream_t st);

}  // namespace kdt

#include "kdt.h"

namespace kdt {

// Fault injection (kdt_fault.cu): true if an injected failure of this kind
// (a kdt_fault value) is due now; it is then consumed.
bool fault_take(int kind);
// The library's device allocations go through here (an injected
// KDT_FAULT_ALLOC fails it without calling cudaMalloc).
cudaError_t dev_malloc(void** p, size_t bytes);

kdt_status build_in_workspace(const float* points, const kdt_params* p, void* workspace, size_t workspace_bytes,
                              uint32_t* out_perm, float* out_split_vals, int8_t* out_split_dims,
                              int64_t* out_node_offsets, int32_t* out_levels, cudaStream_t st);

void launch_finalize_many(const TreeDev* trees, const SlotChunks& sc, cudaStream_t st);

}  // namespace kdt
