// kdt_runs.h -- the runs of tiles whose sums the Fourier estimator writes down
// (host and device).
//
// A cell's tiles are cut into runs of the same number of tiles, from its first
// one on; a run is summed by one CTA, and a cell's runs are added in order. Where
// the cell stands in the step's tile list, and how many CTAs walk that list,
// changes neither the runs nor their sums, so an estimator's tree is a function of
// its points and parameters alone. (The places of a step's cells come from
// atomics: cutting the list into one range per CTA grouped a cell's tiles
// differently from call to call.)
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define KDT_RUNS_FN __host__ __device__ __forceinline__
#else
#define KDT_RUNS_FN inline
#endif

namespace kdt {

// Tiles of a run, for a tree of so many tiles: a tile while the root has at most
// kRootRuns of them (a CTA's share of the list is cut to whole runs, so they are
// kept short; a root's runs are added by one CTA, so they are kept few). With 2048,
// 4096 and 8192 kdt_build of 9,000,011 points, J = 31, twelve levels took 3.98, 3.89
// and 4.00 ms (3.91 with one range of the list per CTA), of 30,000,001, J = 8, ten
// levels 4.42, 4.40 and 4.51 (4.45).
constexpr uint32_t kRootRuns = 4096;
KDT_RUNS_FN uint32_t run_tiles(uint32_t tree_tiles) {
  return tree_tiles > kRootRuns ? (tree_tiles + kRootRuns - 1u) / kRootRuns : 1u;
}

// The first tile at or after `tile`, tile `index` of a cell of `tiles` tiles, that
// starts a run: of the cell, or of the one after it.
KDT_RUNS_FN uint32_t run_start(uint32_t tile, uint32_t index, uint32_t tiles, uint32_t len) {
  const uint32_t over = index % len;
  if (over == 0u) return tile;
  return tile + (len - over < tiles - index ? len - over : tiles - index);
}

}  // namespace kdt
