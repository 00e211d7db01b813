// kdt_engine.h -- host-side driver shared by the plain, batched and served
// builds.
//
// The engine owns the tables of one "forest": up to max_trees trees, each in
// its own slot, whose cells are split together. One tick is one level step of
// the multi-CTA pipeline over every big cell of every tree in flight (each
// tree at its own level), followed by the subtree kernel over every cell that
// became small during the tick. A tree's cells never mix with another tree's
// data; trees join (admit) and leave (finalize) between ticks.
#pragma once
#include <cstddef>
#include <cstdint>
#include <vector>

#include <cuda_runtime.h>

#include "kdt.h"
#include "kdt_launch.h"

namespace kdt {

kdt_status validate_params(const kdt_params* p);
// The parameters a build runs with: a Fourier-estimator build ignores the
// subsets (one subset, no ids), since its statistics are sums.
kdt_params effective_params(const kdt_params& p);

// Memory of one tree (offsets relative to the tree's base, 256-byte aligned).
struct TreePlan {
  int L_cap = 0;
  int small_max = 0;
  int sid_bytes = 0;
  bool sub_wide = false;   // small cells run in the subtree kernel's wide shape
  int sub_tall = 0;        // > 0: in its tall shape, by at most this many CTAs
  int steps = 0;           // level steps that have cells whatever the points are
  bool presorted = false;  // root split by the pipeline, reordered by subset first
  bool leafsort = false;   // subsets not in index order: leaves are sorted at the end
  uint64_t n = 0;
  uint64_t term_cap = 0;
  uint64_t huge_cap = 0;  // terminal cells larger than one CTA's leaf sort
  uint64_t slice_cells = 0;  // a level's cells of one small cell
  uint64_t maxB = 0;      // big cells at one level
  uint64_t cap_small = 0; // small cells over the whole build
  size_t xbuf[2] = {0, 0}, pbuf[2] = {0, 0}, terms = 0, root_off = 0, root_cur = 0,
         huge = 0;
  size_t bytes = 0;
};
// no_subtree: every cell stays in the multi-CTA pipeline (a sharded build's
// trees, whose splits are exchanged level by level). alone: no other tree is
// built with this one.
TreePlan plan_tree(const kdt_params& p, bool no_subtree = false, bool alone = false);

// Capacities of the shared tables, accumulated over the trees they must serve
// at the same time.
struct StepNeeds {
  uint64_t points = 0, maxB = 0, cap_small = 0, nseg = 0, small_off = 0;
  uint32_t max_trees = 0, slice_cells = 0;
  int sub_tall = 0;  // the forest's one tree uses the subtree kernel's tall shape
  bool widest = false;
  bool fourier = false;  // a tree splits by the Fourier-moment estimator
  int max_d = 1, min_d = 1 << 30;  // min_d == max_d: every tree has the same d
  int max_r = 1;                   // the largest subset count: segments per cell
  void add(const kdt_params& p, const TreePlan& tp);
};

struct StepPlan {
  StepNeeds needs;
  // grid_step: the grid scale of the level step's kernels (two per SM);
  // sms: the device's SMs (the subtree kernel's grid is sms x its shape's CTAs,
  // or sub_tall)
  uint32_t maxB = 0, cap_small = 0, max_tiles = 0, nseg_cap = 0, bigseg_cap = 0, grid_step = 0, sms = 0, off_cap = 0,
           small_off_cap = 0;
  size_t trees = 0, words = 0, slot_words = 0, slots_list = 0, admits = 0, big[2] = {0, 0}, small = 0, tiles = 0,
         tile_seg = 0, tile_left = 0, tile_loff = 0, tile_mm = 0, child_mm = 0, kdim = 0, mkey = 0, lcount = 0,
         seg_w = 0, seg_key = 0, seg_med = 0, bigseg = 0, midseg = 0, slices = 0, off[2] = {0, 0}, obase[2] = {0, 0},
         small_off = 0, crow = 0;
  size_t bytes = 0;
};
StepPlan plan_step(const StepNeeds& needs);

class Engine {
 public:
  Engine(const StepPlan& plan, uint8_t* base, cudaStream_t st);

  // Clear every counter (call once before the first admit).
  kdt_status reset();
  // Make the forest's trees 0..shards-1 the shards of one tree (see
  // StepDev::shards); the tables are device memory of the caller.
  void set_sharding(uint32_t shards, uint32_t span, uint32_t* idx, uint32_t* wcount, uint32_t* mm_tmp) {
    s_.shards = shards;
    s_.shard_span = span;
    s_.shard_idx = idx;
    s_.wcount = wcount;
    s_.mm_tmp = mm_tmp;
  }
  // Put a tree into `slot`. tree_base holds TreePlan::bytes of device memory.
  kdt_status admit(uint32_t slot, const float* points, const kdt_params& p, const TreePlan& tp, uint8_t* tree_base,
                   uint32_t* out_perm, float* out_vals, int8_t* out_dims, int64_t* out_offs);
  // One tick (see above). Synchronises the stream once.
  kdt_status tick();
  // True while some cell of some tree still waits for a tick.
  bool busy() const { return big_count_ > 0 || small_count_ > 0 || small_count_w_ > 0; }
  // Slots (among `slots`) whose trees have no cell left.
  kdt_status done_slots(const std::vector<uint32_t>& slots, std::vector<uint32_t>* done);
  // Offsets and sentinels of finished trees, then their status and L.
  kdt_status finalize(const std::vector<uint32_t>& slots, std::vector<kdt_status>* status,
                      std::vector<int32_t>* levels);
  // Run ticks until nothing is left in flight. (Of a forest of one tree, the
  // steps that are sure to have cells are launched without waiting for any;
  // finalize() looks whether they were all.)
  kdt_status run_to_completion();
  // The same with one graph launch: the first tick (new roots) from the
  // host, then every later tick inside a CUDA graph whose conditional while
  // node repeats a pair of recorded ticks until no cell is left.
  kdt_status run_graph();
  // Iterations (pairs of ticks) of the last run_graph.
  uint32_t graph_iters() const { return graph_iters_; }

 private:
  StepPlan plan_;
  uint8_t* base_;
  cudaStream_t st_;
  TreeDev* trees_ = nullptr;      // device [max_trees]
  uint32_t* words_ = nullptr;     // device engine words
  uint32_t* slot_words_ = nullptr;  // device [5][max_trees]: term_count, status, levels, live, huge_count
  uint32_t* slots_list_ = nullptr;  // device [2 max_trees + 1]: SlotChunks
  Cell* big_[2] = {nullptr, nullptr};
  uint32_t* off_[2] = {nullptr, nullptr};
  uint32_t* obase_[2] = {nullptr, nullptr};
  Cell* small_ = nullptr;
  LCell* slices_ = nullptr;
  StepDev s_{};
  int cur_ = 0;
  uint32_t big_count_ = 0, small_count_ = 0, small_count_w_ = 0;  // small: front (narrow), back (wide)
  uint32_t big_tiles_ = 0, big_segs_ = 0;  // of the big cells
  uint64_t big_points_ = 0, small_points_ = 0;
  bool root_dims_ = false;
  bool debug_ = false;
  uint32_t graph_iters_ = 0;
  int ahead_ = 0;            // the one tree's steps to launch without waiting
  bool ahead_wide_ = false;  // its small cells run in the wide shape
  bool unsure_ = false;      // launched so; cells may be left
  // The launches of a step over the current list; s_ holds its counts.
  void launch_step(bool has_roots);
  kdt_status run_ahead();
  // What the device's words say of the current list.
  void read_big(const uint32_t* words);
  // Record a tick over cell list p into the stream's capture (counts on the device).
  kdt_status record_tick(int p);
  // The subtree kernel over the small-cell queue: the narrow (or tall) shape
  // over its front, the wide one over its back (host counts, or the device's).
  void launch_small();
  void launch_small_dev(int wide, uint32_t most);
  // Admitted trees whose records are not on the device yet, and the list
  // their root goes to.
  enum List { kListNone, kListBig, kListSmall, kListSmallWide };
  struct Pending {
    AdmitRec rec;
    List list;
  };
  kdt_status flush_admits(bool* has_big_roots);
  void use_lists(StepDev* s, int p);
  // The coordinate count of every tree of the forest, 0 if they differ.
  int uniform_d() const;
  std::vector<Pending> pending_;
  std::vector<AdmitRec> admitted_;  // the records of the last flush
  std::vector<TreeHost> host_;   // per slot: what the global leaf-sort passes need
  std::vector<uint32_t> recs_;   // per slot: terminal records to expect
  std::vector<uint8_t> sorts_;   // per slot: the tree's leaves are sorted
};

}  // namespace kdt
