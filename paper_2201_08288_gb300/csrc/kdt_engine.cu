// kdt_engine.cu -- the forest engine (see kdt_engine.h).
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "kdt_engine.h"
#include "kdt_trace.h"

namespace kdt {

namespace {

constexpr size_t kAlign = 256;
inline size_t align_up(size_t x) { return (x + kAlign - 1) & ~(kAlign - 1); }

// Engine words.
// Per cell list (parity p): W_BIG + 2p its cells and, next to it, their
// segments; W_TILE + 2p their tiles and points; W_BIGSEG + p, W_MIDSEG + p the
// segment lists of the step over it. W_SMALL, W_SMALL + 1: the subtree queue's
// front and back. W_ITERS: the iterations of a graph-driven run.
enum Word {
  W_BIG = 0, W_TILE = 4, W_SMALL = 8, W_SMALLPTS = 10, W_SMALLOFF, W_BIGSEG = 12, W_MIDSEG = 14, W_HEAD = 16, W_ITERS,
  W_COUNT
};
// a graph-driven run's iterations (two level steps each) before it gives up
constexpr uint32_t kGraphIterMax = KDT_MAX_LEVELS + 4;
// Per-slot words: [which][max_trees].
enum SlotWord { S_TERM = 0, S_STATUS, S_LEVELS, S_LIVE, S_HUGE, S_COUNT };

int device_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return sms;
}

// The SMs that plans are made for.
int plan_sms() {
  const int sms = device_sms();
  return sms > 0 ? sms : 148;
}

kdt_status map_status(int32_t st) {
  switch (st) {
    case ST_OK: return KDT_OK;
    case ST_INVALID_ARG: return KDT_ERR_INVALID_ARG;
    case ST_NAN_INPUT: return KDT_ERR_NAN_INPUT;
    case ST_LEVEL_CAP: return KDT_ERR_LEVEL_CAP;
    case ST_CAPACITY: return KDT_ERR_CAPACITY;
    case ST_TIMEOUT: return KDT_ERR_TIMEOUT;
    default: return KDT_ERR_CUDA;
  }
}

#define ENGINE_TRY(expr)         \
  do {                           \
    if ((expr) != cudaSuccess) { \
      (void)cudaGetLastError();  \
      return KDT_ERR_CUDA;       \
    }                            \
  } while (0)

}  // namespace

kdt_status validate_params(const kdt_params* p) {
  if (!p) return KDT_ERR_INVALID_ARG;
  if (p->n < 0 || p->n > (int64_t)0xffffffffLL) return KDT_ERR_INVALID_ARG;
  if (p->d < 1 || p->d > KDT_MAX_DIMS) return KDT_ERR_INVALID_ARG;
  if (p->r < 1 || p->r > KDT_MAX_SUBSETS) return KDT_ERR_INVALID_ARG;
  if (p->key_rule != KDT_KEY_CYCLIC && p->key_rule != KDT_KEY_WIDEST_SPREAD) return KDT_ERR_INVALID_ARG;
  if (p->subset_mode != KDT_SUBSET_MOD && p->subset_mode != KDT_SUBSET_CONTIGUOUS &&
      p->subset_mode != KDT_SUBSET_EXPLICIT)
    return KDT_ERR_INVALID_ARG;
  if (p->subset_mode == KDT_SUBSET_EXPLICIT && p->n > 0 &&
      ((p->subset_id8 == nullptr) == (p->subset_id16 == nullptr)))
    return KDT_ERR_INVALID_ARG;
  if (p->depth < 0 || p->depth > KDT_MAX_LEVELS) return KDT_ERR_INVALID_ARG;
  if (p->depth == 0) {
    if (p->leaf_size < 1) return KDT_ERR_INVALID_ARG;
    if (p->max_levels < 0 || p->max_levels > KDT_MAX_LEVELS) return KDT_ERR_INVALID_ARG;
  }
  if (p->fourier_j < 0 || p->fourier_j > KDT_FOURIER_MAX_J) return KDT_ERR_INVALID_ARG;
  if (p->combine_rule != KDT_COMBINE_WEIGHTED && p->combine_rule != KDT_COMBINE_UNWEIGHTED)
    return KDT_ERR_INVALID_ARG;
  if (p->fourier_j > 0 && (p->key_rule != KDT_KEY_CYCLIC || p->depth == 0)) return KDT_ERR_INVALID_ARG;
  return KDT_OK;
}

kdt_params effective_params(const kdt_params& p) {
  kdt_params e = p;
  if (p.fourier_j > 0) {  // the estimator's sums do not depend on the subsets
    e.r = 1;
    e.subset_mode = KDT_SUBSET_MOD;
    e.subset_id8 = nullptr;
    e.subset_id16 = nullptr;
  }
  // one subset by index is one block: index order is subset order
  if (e.subset_mode == KDT_SUBSET_MOD && e.r == 1) e.subset_mode = KDT_SUBSET_CONTIGUOUS;
  return e;
}

TreePlan plan_tree(const kdt_params& p0, bool no_subtree, bool alone) {
  const kdt_params p = effective_params(p0);
  TreePlan t;
  const uint64_t n = (uint64_t)p.n;
  t.n = n;
  t.L_cap = p.depth > 0 ? p.depth : p.max_levels;
  // the estimator's splits come from the multi-CTA steps only (no subtree
  // kernel); its cells keep index order (no presort), so no leaf sort either
  const bool fourier = p.fourier_j > 0;
  t.small_max = (fourier || no_subtree) ? 0 : subtree_capacity(p.d);
  t.sub_wide = &subtree_shape(p.d) == &kSubWide;
  const uint64_t live_min = p.depth > 0 ? 1 : (uint64_t)p.leaf_size + 1;  // points of a cell that still splits
  // cells that one small cell of so many points can have on a level (the last
  // has none; a small cell is the root, or lies below a big one)
  auto slice_cells = [&](int points) {
    const uint64_t inner = (uint64_t)1 << std::max(t.L_cap - (n > (uint64_t)points ? 2 : 1), 0);
    return std::max<uint64_t>(32, std::min((uint64_t)points / live_min, inner));
  };
  if (t.small_max > 0 && alone && n > (uint64_t)t.small_max) {
    // the tall shape while its cells, of half its capacity to all of it, are no
    // more than the SMs (a single cell that the other shapes hold finishes sooner
    // there: 1000 points 50 us, 61 in the tall shape)
    const int tall = subtree_capacity(p.d, kSubTall);
    const uint64_t sms = (uint64_t)plan_sms();
    uint64_t cells = 1;
    while (cells <= sms && cells * (uint64_t)tall < n) cells *= 2;
    const uint64_t ctas = std::min<uint64_t>(sms, cells + cells / 4 + 1);
    // (and the cell tables of its levels take no more memory)
    if (cells <= sms && tall > t.small_max &&
        ctas * slice_cells(tall) <= sms * (uint64_t)subtree_shape(p.d).ctas * slice_cells(t.small_max)) {
      t.small_max = tall;
      t.sub_wide = false;
      t.sub_tall = (int)ctas;
    }
  }
  t.slice_cells = t.small_max > 0 ? slice_cells(t.small_max) : 0;
  t.sid_bytes = p.subset_mode == KDT_SUBSET_EXPLICIT ? (p.subset_id16 ? 2 : 1) : 0;
  const bool root_terminal = p.depth > 0 ? (n == 0) : (n <= (uint64_t)p.leaf_size);
  t.leafsort = !root_terminal && p.subset_mode != KDT_SUBSET_CONTIGUOUS && !fourier;
  // a small root is put in subset order by the subtree kernel itself, which
  // counts at most kSubtreeHistWords subsets
  t.presorted = t.leafsort && (n > (uint64_t)t.small_max || !subtree_sorts_root(p.r));
  // a level of 2^k cells of the n points has one of ceil(n / 2^k) or more
  const uint64_t ends = std::max<uint64_t>(t.small_max, p.depth > 0 ? 0 : (uint64_t)p.leaf_size);
  if (!root_terminal && (t.presorted || n > (uint64_t)t.small_max)) t.steps = 1;
  while (t.steps > 0 && t.steps < t.L_cap && ((n - 1) >> t.steps) + 1 > ends) ++t.steps;
  t.huge_cap = t.leafsort ? n / (uint64_t)(kLeafBlockMax + 1) + 1 : 0;
  // cells that still split are disjoint, lie above the last level and hold more
  // than leaf_size points (of a fixed depth: one or more)
  const uint64_t leaves = (uint64_t)1 << t.L_cap, inner = std::max<uint64_t>(leaves / 2, 1);
  t.maxB = std::min<uint64_t>(n / (uint64_t)(t.small_max + 1) + 1, inner);
  // (small ones are children of big ones, two each at most; or the root)
  const uint64_t parents = (uint64_t)t.L_cap * (n / (uint64_t)(t.small_max + 1)) + 1;
  t.cap_small = t.small_max > 0 ? std::min({n / live_min, inner, 2 * parents}) + 1 : 1;
  t.term_cap = leaves + 1;
  size_t off = 0;
  auto take = [&](size_t b) {
    const size_t o = off;
    off += align_up(b);
    return o;
  };
  for (int b = 0; b < 2; ++b) {
    t.xbuf[b] = take((size_t)p.d * n * 4);
    t.pbuf[b] = take(n * 4);
  }
  t.terms = take(t.term_cap * sizeof(TermRec));
  t.root_off = take(((size_t)p.r + 1) * 4);
  t.root_cur = take((size_t)p.r * 4);
  t.huge = take(t.huge_cap * 4);
  t.bytes = off;
  return t;
}

void StepNeeds::add(const kdt_params& p0, const TreePlan& tp) {
  const kdt_params p = effective_params(p0);
  fourier = fourier || p.fourier_j > 0;
  points += tp.n;
  maxB += tp.maxB;
  cap_small += tp.cap_small;
  nseg += tp.maxB * (uint64_t)p.r;
  // rows of subset offsets of the small cells (explicit ids): as many words as
  // two columns of the ids would take
  if (tp.small_max > 0) small_off += tp.n * (uint64_t)tp.sid_bytes / 2;
  max_trees += 1;
  slice_cells = std::max<uint32_t>(slice_cells, (uint32_t)tp.slice_cells);
  sub_tall = tp.sub_tall;
  widest = widest || p.key_rule == KDT_KEY_WIDEST_SPREAD;
  max_d = std::max(max_d, (int)p.d);
  max_r = std::max(max_r, (int)p.r);
  min_d = std::min(min_d, (int)p.d);
}

StepPlan plan_step(const StepNeeds& needs) {
  StepPlan s;
  s.needs = needs;
  const uint64_t clamp = 0xffffffffull;
  s.maxB = (uint32_t)std::min<uint64_t>(needs.maxB, clamp);
  s.cap_small = (uint32_t)std::min<uint64_t>(needs.cap_small, clamp);
  s.max_tiles = (uint32_t)std::min<uint64_t>(needs.points / kTile + needs.maxB + 1, clamp);
  s.nseg_cap = (uint32_t)std::min<uint64_t>(needs.nseg, clamp);
  s.off_cap = (uint32_t)std::min<uint64_t>(needs.nseg + needs.maxB, clamp);
  s.small_off_cap = (uint32_t)std::min<uint64_t>(needs.small_off, clamp);
  s.bigseg_cap = (uint32_t)std::min<uint64_t>(needs.points / (kSelWarpMin + 1) + 1, clamp);
  s.sms = (uint32_t)plan_sms();
  s.grid_step = s.sms * 2u;
  const uint32_t grid_sub_max =
      needs.sub_tall ? (uint32_t)needs.sub_tall : s.sms * (uint32_t)std::max(kSubNarrow.ctas, kSubWide.ctas);
  const uint32_t mt = std::max<uint32_t>(needs.max_trees, 1);
  size_t off = 0;
  auto take = [&](size_t b) {
    const size_t o = off;
    off += align_up(b);
    return o;
  };
  s.trees = take((size_t)mt * sizeof(TreeDev));
  s.words = take(W_COUNT * 4);
  s.slot_words = take((size_t)S_COUNT * mt * 4);
  s.slots_list = take(((size_t)mt * 2 + 1) * 4);  // SlotChunks
  s.admits = take(mt > (uint32_t)kAdmitFew ? (size_t)mt * sizeof(AdmitRec) : 0);
  s.big[0] = take((size_t)s.maxB * sizeof(Cell));
  s.big[1] = take((size_t)s.maxB * sizeof(Cell));
  s.small = take((size_t)s.cap_small * sizeof(Cell));
  s.tiles = take((size_t)s.max_tiles * sizeof(uint2));
  s.tile_seg = take((size_t)s.max_tiles * 4);
  s.tile_left = take((size_t)s.max_tiles * 4);
  s.tile_loff = take((size_t)s.max_tiles * 4);
  s.tile_mm = take(needs.widest || needs.fourier ? (size_t)s.max_tiles * kTileRecWords * 4 : 0);
  s.child_mm = take(needs.widest ? (size_t)s.maxB * 2 * kMaxDims * 2 * 4 : 0);
  s.kdim = take((size_t)s.maxB * 4);
  s.mkey = take((size_t)s.maxB * 4);
  s.lcount = take((size_t)s.maxB * 4);
  s.seg_w = take((size_t)s.nseg_cap * 4);
  s.seg_key = take((size_t)s.nseg_cap * 8);
  s.seg_med = take((size_t)s.nseg_cap * 4);
  s.bigseg = take((size_t)s.bigseg_cap * 4);
  s.midseg = take((size_t)s.nseg_cap * 4);
  s.slices = take((size_t)grid_sub_max * 2 * needs.slice_cells * sizeof(LCell));
  for (int b = 0; b < 2; ++b) {
    s.off[b] = take((size_t)s.off_cap * 4);
    s.obase[b] = take((size_t)s.maxB * 4);
  }
  s.small_off = take((size_t)s.small_off_cap * 4);
  s.crow = take((size_t)s.maxB * 2 * sizeof(uint2));
  s.bytes = off;
  return s;
}

Engine::Engine(const StepPlan& plan, uint8_t* base, cudaStream_t st) : plan_(plan), base_(base), st_(st) {
  const char* dbg = std::getenv("KDT_DEBUG");
  debug_ = dbg && *dbg && *dbg != '0';
  trees_ = (TreeDev*)(base + plan.trees);
  words_ = (uint32_t*)(base + plan.words);
  slot_words_ = (uint32_t*)(base + plan.slot_words);
  slots_list_ = (uint32_t*)(base + plan.slots_list);
  big_[0] = (Cell*)(base + plan.big[0]);
  big_[1] = (Cell*)(base + plan.big[1]);
  small_ = (Cell*)(base + plan.small);
  slices_ = (LCell*)(base + plan.slices);
  s_.tiles = (uint2*)(base + plan.tiles);
  s_.tiles_cap = plan.max_tiles;
  s_.nseg_cap = plan.nseg_cap;
  s_.kdim = (uint32_t*)(base + plan.kdim);
  s_.mkey = (uint32_t*)(base + plan.mkey);
  s_.lcount = (uint32_t*)(base + plan.lcount);
  s_.tile_mm = (uint32_t*)(base + plan.tile_mm);
  s_.child_mm = (uint32_t*)(base + plan.child_mm);
  s_.seg_w = (uint32_t*)(base + plan.seg_w);
  s_.seg_key = (const uint32_t**)(base + plan.seg_key);
  s_.seg_med = (uint32_t*)(base + plan.seg_med);
  s_.bigseg = (uint32_t*)(base + plan.bigseg);
  s_.midseg = (uint32_t*)(base + plan.midseg);
  s_.tile_seg = (uint32_t*)(base + plan.tile_seg);
  s_.tile_left = (uint32_t*)(base + plan.tile_left);
  s_.tile_loff = (uint32_t*)(base + plan.tile_loff);
  s_.small = small_;
  s_.small_ctr = (unsigned long long*)(words_ + W_SMALL);
  s_.small_cap = plan.cap_small;
  s_.next_big_cap = plan.maxB;
  s_.small_points = words_ + W_SMALLPTS;
  for (int b = 0; b < 2; ++b) {
    off_[b] = (uint32_t*)(base + plan.off[b]);
    obase_[b] = (uint32_t*)(base + plan.obase[b]);
  }
  s_.off_cap = plan.off_cap;
  s_.small_off = (uint32_t*)(base + plan.small_off);
  s_.small_off_used = words_ + W_SMALLOFF;
  s_.small_off_cap = plan.small_off_cap;
  s_.bigseg_cap = plan.bigseg_cap;
  s_.midseg_cap = plan.nseg_cap;
  s_.crow = (uint2*)(base + plan.crow);
  const uint32_t mt = std::max<uint32_t>(plan.needs.max_trees, 1);
  host_.assign(mt, TreeHost{});
  recs_.assign(mt, 0);
  sorts_.assign(mt, 0);
}

kdt_status Engine::reset() {
  ENGINE_TRY(prepare_subtree_kernel());
  ENGINE_TRY(prepare_scatter_kernel(uniform_d(), plan_.needs.widest));
  ENGINE_TRY(prepare_step_kernels());
  const uint32_t mt = std::max<uint32_t>(plan_.needs.max_trees, 1);
  // the engine words and, right behind them in the plan, the slots'
  ENGINE_TRY(cudaMemsetAsync(words_, 0, plan_.slot_words - plan_.words + (size_t)S_COUNT * mt * 4, st_));
  cur_ = 0;
  big_count_ = small_count_ = small_count_w_ = 0;
  big_tiles_ = big_segs_ = 0;
  big_points_ = small_points_ = 0;
  root_dims_ = unsure_ = false;
  ahead_ = 0;
  pending_.clear();
  return KDT_OK;
}

// Point a step's tables at cell list p and the other one.
void Engine::use_lists(StepDev* s, int p) {
  s->cells = big_[p];
  s->next_big = big_[p ^ 1];
  s->next_big_ctr = (unsigned long long*)(words_ + W_BIG + 2 * (p ^ 1));
  s->next_tile_ctr = (unsigned long long*)(words_ + W_TILE + 2 * (p ^ 1));
  s->bigseg_count = words_ + W_BIGSEG + p;
  s->bigseg_count_next = words_ + W_BIGSEG + (p ^ 1);
  s->midseg_count = words_ + W_MIDSEG + p;
  s->midseg_count_next = words_ + W_MIDSEG + (p ^ 1);
  s->off_cur = off_[p];
  s->obase_cur = obase_[p];
  s->off_next = off_[p ^ 1];
  s->obase_next = obase_[p ^ 1];
}

int Engine::uniform_d() const { return plan_.needs.min_d == plan_.needs.max_d ? plan_.needs.max_d : 0; }

kdt_status Engine::admit(uint32_t slot, const float* points, const kdt_params& p0, const TreePlan& tp,
                         uint8_t* tb, uint32_t* out_perm, float* out_vals, int8_t* out_dims, int64_t* out_offs) {
  const kdt_params p = effective_params(p0);
  const uint32_t mt = std::max<uint32_t>(plan_.needs.max_trees, 1);
  if (slot >= mt) return KDT_ERR_CAPACITY;
  TreeDev h{};
  h.n = p.n;
  h.d = p.d;
  h.r = p.r;
  h.subset_mode = p.subset_mode;
  h.key_rule = p.key_rule;
  h.depth = p.depth;
  h.leaf_size = p.leaf_size;
  h.max_levels = p.max_levels;
  h.fourier_j = p.fourier_j;
  h.combine_rule = p.combine_rule;
  h.sub_wide = tp.sub_wide ? 1 : 0;
  h.stall_limit = p.key_rule == KDT_KEY_CYCLIC ? p.d : 1;
  h.sid_bytes = tp.sid_bytes;
  h.small_max = tp.small_max;
  h.leafsort = tp.leafsort ? 1 : 0;
  h.presorted = tp.presorted ? 1 : 0;
  h.contig_mul = p.n > 0 ? ((uint64_t)p.r << 32) / (uint64_t)p.n : 0;
  h.x_in = points;
  h.sid_in = p.subset_id16 ? (const void*)p.subset_id16 : (const void*)p.subset_id8;
  for (int b = 0; b < 2; ++b) {
    h.xbuf[b] = (float*)(tb + tp.xbuf[b]);
    h.pbuf[b] = (uint32_t*)(tb + tp.pbuf[b]);
  }
  h.root_off = (uint32_t*)(tb + tp.root_off);
  h.root_cur = (uint32_t*)(tb + tp.root_cur);
  h.huge = (uint32_t*)(tb + tp.huge);
  h.huge_count = slot_words_ + (size_t)S_HUGE * mt + slot;
  h.huge_cap = (uint32_t)std::min<uint64_t>(tp.huge_cap, 0xffffffffull);
  h.out_perm = out_perm;
  h.out_vals = out_vals;
  h.out_dims = out_dims;
  h.out_offs = out_offs;
  h.terms = (TermRec*)(tb + tp.terms);
  h.term_cap = (uint32_t)std::min<uint64_t>(tp.term_cap, 0xffffffffull);
  h.term_count = slot_words_ + (size_t)S_TERM * mt + slot;
  h.status = (int32_t*)(slot_words_ + (size_t)S_STATUS * mt + slot);
  h.levels = (int32_t*)(slot_words_ + (size_t)S_LEVELS * mt + slot);
  h.live = (int32_t*)(slot_words_ + (size_t)S_LIVE * mt + slot);
  // after the build the tree's working buffers are free: the global leaf-sort
  // passes use pbuf[0] as their second buffer and xbuf[0] for tile tables
  host_[slot] = TreeHost{(uint64_t)p.n, out_perm, h.pbuf[0], (void*)h.xbuf[0], (size_t)p.d * p.n * 4, h.huge,
                         h.huge_cap, h.terms, h.term_cap};
  const uint64_t n = (uint64_t)p.n;
  const bool root_terminal = p.depth > 0 ? (n == 0) : (n <= (uint64_t)p.leaf_size);
  // terminal records to expect (sizes the launches that walk them; those take
  // any number): a complete tree's leaves, or about two per leaf_size points
  const uint64_t leaves = (uint64_t)1 << tp.L_cap;
  recs_[slot] = (uint32_t)(p.depth > 0 ? leaves : std::min<uint64_t>(leaves, 2 * n / (uint64_t)p.leaf_size + 2));
  sorts_[slot] = tp.leafsort ? 1 : 0;
  Pending pe;
  pe.rec = AdmitRec{h, slot, root_terminal ? 1u : 0u, nullptr, 0, 0};
  pe.list = root_terminal ? kListNone
            : !(n <= (uint64_t)tp.small_max && !tp.presorted) ? kListBig
            : tp.sub_wide ? kListSmallWide : kListSmall;
  if (pe.list == kListBig && p.key_rule == KDT_KEY_WIDEST_SPREAD) root_dims_ = true;
  if (mt == 1 && !s_.shards) {
    ahead_ = pe.list == kListBig ? tp.steps : 0;
    ahead_wide_ = tp.sub_wide;
  }
  pending_.push_back(pe);
  return KDT_OK;
}

// The admitted trees go to the device together: their records (one copy, or
// none for a few), then one kernel that writes every table entry they need.
kdt_status Engine::flush_admits(bool* has_big_roots) {
  *has_big_roots = false;
  if (pending_.empty()) return KDT_OK;
  std::vector<AdmitRec>& recs = admitted_;  // kept: the copy below may still read it when this returns
  recs.clear();
  recs.reserve(pending_.size());
  uint64_t big = 0, small = 0;
  for (const Pending& pe : pending_) {
    big += pe.list == kListBig;
    small += pe.list == kListSmall || pe.list == kListSmallWide;
  }
  if (big_count_ + big > plan_.maxB || (uint64_t)small_count_ + small_count_w_ + small > plan_.cap_small)
    return KDT_ERR_CAPACITY;
  for (Pending& pe : pending_) {
    const uint64_t n = (uint64_t)pe.rec.tree.n;
    if (pe.list == kListBig) {
      pe.rec.root_dst = big_[cur_] + big_count_++;
      pe.rec.tile0 = big_tiles_;
      pe.rec.seg0 = big_segs_;
      big_tiles_ += tiles_of((uint32_t)n);
      big_segs_ += (uint32_t)pe.rec.tree.r;
      big_points_ += n;
    } else if (pe.list == kListSmall) {
      pe.rec.root_dst = small_ + small_count_++;
      small_points_ += n;
    } else if (pe.list == kListSmallWide) {  // the back of the queue runs downwards
      pe.rec.root_dst = small_ + plan_.cap_small - 1 - small_count_w_++;
      small_points_ += n;
    }
    recs.push_back(pe.rec);
  }
  *has_big_roots = big > 0;
  pending_.clear();
  ENGINE_TRY(launch_admit(recs, (AdmitRec*)(base_ + plan_.admits), trees_, st_));
  return KDT_OK;
}

void Engine::launch_step(bool has_roots) {
  s_.few_segs = step_selects_all(s_.nseg, big_points_, plan_.sms) ? 1u : 0u;
  // (not for shards: one segment of a shard's cell is a part of the cell's)
  s_.wide_segs = !s_.shards && step_selects_wide(s_.nseg, big_points_) ? 1u : 0u;
  const SelectTuning tune = current_tuning();
  s_.tiny_max = tune.tiny_max;
  s_.bitonic_max = tune.bitonic_max;
  s_.warp_max = tune.warp_max;
  launch_big_step(trees_, s_, s_.ntiles, s_.nseg, plan_.bigseg_cap, has_roots, root_dims_, plan_.needs.widest,
                  plan_.needs.max_r, uniform_d(), tune, big_points_,
                  plan_.grid_step, st_, plan_.needs.fourier);
  root_dims_ = false;
}

void Engine::read_big(const uint32_t* w) {
  const uint32_t* wb = w + W_BIG + 2 * cur_;
  const uint32_t* wt = w + W_TILE + 2 * cur_;
  big_count_ = std::min(wb[0], plan_.maxB);
  big_segs_ = std::min(wb[1], plan_.nseg_cap);
  big_tiles_ = std::min(wt[0], plan_.max_tiles);
  big_points_ = wt[1];
}

// The steps of a tree built alone that have cells whatever its points are, and
// then the subtree kernel, without a wait: a step's grids are sized for the
// cells that halving gives at most, and its kernels read how many there are.
// (Waiting for the counts of each level and launching the next left the GPU idle
// for 10 to 17 us a level.)
kdt_status Engine::run_ahead() {
  bool has_roots = false;
  const kdt_status f = flush_admits(&has_roots);
  if (f != KDT_OK) return f;
  s_.init_small = s_.init_small_w = s_.init_small_points = 0;
  uint64_t cells = 1;  // of the step, at most
  for (int k = 0; k < ahead_; ++k) {
    use_lists(&s_, cur_);
    if (k > 0) {
      s_.ncells_dev = words_ + W_BIG + 2 * cur_;
      s_.nseg_dev = words_ + W_BIG + 2 * cur_ + 1;
      s_.ntiles_dev = words_ + W_TILE + 2 * cur_;
      s_.bounded = s_.keep_small = 1;
    }
    s_.ncells = (uint32_t)cells;
    s_.ntiles = (uint32_t)std::min<uint64_t>(k == 0 ? big_tiles_ : big_points_ / kTile + cells, plan_.max_tiles);
    s_.nseg = (uint32_t)std::min<uint64_t>(cells * (uint64_t)plan_.needs.max_r, plan_.nseg_cap);
    launch_step(has_roots && k == 0);
    ENGINE_TRY(cudaGetLastError());
    cur_ ^= 1;
    cells = std::min<uint64_t>(2 * cells, plan_.maxB);
  }
  s_.ncells_dev = s_.nseg_dev = s_.ntiles_dev = nullptr;
  s_.bounded = s_.keep_small = 0;
  // small cells: disjoint, none deeper than the steps
  const uint32_t most = (uint32_t)std::min<uint64_t>((uint64_t)1 << ahead_, plan_.cap_small);
  if (!plan_.needs.fourier) launch_small_dev(ahead_wide_ ? 1 : 0, most);
  ENGINE_TRY(cudaGetLastError());
  big_count_ = 0;
  unsure_ = true;
  ahead_ = 0;
  return KDT_OK;
}

kdt_status Engine::tick() {
  // new roots join the lists of this tick
  bool has_roots = false;
  const kdt_status f = flush_admits(&has_roots);
  if (f != KDT_OK) return f;

  if (big_count_ > 0) {
    s_.init_small = small_count_;
    s_.init_small_w = small_count_w_;
    s_.init_small_points = (uint32_t)small_points_;
    use_lists(&s_, cur_);
    s_.ncells = big_count_;
    s_.ntiles = std::min(big_tiles_, plan_.max_tiles);
    s_.nseg = std::min(big_segs_, plan_.nseg_cap);
    launch_step(has_roots);
    ENGINE_TRY(cudaGetLastError());
    uint32_t w[W_COUNT];
    ENGINE_TRY(cudaMemcpyAsync(w, words_, sizeof(w), cudaMemcpyDeviceToHost, st_));
    ENGINE_TRY(cudaStreamSynchronize(st_));
    if (debug_) {  // KDT_DEBUG=1: per-tick counts and raw tree statuses on stderr
      const uint32_t mt = std::max<uint32_t>(plan_.needs.max_trees, 1);
      std::vector<int32_t> stv(mt);
      ENGINE_TRY(cudaMemcpy(stv.data(), slot_words_ + (size_t)S_STATUS * mt, (size_t)mt * 4, cudaMemcpyDeviceToHost));
      std::fprintf(stderr, "kdt tick: big %u -> %u, small %u + %u\n", big_count_, w[W_BIG + 2 * (cur_ ^ 1)], w[W_SMALL],
                   w[W_SMALL + 1]);
      for (uint32_t k = 0; k < mt; ++k)
        if (stv[k]) std::fprintf(stderr, "kdt tick: slot %u status %d\n", k, stv[k]);
    }
    cur_ ^= 1;
    read_big(w);
    small_count_ = std::min(w[W_SMALL], plan_.cap_small);
    small_count_w_ = std::min(w[W_SMALL + 1], plan_.cap_small - small_count_);
    small_points_ = w[W_SMALLPTS];
  }
  if (small_count_ > 0 || small_count_w_ > 0) {
    launch_small();
    ENGINE_TRY(cudaGetLastError());
    small_count_ = small_count_w_ = 0;
    small_points_ = 0;
  }
  return KDT_OK;
}

// The queue with its counts on the device: the narrow (or tall) front, or the
// wide back walked from the end; it holds at most `most` cells.
void Engine::launch_small_dev(int wide, uint32_t most) {
  const SubtreeShape& sh = wide ? kSubWide : plan_.needs.sub_tall ? kSubTall : kSubNarrow;
  const uint32_t g = !wide && plan_.needs.sub_tall ? (uint32_t)plan_.needs.sub_tall : plan_.sms * (uint32_t)sh.ctas;
  launch_subtree(sh, trees_, wide ? small_ + (plan_.cap_small - most) : small_, most, words_ + W_SMALL + wide, wide != 0,
                 s_.small_off, words_ + W_HEAD, slices_, plan_.needs.slice_cells, std::min(g, most), 0, st_);
}

void Engine::launch_small() {
  const uint32_t cap = plan_.cap_small;
  const SubtreeShape& front = plan_.needs.sub_tall ? kSubTall : kSubNarrow;
  const uint32_t gn = plan_.needs.sub_tall ? (uint32_t)plan_.needs.sub_tall : plan_.sms * (uint32_t)front.ctas;
  const uint32_t gw = plan_.sms * (uint32_t)kSubWide.ctas;
  const uint64_t pts = small_points_;
  if (small_count_ > 0)
    launch_subtree(front, trees_, small_, small_count_, nullptr, false, s_.small_off, words_ + W_HEAD, slices_,
                   plan_.needs.slice_cells, std::min(gn, small_count_), pts, st_);  // the points of both
  if (small_count_w_ > 0)
    launch_subtree(kSubWide, trees_, small_ + cap - small_count_w_, small_count_w_, nullptr, false,
                   s_.small_off, words_ + W_HEAD, slices_, plan_.needs.slice_cells, std::min(gw, small_count_w_),
                   small_count_ ? 0 : pts, st_);
}

kdt_status Engine::done_slots(const std::vector<uint32_t>& slots, std::vector<uint32_t>* done) {
  const uint32_t mt = std::max<uint32_t>(plan_.needs.max_trees, 1);
  std::vector<int32_t> live(mt);
  ENGINE_TRY(cudaMemcpyAsync(live.data(), slot_words_ + (size_t)S_LIVE * mt, (size_t)mt * 4,
                             cudaMemcpyDeviceToHost, st_));
  ENGINE_TRY(cudaStreamSynchronize(st_));
  done->clear();
  for (uint32_t s : slots)
    if (s < mt && live[s] <= 0) done->push_back(s);
  return KDT_OK;
}

kdt_status Engine::finalize(const std::vector<uint32_t>& slots, std::vector<kdt_status>* status,
                            std::vector<int32_t>* levels) {
  const uint32_t mt = std::max<uint32_t>(plan_.needs.max_trees, 1);
  status->assign(slots.size(), KDT_OK);
  levels->assign(slots.size(), 0);
  if (slots.empty()) return KDT_OK;
  bool has_roots = false;  // trees that were terminal from the start may not have met a tick
  const kdt_status f = flush_admits(&has_roots);
  if (f != KDT_OK) return f;
  // offsets, sentinels and the leaves' order (trees with an error get none of
  // it: their outputs are undefined); the kernels read the trees' statuses and
  // record counts themselves, so nothing is waited for in between
  SlotChunks sc{nullptr, (uint32_t)slots.size(), 0};
  std::vector<uint32_t> list;
  if (slots.size() == 1 && slots[0] == 0) {
    // a warp per record, or a CTA where the leaves are larger than a warp sorts
    const uint32_t per = host_[0].n > (uint64_t)kLeafWarpMax * recs_[0] ? 1u : 8u;
    sc.chunks = std::max<uint32_t>(1, std::min<uint32_t>((recs_[0] + per - 1) / per, 8192));
  } else {
    list = slots;
    for (uint32_t s : slots) {
      list.push_back(sc.chunks);
      sc.chunks += std::max<uint32_t>(1, std::min<uint32_t>((recs_[s] + kChunkRecords - 1) / kChunkRecords, 2048));
    }
    list.push_back(sc.chunks);
    sc.slots = slots_list_;
    ENGINE_TRY(cudaMemcpyAsync(slots_list_, list.data(), list.size() * 4, cudaMemcpyHostToDevice, st_));
  }
  bool any_sort = false;
  for (uint32_t s : slots) any_sort = any_sort || sorts_[s];
  // the engine's words and, behind them in the plan, the slots'
  const size_t lead = unsure_ ? (plan_.slot_words - plan_.words) / 4 : 0;
  std::vector<uint32_t> words(lead + (size_t)S_COUNT * mt);
  for (;;) {
    launch_finalize_many(trees_, sc, st_);
    ENGINE_TRY(cudaGetLastError());
    if (any_sort) {
      launch_leaf_sort(trees_, sc, st_);
      ENGINE_TRY(cudaGetLastError());
    }
    ENGINE_TRY(cudaMemcpyAsync(words.data(), slot_words_ - lead, words.size() * 4, cudaMemcpyDeviceToHost, st_));
    ENGINE_TRY(cudaStreamSynchronize(st_));
    if (!unsure_) break;
    unsure_ = false;
    read_big(words.data());
    if (big_count_ == 0) break;
    // cells are left (unequal halves): the kernels above did nothing yet
    const kdt_status r = run_to_completion();
    if (r != KDT_OK) return r;
  }
  const uint32_t* sw = words.data() + lead;
  const uint32_t* tc = sw + (size_t)S_TERM * mt;
  const int32_t* st = (const int32_t*)sw + (size_t)S_STATUS * mt;
  const int32_t* lv = (const int32_t*)sw + (size_t)S_LEVELS * mt;
  const uint32_t* huge = sw + (size_t)S_HUGE * mt;
  for (uint32_t s : slots) {  // leaves too large for one CTA (shallow trees, cells that stop splitting)
    const TreeHost& h = host_[s];
    const uint32_t nh = std::min(huge[s], h.huge_cap);
    if (nh == 0 || st[s] != ST_OK) continue;
    std::vector<uint32_t> idx(nh);
    std::vector<TermRec> all(std::min(tc[s], h.term_cap)), recs;
    ENGINE_TRY(cudaMemcpyAsync(idx.data(), h.huge, (size_t)nh * 4, cudaMemcpyDeviceToHost, st_));
    ENGINE_TRY(cudaMemcpyAsync(all.data(), h.terms, all.size() * sizeof(TermRec), cudaMemcpyDeviceToHost, st_));
    ENGINE_TRY(cudaStreamSynchronize(st_));
    for (uint32_t k : idx)
      if (k < all.size()) recs.push_back(all[k]);
    ENGINE_TRY(leaf_sort_huge(h, recs, st_));
    ENGINE_TRY(cudaStreamSynchronize(st_));
  }
  for (size_t i = 0; i < slots.size(); ++i) {
    (*status)[i] = map_status(st[slots[i]]);
    (*levels)[i] = lv[slots[i]];
  }
  return KDT_OK;
}

kdt_status Engine::record_tick(int p) {
  StepDev sd = s_;
  sd.init_small = sd.init_small_w = sd.init_small_points = 0;
  use_lists(&sd, p);
  sd.ncells = plan_.maxB;  // capacities: the counts are the device words
  sd.ncells_dev = words_ + W_BIG + 2 * p;
  sd.nseg_dev = words_ + W_BIG + 2 * p + 1;
  sd.ntiles_dev = words_ + W_TILE + 2 * p;
  sd.few_segs = sd.wide_segs = 0;
  const SelectTuning tune = current_tuning();
  sd.tiny_max = tune.tiny_max;
  sd.bitonic_max = tune.bitonic_max;
  sd.warp_max = tune.warp_max;
  launch_big_step(trees_, sd, plan_.max_tiles, plan_.nseg_cap, plan_.bigseg_cap, false, false, plan_.needs.widest,
                  plan_.needs.max_r, uniform_d(), tune, 0,
                  plan_.grid_step, st_, plan_.needs.fourier);
  ENGINE_TRY(cudaGetLastError());
  launch_small_dev(0, plan_.cap_small);
  launch_small_dev(1, plan_.cap_small);
  ENGINE_TRY(cudaGetLastError());
  return KDT_OK;
}

kdt_status Engine::run_graph() {
  // the roots' step (presort, root dims) is sized and launched by the host
  if (!pending_.empty()) {
    const kdt_status s = tick();
    if (s != KDT_OK) return s;
  }
  if (!busy()) return KDT_OK;
  // every later step runs inside one graph launch: a while loop whose body is
  // a step over list p0 then one over list p0 ^ 1, each reading its count
  // from the device, until a step leaves no cell (the tick above has
  // launched the subtree kernel over its queue, so that queue is empty)
  const int p0 = cur_;
  // (the tick above left the list's counts in their device words)
  ENGINE_TRY(cudaMemsetAsync(words_ + W_ITERS, 0, 4, st_));
  // the steps are recorded on a private stream (the caller's may be the
  // legacy default stream, which cannot be captured); the graph runs on the
  // caller's stream
  struct Graphs {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ex = nullptr;
    cudaStream_t cs = nullptr;
    ~Graphs() {
      if (ex) cudaGraphExecDestroy(ex);
      if (g) cudaGraphDestroy(g);
      if (cs) cudaStreamDestroy(cs);
    }
  } gr;
  auto fail = [&](const char* what, cudaError_t e) {
    (void)cudaGetLastError();
    if (debug_) std::fprintf(stderr, "kdt graph run: %s: %s\n", what, cudaGetErrorString(e));
    return KDT_ERR_CUDA;
  };
  cudaError_t e;
  if ((e = cudaStreamCreateWithFlags(&gr.cs, cudaStreamNonBlocking)) != cudaSuccess) return fail("stream", e);
  if ((e = cudaGraphCreate(&gr.g, 0)) != cudaSuccess) return fail("graph", e);
  cudaGraphConditionalHandle h;
  if ((e = cudaGraphConditionalHandleCreate(&h, gr.g, 1, cudaGraphCondAssignDefault)) != cudaSuccess)
    return fail("conditional handle", e);
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t loop;
  if ((e = cudaGraphAddNode(&loop, gr.g, nullptr, nullptr, 0, &cp)) != cudaSuccess) return fail("while node", e);
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  if ((e = cudaStreamBeginCaptureToGraph(gr.cs, body, nullptr, nullptr, 0, cudaStreamCaptureModeThreadLocal)) !=
      cudaSuccess)
    return fail("begin capture", e);
  const cudaStream_t caller = st_;
  st_ = gr.cs;
  const uint64_t l0 = kdt_launch_count();
  kdt_status rec = record_tick(p0);
  if (rec == KDT_OK) rec = record_tick(p0 ^ 1);
  if (rec == KDT_OK) launch_loop_cond(h, words_ + W_BIG + 2 * p0, words_ + W_ITERS, kGraphIterMax, st_);
  const uint64_t per_iter = kdt_launch_count() - l0;
  st_ = caller;
  cudaGraph_t captured = nullptr;
  const cudaError_t ce = cudaStreamEndCapture(gr.cs, &captured);
  if (rec != KDT_OK) return rec;
  if (ce != cudaSuccess) return fail("end capture", ce);
  if ((e = cudaGetLastError()) != cudaSuccess) return fail("recording", e);
  if ((e = cudaGraphInstantiate(&gr.ex, gr.g, 0)) != cudaSuccess) return fail("instantiate", e);
  if ((e = cudaGraphLaunch(gr.ex, st_)) != cudaSuccess) return fail("launch", e);
  uint32_t fin[W_COUNT];
  ENGINE_TRY(cudaMemcpyAsync(fin, words_, sizeof(fin), cudaMemcpyDeviceToHost, st_));
  ENGINE_TRY(cudaStreamSynchronize(st_));
  const uint32_t iters = fin[W_ITERS];
  if (iters > 1) trace_add_launches((uint64_t)(iters - 1) * per_iter);  // replays beyond the recorded one
  graph_iters_ = iters;
  if (fin[W_BIG + 2 * p0] != 0) return KDT_ERR_CUDA;  // stopped at the iteration cap with cells left
  big_count_ = small_count_ = small_count_w_ = 0;
  big_points_ = small_points_ = 0;
  return KDT_OK;
}

kdt_status Engine::run_to_completion() {
  // (a traced launch states its points, which only the host's counts tell)
  if (ahead_ > 0 && !trace_enabled()) return run_ahead();
  for (int guard = 0; busy() || !pending_.empty(); ++guard) {
    if (guard > 2 * KDT_MAX_LEVELS + 4) return KDT_ERR_CUDA;
    const kdt_status s = tick();
    if (s != KDT_OK) return s;
  }
  return KDT_OK;
}

}  // namespace kdt
