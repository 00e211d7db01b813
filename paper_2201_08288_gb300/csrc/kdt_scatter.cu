// kdt_scatter.cu -- the stable partition of one level, with its loads staged
// through shared memory by the bulk-copy (TMA) engine and a producer warp.
//
// For every tile of a big cell (paper, Sec. 2: after a cell's split, its
// points go to the two children; ties go left), in sub-tiles of T points:
//   producer warp (warp 8): waits until one of two shared-memory buffers is
//     free ("empty" mbarrier), writes the sub-tile's metadata (output
//     pointers, which children are terminal, what to compute), raises the
//     buffer's expected byte count, starts bulk copies (cp.async.bulk) of
//     the aligned middle of every coordinate column and of the permutation,
//     copies the ragged 16-byte edges (4-byte cp.async) and arrives on the
//     buffer's "full" mbarrier; the next tile's record is loaded one tile
//     ahead;
//   consumer warps (0-7): wait for "full" (bounded), compute each point's
//     left/right flag from its key and its rank by warp ballots in position
//     order (so the partition is stable), store every value straight from
//     shared memory to its destination, two columns at a time, and release
//     the buffer.
// A child that is terminal receives only its permutation, in out_perm. For
// widest spread the consumers also reduce each child's min and max key per
// coordinate (per warp, then one shared-memory reduction per warp and
// column, fire-and-forget). Points of a cell arrive in subset order
// (contiguous segments), and a stable partition keeps that order in both
// children: a segment that starts at position p of the cell starts in the
// left child at the number of left points before p, in the right child at p
// minus that. So the children's subset offset tables come from the cell's own
// table, one thread per segment start of the sub-tile, and no subset id moves
// with the points. (Finding the starts by comparing neighbouring points'
// subsets, ids staged and stored as one more column or computed from the
// permutation by a division per point, took 33.1 instead of 26.8 ms per build
// of 2^27 points with d = 8 and 256 explicit subsets; the bytes alone, 72
// against 74 per point and level, are 25.9 ms at 6.8 TB/s.)
#include <algorithm>
#include <type_traits>

#include "kdt_internal.cuh"
#include "kdt_launch.h"
#include "kdt_ptx.cuh"
#include "kdt_trace.h"

namespace kdt {

namespace {

constexpr int kCW = 8;                // consumer warps
constexpr int kCT = kCW * 32;         // consumer threads
constexpr int kST = kCT + 32;         // + one producer warp
constexpr uint32_t kConsumerBar = 1;  // named barrier of the consumer warps

// Words of one staged column of T points (room for the alignment phase).
__host__ __device__ constexpr uint32_t col_stride(uint32_t T) { return T + 4u; }

// Bytes of the two buffers for d coordinate columns and the permutation.
__host__ __device__ constexpr uint32_t buf_bytes(int d, uint32_t T) { return (uint32_t)(d + 1) * col_stride(T) * 4u; }

// The instances: one for d = 1 to 8, 12 and 16 each, one for steps whose trees all
// have another d, and one for trees of mixed d.
constexpr int kMixedD = 0, kOtherD = -1;

// Dynamic shared memory of two buffers at most.
__host__ __device__ constexpr uint32_t most_smem(int kD) { return kD == kOtherD ? kScatterLargeSmemBytes : kScatterSmemBytes; }

// Points of which two buffers in so many bytes have room, at most 1024.
__host__ __device__ constexpr uint32_t sub_tile_room(int d, uint32_t smem) {
  const uint32_t most = smem / 8u / (uint32_t)(d + 1) - 4u;
  return most < 1024u ? most : 1024u;
}
// Points of a sub-tile. An instance for one d gives every consumer thread the
// same number of them: a power of two. The others take as few equal parts of a
// tile as have room, in whole warps: how many points are in flight bounds them,
// and a power of two would leave up to half of the buffers empty. kdt_build of
// 2,000,003 points, 64 subsets, leaves of 64, widest spread, at d = 9, 23, 40 and
// 64: 1.86, 4.51, 11.6 and 18.1 ms with a power of two and three CTAs per SM, 1.70,
// 3.81, 8.6 and 18.1 with parts of a tile, 1.54, 3.14, 6.5 and 13.8 with parts, two
// CTAs and kScatterLargeSmemBytes each.
__host__ __device__ constexpr uint32_t sub_tile_one(int d) {
  uint32_t T = 1024;
  while (T > sub_tile_room(d, kScatterSmemBytes)) T >>= 1;
  return T;
}
__host__ __device__ constexpr uint32_t sub_tile_any(int d, uint32_t smem) {
  const uint32_t room = sub_tile_room(d, smem) / 32u * 32u, parts = ((uint32_t)kTile + room - 1u) / room;
  return ((uint32_t)kTile + 32u * parts - 1u) / (32u * parts) * 32u;
}
static_assert(sub_tile_any(kMaxDims, kScatterSmemBytes) >= 32u, "every d has a sub-tile");

// Resident CTAs per SM of an instance. A sub-tile costs its barriers, its scan
// and a round trip to L2 whatever it holds, so what bounds a launch of few
// columns is how many sub-tiles are in flight: at d = 3, 2^24 points and 14
// levels the scatter took 2.62 ms per build with two CTAs, 1.42 with three and
// 1.37 with four (0.18 per level at 6.8 TB/s would be 1.1). At d = 8 without
// min / max two buffers of nine columns fit three times; with them the
// accumulators take 94 registers, and three CTAs spill (28.0 against 26.8 ms
// per build of 2^27 points). The instance for mixed d takes
// 72 registers, so three CTAs too: a forest of 512 trees spent 2.38 ms in it
// with two CTAs of 100 KB each, 1.81 with three of 72.5.
constexpr int scatter_ctas(int kD, bool kMM) {
  if (((kD == 7 || kD == 8) && kMM) || kD == kOtherD) return 2;
  return kD >= 2 && kD <= 5 && !kMM ? 4 : 3;
}

// What the consumers need about the sub-tile in a buffer.
struct SubMeta {
  float* xout;           // coordinate columns of the next level
  uint32_t* pout;        // permutation of the next level
  uint32_t* out_perm;    // final permutation (terminal children)
  const uint32_t* off;   // the cell's subset offsets
  uint32_t* row[2];      // the children's subset offsets (null: none kept)
  int32_t* status;
  int64_t n;
  uint32_t cell_begin, cell_count, cell_idx, sub, mcnt, T, dim, mkey, L, loff, tile_start;
  uint32_t u0, u1;       // segment starts off[u0, u1) lie in this tile
  int32_t d;
  uint8_t term_left, term_right, want_mm, want_off, nan_check;
  uint8_t run_more;      // this CTA's next tile is of the same cell (its min / max run goes on)
  uint8_t pad1, pad2;
  uint32_t ph[kMaxDims + 1];  // alignment phase of each staged word column
};

// kD > 0: compiled for trees of kD coordinates (the column loops unroll); else
// any d. kMM: some tree of the step uses widest spread.
template <int kD, bool kMM>
__global__ void __launch_bounds__(kST, scatter_ctas(kD, kMM)) k_scatter_tma(const TreeDev* trees, StepDev s) {
  chain_wait();
  constexpr int kMaxItems = kD > 0 ? (int)(sub_tile_one(kD > 0 ? kD : 1) / kCT) : 4;  // points per consumer thread
  // words of a buffer (for any d: trees of several d may follow one another, so
  // the halves are fixed)
  constexpr uint32_t kBufWords =
      (kD > 0 ? buf_bytes(kD > 0 ? kD : 1, (uint32_t)(kMaxItems * kCT)) : most_smem(kD) / 2) / 4;
  extern __shared__ __align__(128) uint32_t sm[];
  __shared__ __align__(8) uint64_t full[2], empty[2];
  __shared__ SubMeta meta[2];
  __shared__ uint32_t wcnt[kMaxItems][kCW];
  __shared__ unsigned wbal[kMaxItems][kCW];   // each (round, warp) block's left flags
  __shared__ uint32_t tmm[2][kMaxDims][2];    // this CTA's run of tiles of one cell: per child,
                                              // min / max key per coordinate
  __shared__ uint32_t s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t ntiles = ntiles_of(s);
  // this CTA's contiguous range of tiles: consecutive tiles mostly share a
  // cell, so the per-cell min / max stay in the CTA for long runs
  const uint32_t t_begin = (uint32_t)(((uint64_t)blockIdx.x * ntiles) / gridDim.x);
  const uint32_t t_end = (uint32_t)(((uint64_t)(blockIdx.x + 1) * ntiles) / gridDim.x);
  for (int j = tid; j < 2 * kMaxDims * 2; j += kST) (&tmm[0][0][0])[j] = (j & 1) ? 0u : 0xffffffffu;
  if (tid == 0) {
    mbar_init(&full[0], 1);
    mbar_init(&full[1], 1);
    mbar_init(&empty[0], kCW);
    mbar_init(&empty[1], kCW);
    mbar_init_fence();
    s_fail = 0;
  }
  __syncthreads();

  if (warp == kCW) {
    // ================================================================ producer
    uint32_t ephase = 0u;  // bit b: parity of buffer b's next "empty" phase
    uint32_t k = 0;
    // the next tile's record and cell are loaded one tile ahead
    uint2 tl_next = t_begin < t_end ? s.tiles[t_begin] : make_uint2(0, 0);
    Cell c_next = s.cells[tl_next.x];
    for (uint32_t tile = t_begin; tile < t_end; ++tile) {
      const uint2 tl = tl_next;
      const Cell c = c_next;
      if (tile + 1 < t_end) {
        tl_next = s.tiles[tile + 1];
        c_next = s.cells[tl_next.x];
      }
      const bool run_more = tile + 1 < t_end && tl_next.x == tl.x;
      const TreeDev& tg = trees[c.tree];
      const int d = kD > 0 ? kD : tg.d, ncols = d + 1;
      const uint32_t T = kD > 0 ? (uint32_t)(kMaxItems * kCT) : sub_tile_any(d, most_smem(kD)), stride = col_stride(T);
      const uint32_t tend = min(tl.y + (uint32_t)kTile, c.count);
      const float* X = src_cols(tg, c.level);
      const uint32_t* P = src_perm(tg, c.level);
      const uint32_t dim = s.kdim[tl.x], mkey = s.mkey[tl.x], L = s.lcount[tl.x], loff = s.tile_loff[tile];
      const uint2 cr0 = s.crow[2 * tl.x], cr1 = s.crow[2 * tl.x + 1];
      const int child_stall = (c.count == L) ? c.stall + 1 : 0;
      const bool term_left = is_terminal(tg, L, c.level + 1, child_stall);
      const bool term_right = is_terminal(tg, c.count - L, c.level + 1, child_stall);
      // the children's rows of subset offsets: a big child's, or that of a
      // small one that has one (the Fourier estimator reads no segments: its
      // cells carry no offsets)
      auto row_of = [&](uint2 cr) -> uint32_t* {
        if (tg.fourier_j) return nullptr;
        if (cr.x != kNoRow) return s.off_next + cr.y;
        if (cr.y == kNoRow || tg.subset_mode != SUB_EXPLICIT) return nullptr;
        const uint32_t row = s.small[cr.y].row;
        return row == kNoRow ? nullptr : s.small_off + row;
      };
      uint32_t* const row0 = row_of(cr0);
      uint32_t* const row1 = row_of(cr1);
      const bool want_off = row0 || row1;
      uint32_t u0 = 0, u1 = 0;
      if (want_off) {
        u0 = s.tile_seg[tile];
        u1 = tl.y + (uint32_t)kTile < c.count ? min(s.tile_seg[tile + 1], (uint32_t)tg.r + 1u) : (uint32_t)tg.r + 1u;
      }
      for (uint32_t sub = tl.y; sub < tend; sub += T, ++k) {
        const int b = k & 1;
        if (k >= 2) {
          if (!mbar_wait_bounded(&empty[b], (ephase >> b) & 1u)) {
            if (lane == 0) atomicExch(&s_fail, 1u);
            return;
          }
          ephase ^= 1u << b;
        }
        if (s_fail) return;
        const uint32_t mcnt = min(T, tend - sub);
        const uint32_t g0 = c.begin + sub;
        SubMeta& m = meta[b];
        uint32_t* A = sm + (size_t)b * kBufWords;
        if (lane == 0) {
          m.xout = tg.xbuf[c.level & 1];
          m.pout = tg.pbuf[c.level & 1];
          m.out_perm = tg.out_perm;
          m.off = c.level == 0 ? tg.root_off : s.off_cur + s.obase_cur[tl.x];
          m.status = tg.status;
          m.n = tg.n;
          m.cell_begin = c.begin;
          m.cell_count = c.count;
          m.cell_idx = tl.x;
          m.sub = sub;
          m.mcnt = mcnt;
          m.T = T;
          m.dim = dim;
          m.mkey = mkey;
          m.L = L;
          m.loff = loff;
          m.tile_start = tl.y;
          m.row[0] = row0;
          m.row[1] = row1;
          m.u0 = u0;
          m.u1 = u1;
          m.d = d;
          m.term_left = term_left;
          m.term_right = term_right;
          m.want_mm = tg.key_rule == KEY_WIDEST && !(term_left && term_right);
          m.want_off = want_off;
          // the input's NaN check: the root's first pass over its columns (a
          // presorted root's presort checks them)
          m.nan_check = c.level == 0 && !tg.presorted;
          m.run_more = run_more;
        }
        uint32_t total = 0u;
        for (int c0 = 0; c0 < ncols; c0 += 32) {
          const int col = c0 + lane;
          uint32_t bytes = 0;
          if (col < ncols) {
            const uint32_t* src = col < d ? (const uint32_t*)(X + (int64_t)col * tg.n) : P;
            uint32_t ph = 0;
            if (src) {
              ph = (uint32_t)(((uintptr_t)(src + g0) >> 2) & 3u);
              const uint32_t a0 = min(g0 + ((4u - ph) & 3u), g0 + mcnt);
              bytes = ((g0 + mcnt - a0) & ~3u) * 4u;
            }
            m.ph[col] = ph;
          }
          total += __reduce_add_sync(0xffffffffu, bytes);
        }
        if (lane == 0) mbar_expect_tx(&full[b], total);
        __syncwarp();
        for (int c0 = 0; c0 < ncols; c0 += 32) {
          const int col = c0 + lane;
          if (col >= ncols) continue;
          const uint32_t* src = col < d ? (const uint32_t*)(X + (int64_t)col * tg.n) : P;
          if (!src) continue;  // level 0 without a presort: the identity permutation, filled below
          uint32_t* dst = A + (size_t)col * stride;
          const uint32_t ph = (uint32_t)(((uintptr_t)(src + g0) >> 2) & 3u);
          const uint32_t a0 = min(g0 + ((4u - ph) & 3u), g0 + mcnt);
          const uint32_t a1 = a0 + ((g0 + mcnt - a0) & ~3u);
          if (a1 > a0) bulk_g2s(dst + ph + (a0 - g0), src + a0, (a1 - a0) * 4u, &full[b]);
          for (uint32_t idx = g0; idx < a0; ++idx) cp_async4(dst + ph + (idx - g0), src + idx);
          for (uint32_t idx = a1; idx < g0 + mcnt; ++idx) cp_async4(dst + ph + (idx - g0), src + idx);
        }
        if (!P)
          for (uint32_t i = lane; i < mcnt; i += 32) A[(size_t)d * stride + i] = g0 + i;
        cp_async_mbar_arrive(&full[b]);  // this lane's edge copies count toward the phase
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[b]);
      }
    }
    return;
  }

  // ================================================================== consumers
  const unsigned lt_mask = (1u << lane) - 1u;
  uint32_t fphase = 0u;  // bit b: parity of buffer b's next "full" phase
  uint32_t lnext = 0, rnext = 0;
  bool saw_nan = false;
  // For a compile-time d of at most 8 every lane keeps the min / max of its
  // points per coordinate and child over the whole run of the cell's tiles
  // (registers), reduced over the warp once at the run's end; otherwise the
  // warps reduce after every sub-tile.
  constexpr bool kAcc = kMM && kD > 0 && kD <= 8;
  constexpr int kAD = kAcc ? kD : 1;
  const float inf = __int_as_float(0x7f800000);
  float acc[kAD][2][2];  // [coordinate][child][min, max]
#pragma unroll
  for (int l = 0; l < kAD; ++l)
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      acc[l][side][0] = inf;
      acc[l][side][1] = -inf;
    }
  uint32_t k = 0;
  for (uint32_t tile = t_begin; tile < t_end; ++tile) {
    for (bool more = true; more; ++k) {
      const int b = k & 1;
      // one consumer thread waits for the sub-tile (a waiting thread keeps
      // issuing try_wait); the named barrier parks the others and makes what
      // the copies wrote visible to them
      if (tid == 0 && !mbar_wait_bounded(&full[b], (fphase >> b) & 1u)) atomicExch(&s_fail, 1u);
      fphase ^= 1u << b;
      named_sync(kConsumerBar, kCT);
      if (s_fail) return;
      const SubMeta& m = meta[b];
      const int d = kD > 0 ? kD : m.d;
      const int64_t n = m.n;
      const uint32_t T = kD > 0 ? (uint32_t)(kMaxItems * kCT) : m.T, stride = col_stride(T);
      const uint32_t mcnt = m.mcnt, L = m.L;
      const uint32_t cbeg = m.cell_begin, ccount = m.cell_count;
      const uint32_t tend = min(m.tile_start + (uint32_t)kTile, ccount);
      const bool term_left = m.term_left, term_right = m.term_right;
      const bool want_mm = kMM && m.want_mm, want_off = m.want_off, nan_check = m.nan_check;
      // this thread's first segment start of the tile, loaded ahead of its use
      const uint32_t u_first = m.u0 + (uint32_t)tid;
      uint32_t u_pos = want_off && u_first < m.u1 ? __ldg(m.off + u_first) : 0xffffffffu;
      if (m.sub == m.tile_start) {
        lnext = cbeg + m.loff;
        rnext = cbeg + L + (m.tile_start - m.loff);
      }
      const uint32_t* A = sm + (size_t)b * kBufWords;

      // ---- flags and ranks (position order)
      bool left[kMaxItems];
      unsigned bal[kMaxItems];
      const uint32_t* keycol = A + (size_t)m.dim * stride + m.ph[m.dim];
      const uint32_t* pa = A + (size_t)d * stride + m.ph[d];
#pragma unroll
      for (int q = 0; q < kMaxItems; ++q) {
        const uint32_t i = tid + q * kCT;
        left[q] = i < mcnt && ord_key(__uint_as_float(keycol[i])) <= m.mkey;
        bal[q] = __ballot_sync(0xffffffffu, left[q]);
        if (lane == 0) {
          wcnt[q][warp] = __popc(bal[q]);
          wbal[q][warp] = bal[q];
        }
      }
      named_sync(kConsumerBar, kCT);
      // left points before each (round, warp) block: one scan over the at
      // most 32 block counts in position order
      static_assert(kMaxItems >= 1 && kMaxItems * kCW <= 32, "one lane per (round, warp) block");
      const uint32_t wv = lane < kMaxItems * kCW ? (&wcnt[0][0])[lane] : 0u;
      const uint32_t winc = warp_incl_scan(wv);
      const uint32_t wexc = winc - wv;
      const uint32_t nL = __shfl_sync(0xffffffffu, winc, 31);
      uint32_t dst[kMaxItems];
      bool keep[kMaxItems];  // the point's child is not terminal: its columns move
#pragma unroll
      for (int q = 0; q < kMaxItems; ++q) {
        const uint32_t i = tid + q * kCT;
        const uint32_t lr = __shfl_sync(0xffffffffu, wexc, q * kCW + warp) + __popc(bal[q] & lt_mask);
        dst[q] = left[q] ? lnext + lr : rnext + (i - lr);
        keep[q] = i < mcnt && !(left[q] ? term_left : term_right);
      }

      // ---- permutation
#pragma unroll
      for (int q = 0; q < kMaxItems; ++q) {
        const uint32_t i = tid + q * kCT;
        if (i >= mcnt) continue;
        if (keep[q])
          m.pout[dst[q]] = pa[i];
        else
          m.out_perm[dst[q]] = pa[i];
      }

      // ---- coordinate columns, two at a time, straight from shared memory
#pragma unroll
      for (int c = 0; c < d; c += 2) {
        const bool two = c + 1 < d;
        const uint32_t* a0 = A + (size_t)c * stride + m.ph[c];
        const uint32_t* a1 = two ? A + (size_t)(c + 1) * stride + m.ph[c + 1] : a0;
        float* o0 = m.xout + (int64_t)c * n;
        float* o1 = m.xout + (int64_t)(c + 1) * n;
        uint32_t v0[kMaxItems], v1[kMaxItems];
#pragma unroll
        for (int q = 0; q < kMaxItems; ++q) {
          const uint32_t i = tid + q * kCT;
          v0[q] = i < mcnt ? a0[i] : 0u;
          v1[q] = i < mcnt ? a1[i] : 0u;
        }
        if (nan_check)
#pragma unroll
          for (int q = 0; q < kMaxItems; ++q)
            saw_nan |= (tid + q * kCT < mcnt) &&
                       (is_nan_bits(__uint_as_float(v0[q])) || is_nan_bits(__uint_as_float(v1[q])));
#pragma unroll
        for (int q = 0; q < kMaxItems; ++q)
          if (keep[q]) {
            o0[dst[q]] = __uint_as_float(v0[q]);
            if (two) o1[dst[q]] = __uint_as_float(v1[q]);
          }
        if (want_mm && kAcc) {
          // min / max as floats (the widest rule only uses max - min, which -0
          // and +0 do not change); keys are formed at the run's end
          const int c1 = two ? c + 1 : c;
#pragma unroll
          for (int q = 0; q < kMaxItems; ++q)
            if (keep[q]) {
              const float x0 = __uint_as_float(v0[q]), x1 = __uint_as_float(v1[q]);
              const int side = left[q] ? 0 : 1;
              if (side == 0) {
                acc[c % kAD][0][0] = fminf(acc[c % kAD][0][0], x0);
                acc[c % kAD][0][1] = fmaxf(acc[c % kAD][0][1], x0);
                if (two) {
                  acc[c1 % kAD][0][0] = fminf(acc[c1 % kAD][0][0], x1);
                  acc[c1 % kAD][0][1] = fmaxf(acc[c1 % kAD][0][1], x1);
                }
              } else {
                acc[c % kAD][1][0] = fminf(acc[c % kAD][1][0], x0);
                acc[c % kAD][1][1] = fmaxf(acc[c % kAD][1][1], x0);
                if (two) {
                  acc[c1 % kAD][1][0] = fminf(acc[c1 % kAD][1][0], x1);
                  acc[c1 % kAD][1][1] = fmaxf(acc[c1 % kAD][1][1], x1);
                }
              }
            }
        } else if (want_mm) {
          // min / max as floats, then keys once per warp and sub-tile
          float mm[2][2][2] = {{{inf, -inf}, {inf, -inf}}, {{inf, -inf}, {inf, -inf}}};  // [col][side][min,max]
#pragma unroll
          for (int q = 0; q < kMaxItems; ++q)
            if (keep[q]) {
              const float x0 = __uint_as_float(v0[q]), x1 = __uint_as_float(v1[q]);
              if (left[q]) {
                mm[0][0][0] = fminf(mm[0][0][0], x0);
                mm[0][0][1] = fmaxf(mm[0][0][1], x0);
                mm[1][0][0] = fminf(mm[1][0][0], x1);
                mm[1][0][1] = fmaxf(mm[1][0][1], x1);
              } else {
                mm[0][1][0] = fminf(mm[0][1][0], x0);
                mm[0][1][1] = fmaxf(mm[0][1][1], x0);
                mm[1][1][0] = fminf(mm[1][1][0], x1);
                mm[1][1][1] = fmaxf(mm[1][1][1], x1);
              }
            }
#pragma unroll
          for (int cc = 0; cc < 2; ++cc) {
            if (cc == 1 && !two) break;
#pragma unroll
            for (int side = 0; side < 2; ++side) {
              const uint32_t lo = __reduce_min_sync(0xffffffffu, ord_key(mm[cc][side][0]));
              const uint32_t hi = __reduce_max_sync(0xffffffffu, ord_key(mm[cc][side][1]));
              if (lane == 0) {
                atomic_min_shared(&tmm[side][c + cc][0], lo);
                atomic_max_shared(&tmm[side][c + cc][1], hi);
              }
            }
          }
        }
      }
      // ---- subset offsets of the children: each segment start off[u] = p of
      // the cell that lies in this sub-tile (the cell's end in its last one)
      // becomes the left child's start, the left points before p, and the
      // right child's, p minus that (rows of r + 1 words, checked against
      // their pool when they were handed out)
      if (want_off) {
        uint32_t* const row0 = m.row[0];
        uint32_t* const row1 = m.row[1];
        for (uint32_t ub = m.u0; ub < m.u1; ub += kCT) {
          const uint32_t u = ub + (uint32_t)tid;
          if (ub != m.u0) u_pos = u < m.u1 ? __ldg(m.off + u) : 0xffffffffu;
          const uint32_t i = u_pos - m.sub;  // wraps for starts before the sub-tile
          const bool end = u_pos == ccount && m.sub + mcnt == ccount;
          const bool mine = u < m.u1 && u_pos >= m.sub && (i < mcnt || end);
          if (!__any_sync(0xffffffffu, mine)) continue;
          const uint32_t blk = min(i >> 5, 31u);  // i < 32 kMaxItems kCW where it counts
          uint32_t lk = lnext - cbeg + __shfl_sync(0xffffffffu, wexc, blk);
          if (mine) {
            lk = end ? L : lk + (uint32_t)__popc((&wbal[0][0])[blk] & ((1u << (i & 31u)) - 1u));
            if (row0) row0[u] = lk;
            if (row1) row1[u] = u_pos - lk;
          }
        }
      }
      lnext += nL;
      rnext += mcnt - nL;
      more = m.sub + T < tend;
      if (!more) {  // last sub-tile of the tile
        if (saw_nan) atomicCAS(m.status, ST_OK, ST_NAN_INPUT);
        saw_nan = false;
        if (want_mm) {
          // keep reducing while this CTA's next tile is of the same cell (the
          // producer, which reads the tile list ahead, says so); else add the
          // run's min / max to the cell's with atomics
          if (!m.run_more) {
            if (kAcc) {
              // transpose-reduce over the warp: value u = (l * 2 + side) * 2 +
              // which, maxima negated so that every step is a minimum; after
              // the steps lane u holds value u reduced over all 32 lanes
              constexpr int kV = 4 * kAD;
              constexpr int kVP = kV <= 8 ? 8 : (kV <= 16 ? 16 : 32);
              float v[kVP];
#pragma unroll
              for (int u = 0; u < kVP; ++u) {
                const int l = u / 4, side = (u / 2) & 1, which = u & 1;
                v[u] = u >= kV ? inf : (which ? -acc[l % kAD][side][1] : acc[l % kAD][side][0]);
              }
#pragma unroll
              for (int h = kVP / 2; h >= 1; h >>= 1) {
                const bool upper = (lane & h) != 0;
#pragma unroll
                for (int i = 0; i < h; ++i) {
                  const float keep = upper ? v[i + h] : v[i];
                  const float send = upper ? v[i] : v[i + h];
                  v[i] = fminf(keep, __shfl_xor_sync(0xffffffffu, send, h));
                }
              }
#pragma unroll
              for (int o = kVP; o < 32; o <<= 1) v[0] = fminf(v[0], __shfl_xor_sync(0xffffffffu, v[0], o));
              if (lane < kV) {
                const int l = lane / 4, side = (lane / 2) & 1;
                if (lane & 1)
                  atomic_max_shared(&tmm[side][l][1], ord_key(-v[0]));
                else
                  atomic_min_shared(&tmm[side][l][0], ord_key(v[0]));
              }
#pragma unroll
              for (int l = 0; l < kAD; ++l)
#pragma unroll
                for (int side = 0; side < 2; ++side) {
                  acc[l][side][0] = inf;
                  acc[l][side][1] = -inf;
                }
            }
            named_sync(kConsumerBar, kCT);
            // add the run's min / max to the cell's; reset the table
            for (int j = tid; j < 4 * d; j += kCT) {
              const int side = j / (2 * d), l = (j / 2) % d, which = j & 1;
              uint32_t* dst = &s.child_mm[(((size_t)m.cell_idx * 2 + side) * kMaxDims + l) * 2 + which];
              if (which) atomicMax(dst, tmm[side][l][which]); else atomicMin(dst, tmm[side][l][which]);
              tmm[side][l][which] = which ? 0u : 0xffffffffu;
            }
          }
        }
      }
      // ---- release the buffer: each warp's reads of it precede the next bulk
      // writes; the "empty" barrier counts the consumer warps (the next
      // sub-tile's first barrier orders the reuse of wcnt and wbal)
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[b]);
    }
  }
}

}  // namespace

// Dynamic shared memory of an instance (for any d: the most a mix can need).
constexpr uint32_t scatter_smem(int kD) { return kD > 0 ? 2u * buf_bytes(kD, sub_tile_one(kD)) : most_smem(kD); }

template <int kD, bool kMM>
cudaError_t prepare_one() {
  return cudaFuncSetAttribute(k_scatter_tma<kD, kMM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)scatter_smem(kD));
}

template <int kD, bool kMM>
void launch_one(const TreeDev* trees, const StepDev& s, uint32_t max_tiles, uint32_t sms, cudaStream_t st) {
  // two waves of resident CTAs, each taking a contiguous range of tiles
  const uint32_t grid = std::max<uint32_t>(1, std::min(max_tiles, sms * 2u * (uint32_t)scatter_ctas(kD, kMM)));
  launch_chained(k_scatter_tma<kD, kMM>, grid, kST, scatter_smem(kD), st, trees, s);
}

// f(instance) for the trees' coordinate count (0: they differ).
// (3,000,017 points in 5 coordinates, depth rule: the scatters of a build took
// 0.67 ms in the instance for any d and take 0.49 ms in their own.)
template <bool kMM, class F>
auto with_d(int uniform_d, F f) {
  switch (uniform_d) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    case 5: return f(std::integral_constant<int, 5>{});
    case 6: return f(std::integral_constant<int, 6>{});
    case 7: return f(std::integral_constant<int, 7>{});
    case 8: return f(std::integral_constant<int, 8>{});
    case 12: return f(std::integral_constant<int, 12>{});
    case 16: return f(std::integral_constant<int, 16>{});
    default:
      return uniform_d > 0 ? f(std::integral_constant<int, kOtherD>{}) : f(std::integral_constant<int, kMixedD>{});
  }
}

template <bool kMM>
cudaError_t prepare_d(int uniform_d) {
  return with_d<kMM>(uniform_d, [](auto k) { return prepare_one<decltype(k)::value, kMM>(); });
}

template <bool kMM>
void launch_d(const TreeDev* trees, const StepDev& s, uint32_t max_tiles, uint32_t sms, int uniform_d,
              cudaStream_t st) {
  with_d<kMM>(uniform_d, [&](auto k) { launch_one<decltype(k)::value, kMM>(trees, s, max_tiles, sms, st); });
}

cudaError_t prepare_scatter_kernel(int uniform_d, bool any_widest) {
  return any_widest ? prepare_d<true>(uniform_d) : prepare_d<false>(uniform_d);
}

void launch_scatter(const TreeDev* trees, const StepDev& s, uint32_t max_tiles, uint32_t sms, uint64_t points,
                    int uniform_d, bool any_widest, cudaStream_t st) {
  TraceScope ts(K_PART_SCATTER, st, points);
  if (any_widest)
    launch_d<true>(trees, s, max_tiles, sms, uniform_d, st);
  else
    launch_d<false>(trees, s, max_tiles, sms, uniform_d, st);
}

}  // namespace kdt
