// How a launch of the fused decode kernel is cut up: token ranges per unit (splits), groups of four query rows per launch
// (passes).  Host arithmetic only, no CUDA headers: the host test (tests/host_split_check.cpp) includes it as it is.
#pragma once
#include <algorithm>

#include "innerq_layout.h"

namespace iq {

constexpr int kSplitWarps = 8;          // warps of a decode CTA: each takes its own token range
constexpr int kCtaSlots = 2 * 148;      // resident decode CTAs: two per SM

// The parameters of a launch that follow from the split (base of DecodeArgs).
struct SplitArgs {
  int n_q;               // consecutive query tokens per sequence (1: plain decode).  Row v = i * r + h of a KV head is
                         // head h of query token i; q / out are [B, n_q, Hq, D]; query i does not see the newest
                         // n_q - 1 - i tokens (all of them outside the chunks where keys AND values are packed)
  int grid_y;            // grid rows (blockIdx.y) that work on this cache: the launch's gridDim.y, or fewer for a
                         // short sequence of a batched launch (the rows beyond it return at once)
  int n_splits;          // CTAs per unit that stream packed chunks (blockIdx.y < n_splits <= grid_y)
  int n_tail_tiles;      // tiles of 16 tokens outside the packed-K/packed-V range: skew tiles first, then fp16 tiles;
                         // tile x belongs to CTA x % grid_y, warp (x / grid_y) % 8
  int n_skew_tiles;      // of those, tiles whose keys are packed rows (values still fp16)
  int tiles_q0, tiles_rem;   // n_tail_tiles / grid_y and n_tail_tiles % grid_y
  int units_per_split;   // range units (max(value group, iteration) of chunks) per CTA, before the tail discount
  int tail_cost_units;   // a warp streams this many range units less per tail tile it handles (load balance)
  int passes;            // groups of four query rows per unit in this launch: block x = (unit, pass), pass p takes the rows
                         // head0 + 4 p ..; the passes of a unit read the same records at the same time, through L2
  int ticket_bits;       // every pass counts its arriving CTAs in its own field of the unit's ticket word
  int row_cap;           // most grid rows: what a ticket field and part_stride hold
  int part_stride;       // split partials per query row in `partials`
  int ref_splits;        // > 0: the split count whose ranges the soft-max references follow (see kernel), else 0
  int reset_iters;       // ... as loop iterations between two fresh references of a warp (0: none but the first)
};

// Partial slots per query head: token-range splits (two waves of CTAs for all units, 64 at most) plus one per 32 tokens of
// the fp16 tail.
inline int max_splits_for(int n_units, int w_sink, int w_recent, int G) {
  const int waves = (2 * kCtaSlots + n_units - 1) / n_units;
  return std::min(64, std::max(1, waves)) + (w_sink + w_recent + G + 31) / 32 + 1;
}

// One wave of CTAs.
inline int default_splits(const Layout& L, int n_units_total) {
  return std::min(std::max(1, kCtaSlots / n_units_total), std::min(L.max_splits, 128));
}

// Groups of four query rows that one launch takes (passes), and what follows from it.  All of them go into one launch,
// up to eight (more: launches of equal size): one start, one end and one read of the records from HBM instead of one per
// group.  Fewer where the split count does not fit: with p passes a pass has 32 / p bits of a unit's ticket word to
// count its CTAs in and, with several query tokens (whose partials live in scratch of four rows per unit), 1 / p of a
// row's split partials, which has to be one at least (many units with short windows have fewer than eight).
inline int fill_pass_args(const Layout& L, SplitArgs& a, int n_splits) {
  const int total = (L.r * a.n_q + 3) / 4, launches = (total + 7) / 8;
  int per = (total + launches - 1) / launches;
  auto by_ticket = [&](int p) { return p == 1 ? L.max_splits : std::min(L.max_splits, (1 << (32 / p)) - 1); };
  auto by_part = [&](int p) { return a.n_q > 1 ? L.max_splits / p : L.max_splits; };
  auto fits = [&](int p) {
    if (by_part(p) < 1) return false;
    if (n_splits > 0) return n_splits <= std::min(by_ticket(p), by_part(p));      // the caller's choice
    return std::min(default_splits(L, L.U * p), by_part(p)) <= by_ticket(p);
  };
  while (per > 1 && !fits(per)) --per;
  a.passes = per;
  a.ticket_bits = 32 / per;
  a.row_cap = std::min(by_ticket(per), by_part(per));
  a.part_stride = by_part(per);
  return per;
}

// The split of a call: passes and the split count (n_splits > 0: the caller's choice), which is returned.
inline int plan_call(const Layout& L, SplitArgs& a, int n_splits) {
  n_splits = std::min(n_splits, std::min(L.max_splits, 128));      // 128: slots of the merge tables in shared memory
  const int per = fill_pass_args(L, a, n_splits);
  a.ref_splits = a.reset_iters = 0;
  if (n_splits > 0) return n_splits;
  if (per > 1) a.ref_splits = default_splits(L, L.U);
  return default_splits(L, L.U * per);
}

// Split-dependent launch parameters of one cache for a grid of grid_y rows (0: choose it): how many of the rows
// stream packed chunks, the range units (ru chunks each) per row, the tail tiles per row.  Returns grid_y.
inline int fill_split_args(const Layout& L, const Counts& cn, SplitArgs& a, int ru, bool outer, int n_splits, int grid_y) {
  const int n_chunks = (outer ? cn.n_qk : cn.n_qv) / kChunk;
  const int n_units = (n_chunks + ru - 1) / ru;
  const int by_work = (n_units + kSplitWarps - 1) / kSplitWarps;      // at least one range unit per warp
  if (n_splits > by_work) n_splits = by_work;
  if (n_units == 0) n_splits = 0;
  if (grid_y <= 0) {
    // without packed chunks the CTAs only share the tail tiles (eight per CTA)
    grid_y = n_splits > 0 ? n_splits : (a.n_tail_tiles + kSplitWarps - 1) / kSplitWarps;
    if (grid_y < 1) grid_y = 1;
    if (grid_y > a.row_cap) grid_y = a.row_cap;
  }
  if (n_splits > grid_y) n_splits = grid_y;
  a.grid_y = grid_y;
  a.n_splits = n_splits;
  a.tail_cost_units = n_splits ? 1 : 0;     // a tail tile costs a warp about as much as one value group's chunks
  const int virt = n_units + a.tail_cost_units * a.n_tail_tiles;
  a.units_per_split = n_splits ? (virt + n_splits - 1) / n_splits : 0;
  a.tiles_q0 = a.n_tail_tiles / grid_y;
  a.tiles_rem = a.n_tail_tiles % grid_y;
  return grid_y;
}

}  // namespace iq
