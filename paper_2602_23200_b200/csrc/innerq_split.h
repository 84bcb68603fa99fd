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
  int reset_iters;       // ... as loop iterations between two fresh references of a warp (0: none but the first); see
                         // fill_reference_args
};

// Whether the CTAs of a unit (and group) are a cluster that merges through distributed shared memory instead of through
// global memory and a ticket.  That saves three dependent trips to L2 at the end of a launch (8 KV heads x 1001 tokens, r 4,
// 3-bit keys: 13.3 -> 11.2 us alone, 6.0 -> 4.2 us in a chain), but a cluster starts only when all its CTAs find room in one
// GPC: next to the launches before and after it in a chain it may have to wait.  So the rule goes by the chain (a call alone
// gains 5 to 20 % at nearly every point below).  `room`: most clusters of this size that are resident at once (ClusterRoom);
// `warp_chunks`: chunks (of 32 tokens) that a warp streams; `rows`: query rows merged, which the ticket's last CTA takes one
// after the other.  Chain, tickets -> clusters, over some 2500 points (2, 3, 4 bits, G 32, 64, 128) of decodes, and 1000 of
// appends and decodes in turn:
//  * Three and four rows, short ranges: as long as the clusters of two launches fit at once.  With room for 14 of 16 CTAs, 7
//    took 6.3 -> 4.8 us (2 bits) and 6.6 -> 5.4 (4 bits), 8 took 6.5 -> 6.6 and 6.7 -> 7.6; 16 of 8 (room 33) 6.5 -> 5.4 and
//    6.6 -> 6.1, 18 of them 6.5 -> 6.7 and 6.9 -> 8.1.  Three rows lose where a warp streams much (15 clusters of 9, 4 bits,
//    G 128: 7.1 -> 7.6).  So do steps with clusters of 3 to 8 above half a CTA per SM: 108 CTAs, 4 bits, G 64: decodes 6.4 ->
//    6.1 but steps 8.3 -> 9.3.
//  * Three and four rows, pairs: to the last slot (one SM's two will do), at every length.  128 pairs: 11.7 -> 9.6 us (4 bits,
//    G 32, 1200 tokens), 26.3 -> 25.7 on average at 8192 tokens.
//  * Three and four rows, long ranges (a caller's split count): 16 CTAs a unit, 2 bits, 60000 tokens: 32 of them 6.6
//    -> 5.3, 64 7.8 -> 7.5, 112 9.7 -> 10.6, 128 10.0 -> 13.1.
//  * Two rows and one (and such three): the ticket costs less and the chain hardly changes (4.5 -> 4.5 us); above 40 CTAs, 80
//    where a warp streams little, it loses: 64 CTAs of 8, 4 bits, G 64: 4.5 -> 5.1; 112 of 4, 2 bits, G 32: 5.0 -> 5.2; 148:
//    5.1 -> 6.2.
//  * One CTA (its merge needs no other): to 48 of them chains and steps gain up to 2 %; 64 units, one row, 4 bits, G 128: steps
//    11.6 -> 12.0; 128, 2 bits, G 64: decodes 8.1 -> 8.9.
//  * Pairs of few rows: one CTA per SM at most (148: 6.2 -> 5.8); one row above that between 5 % faster and 10 % slower
//    (128 pairs x 16384 tokens, 2 bits, G 32: 32.4 -> 35.1); two rows 10.9 -> 8.9 (148 pairs x 649 tokens), 13.0 -> 12.3 (128 x
//    2500), but 18.5 -> 18.7 (100 x 8192), and just above one CTA per SM 6.1 -> 6.4.
constexpr int kClusterCtas = 16;
inline bool merges_in_cluster(const Layout& L, int n_clusters, int grid_y, int rows, int warp_chunks, int room) {
  if (grid_y > kClusterCtas || n_clusters > room) return false;
  const int ctas = n_clusters * grid_y;
  const int streamed = warp_chunks * (L.k.bits + L.v.bits);
  const bool is_short = warp_chunks <= 6;
  if (grid_y == 1) return is_short && ctas <= 48;
  if (rows >= 4 || (rows == 3 && (grid_y == 2 || streamed <= 16))) {
    if (grid_y == 2) return true;
    return is_short ? 2 * n_clusters <= room && (streamed < 16 || grid_y > 8 || ctas <= 72) : ctas <= 40;
  }
  if (grid_y == 2 && rows == 2 && ctas >= 200) return warp_chunks <= 8;
  return is_short && ctas <= (grid_y == 2 ? kCtaSlots / 2 : streamed <= 8 ? 80 : 40);
}

// The longest range of a warp, in chunks (see merges_in_cluster).
inline int warp_chunks_of(const Counts& cn, const SplitArgs& a, bool outer) {
  const int n_chunks = (outer ? cn.n_qk : cn.n_qv) / kChunk, warps = kSplitWarps * std::max(1, a.n_splits);
  return (n_chunks + warps - 1) / warps;
}

// Launches a decode: launch(merge in a cluster?) says whether it was accepted.  A cluster that is refused goes without.
template <typename Launch> inline bool launch_merging(bool cluster, Launch launch) {
  return (cluster && launch(true)) || launch(false);
}

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

// Most grid rows of a launch of p passes: a pass counts its CTAs in 32 / p bits of a unit's ticket word and, with several
// query tokens (whose partials live in scratch of four rows per unit), has 1 / p of a row's split partials.
inline int partial_slots(const Layout& L, int n_q, int p) { return n_q > 1 ? L.max_splits / p : L.max_splits; }
inline int most_rows(const Layout& L, int n_q, int p) {
  const int by_ticket = p == 1 ? L.max_splits : std::min(L.max_splits, (1 << (32 / p)) - 1);
  return std::min(by_ticket, partial_slots(L, n_q, p));
}

// The split of a call: groups of four query rows per launch (passes), and the split count (n_splits > 0: the caller's
// choice), which is returned.  All groups go into one launch, up to eight, with one wave of CTAs together: one start, one
// end and one read of the records from HBM instead of one per group.  Two things can make that slower for a call that runs
// alone than one launch per group, on long contexts by up to a factor of two: a wave that leaves slots idle (40 units with
// five groups: one split each, 200 CTAs), and few units whose partials do not hold enough splits for every group (one unit
// with eight groups: 8 of 37).  Time alone, in chunks (of 32 tokens, 0.16 us):
//   waves * (chunks per CTA + 18) + 14 per further launch
// with 18 for a CTA's start and end; launches overlap, so the waves are those of all CTAs together; a last half wave counts
// 0.65, its CTAs have an SM each.  Where that is less with one launch per group, the launches that could be made (groups
// per launch, splits that fill half a wave more at a time) are compared, and of those within 6 % of the best the fewest
// launches and longest ranges are taken: they leave most to the neighbours in a chain of calls.
// Alone / in a chain, us: one launch per group; always one wave; chosen.  40 units x 16384 tokens, r 4, n_q 5, 4 bits:
// 109.7 / 95.7; 116.0 / 79.6; 96.7 / 77.7.  80 x 16384, r 8: 81.6 / 62.4; 106.1 / 60.6; 79.0 / 59.1.  1 x 524288, n_q 8:
// 128.3 / 98.4; 209.1 / 83.9; 107.5 / 83.7.
inline int plan_call(const Layout& L, const Counts& cn, SplitArgs& a, bool outer, int n_splits) {
  const int total = (L.r * a.n_q + 3) / 4, ru = L.G / kChunk, n_chunks = (outer ? cn.n_qk : cn.n_qv) / kChunk;
  const int alone = default_splits(L, L.U);                        // splits of a launch of one group
  n_splits = std::min(n_splits, std::min(L.max_splits, 128));      // 128: slots of the merge tables in shared memory
  const bool chosen = n_splits > 0;
  auto one_wave = [&](int p) { return std::min(default_splits(L, L.U * p), most_rows(L, a.n_q, p)); };
  auto holds = [&](int p) {      // a launch of p groups has the partials and ticket bits for its splits
    if (partial_slots(L, a.n_q, p) < 1) return false;
    if (chosen) return n_splits <= most_rows(L, a.n_q, p);
    return std::min(default_splits(L, L.U * p), partial_slots(L, a.n_q, p)) == one_wave(p);
  };
  const int fewest = (total + 7) / 8;
  int best_p = (total + fewest - 1) / fewest;
  while (best_p > 1 && !holds(best_p)) --best_p;
  int best_s = chosen ? n_splits : one_wave(best_p);
  if (!chosen && best_p > 1) {
    const int by_work = std::max(1, ((n_chunks + ru - 1) / ru + kSplitWarps - 1) / kSplitWarps);      // see fill_split_args
    auto time = [&](int p, int s) {
      const int used = std::min(s, by_work);
      const long long ctas = (long long)L.U * total * used, rest = ctas % kCtaSlots;
      const float waves = (float)(ctas / kCtaSlots) + (rest == 0 ? 0.f : rest <= kCtaSlots / 2 ? 0.65f : 1.f);
      // outer grouping: the instance that renews its references takes 3-8 % longer
      const float slower = outer && used < std::min(alone, by_work) ? 1.05f : 1.f;
      return waves * ((float)n_chunks / (float)used + 18.f) * slower + 14.f * (float)((total + p - 1) / p - 1);
    };
    if (time(best_p, best_s) > time(1, alone)) {
      struct { int p, s; float t; } cand[8 * 12];
      int n = 0;
      float least = time(1, alone);
      auto add = [&](int p, int s) {
        cand[n] = {p, s, time(p, s)};
        least = std::min(least, cand[n++].t);
      };
      for (int launches = fewest, last = 0; launches <= total; ++launches) {
        const int p = (total + launches - 1) / launches;
        if (p == last || most_rows(L, a.n_q, p) < 1) continue;
        last = p;
        const int most = std::min(alone, most_rows(L, a.n_q, p));
        add(p, one_wave(p));
        for (int half = 3; half <= 10; ++half) {
          const int s = (int)((long long)half * (kCtaSlots / 2) / ((long long)L.U * p));
          if (s > cand[n - 1].s && s < most) add(p, s);
        }
        if (most > cand[n - 1].s) add(p, most);
      }
      for (int i = n - 1; i >= 0; --i)
        if (cand[i].t <= 1.06f * least) { best_p = cand[i].p; best_s = cand[i].s; }
    }
  }
  a.passes = best_p;
  a.ticket_bits = 32 / best_p;
  a.row_cap = most_rows(L, a.n_q, best_p);
  a.part_stride = partial_slots(L, a.n_q, best_p);
  a.ref_splits = !chosen && total > 1 ? alone : 0;
  a.reset_iters = 0;
  return best_s;
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

// Iterations (of cpi chunks) between two fresh soft-max references: where the groups of a call share the CTA slots, a warp's
// range is several times what it would be in a launch of one group, and a reference for all of it would resolve p less; so
// it is renewed after every range that the warp would have had (whole value groups, one at least).  Outer grouping, where
// that takes an instance of its own: only if the ranges are longer, and the nearest number of groups (a renewal there costs
// as much as a tenth of an iteration with its group).
inline void fill_reference_args(const Counts& cn, SplitArgs& a, int ru, int cpi, bool outer) {
  const int n_units = ((outer ? cn.n_qk : cn.n_qv) / kChunk + ru - 1) / ru;
  const int ref_splits = std::min(a.ref_splits, (n_units + kSplitWarps - 1) / kSplitWarps);      // as in fill_split_args
  const bool renew = ref_splits > 0 && (outer ? ref_splits > a.n_splits : ref_splits >= a.n_splits);
  const int per_warp = kSplitWarps * ref_splits;
  const int units = renew ? std::max(1, (n_units + (outer ? per_warp / 2 : 0)) / per_warp) : 0;
  a.reset_iters = renew ? std::max(1, units * ru / cpi) : 0;
}

}  // namespace iq
