// Host check of csrc/innerq_split.h over the shapes that the library accepts (no GPU): every launch has a grid, its split
// partials fit the memory they are given, its CTAs fit the ticket field that counts them, the tail tiles are all dealt,
// and groups of query rows share a launch only where that pays.
// Prints one line per failed property and returns 1 if there were any.  With eight arguments it prints the plan of one call.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "innerq_split.h"

using namespace iq;

namespace {

// The plan of one call as "passes splits default_splits reset_iters(one chunk per iteration) reset_iters(two)".
int print_plan(char** v) {
  const int U = std::atoi(v[1]), r = std::atoi(v[2]), n_q = std::atoi(v[3]), w_sink = std::atoi(v[4]), w_recent = std::atoi(v[5]),
            G = std::atoi(v[6]), N = std::atoi(v[7]);
  const bool outer = std::atoi(v[8]) != 0;
  Layout L = {};
  L.U = U; L.r = r; L.G = G; L.w_sink = w_sink; L.w_recent = w_recent;
  L.max_splits = max_splits_for(U, w_sink, w_recent, G);
  L.k.kind = outer ? kBlock : kRow; L.v.kind = outer ? kRow : kBlock;
  const Counts cn = counts_for(L, N);
  SplitArgs a = {};
  a.n_q = n_q;
  const int n = plan_call(L, cn, a, outer, 0);
  fill_split_args(L, cn, a, G / kChunk, outer, n, 0);
  fill_reference_args(cn, a, G / kChunk, 1, outer);
  const int one = a.reset_iters;
  fill_reference_args(cn, a, G / kChunk, 2, outer);
  std::printf("%d %d %d %d %d\n", a.passes, a.n_splits, default_splits(L, U), one, a.reset_iters);
  return 0;
}

}  // namespace

int main(int argc, char** argv) {
  if (argc == 9) return print_plan(argv);
  long long failures = 0, calls = 0;
  const int windows[][2] = {{0, 0}, {4, 32}, {4, 64}, {0, 64}, {32, 96}, {4, 128}, {4, 256}, {64, 2000}};
  for (int U = 1; U <= 65535; U = U < 700 ? U + 1 : U * 5 / 4)
    for (const auto& w : windows)
      for (int G : {32, 64, 128})
        for (int r : {1, 2, 3, 4, 5, 8, 16, 33, 64})
          for (int n_q : {1, 2, 4, 5, 7, 8, 16, 33}) {
            if (n_q - 1 > w[1] || r * n_q > 128) continue;
            for (int n_splits : {0, 1, 3, 148, 1000})
              for (int N : {1, 300, 5000, 200000}) {
                if ((U > 64 && n_splits > 3) || (U > 700 && N == 5000)) continue;
                Layout L = {};
                L.U = U; L.r = r; L.G = G; L.w_sink = w[0]; L.w_recent = w[1];
                L.max_splits = max_splits_for(U, w[0], w[1], G);
                L.k.kind = kRow; L.v.kind = kBlock;
                const Counts cn = counts_for(L, N);
                SplitArgs a = {};
                a.n_q = n_q;
                const int n = plan_call(L, cn, a, false, n_splits);
                auto check = [&](bool ok, const char* what) {
                  if (!ok && failures++ < 20)
                    std::printf("FAIL %s: units %d windows %d %d G %d r %d n_q %d splits %d N %d: passes %d row_cap %d\n", what, U,
                                w[0], w[1], G, r, n_q, n_splits, N, a.passes, a.row_cap);
                  return ok;
                };
                // an explicit split count is kept as long as a launch of one group can hold it
                check(n_splits == 0 || n == std::min(n_splits, std::min(L.max_splits, 128)), "the caller's splits");
                a.n_skew_tiles = (cn.n_qk - cn.n_qv + 15) / 16;
                a.n_tail_tiles = a.n_skew_tiles + (cn.n_sink + cn.n_k_recent + 15) / 16;
                ++calls;
                const bool cap = check(a.row_cap >= 1 && a.row_cap <= a.part_stride, "a row of the grid");
                check(a.passes >= 1 && a.passes <= 8 && n >= 1, "passes");
                check(a.part_stride * (n_q > 1 ? a.passes : 1) <= L.max_splits, "partials fit their memory");
                if (n_splits == 0) {
                  // what the launches take, in chunks per CTA slot (starts and ends: 18; a half wave has its SMs to itself):
                  // never much more than with one launch per group of four rows
                  const int total = (r * n_q + 3) / 4, units = (cn.n_qv / kChunk + G / kChunk - 1) / (G / kChunk);
                  auto time = [&](int p, int s) {
                    s = std::min(s, std::max(1, (units + 7) / 8));
                    const double ctas = (double)U * total * s, full = std::floor(ctas / 296), rest = ctas - 296 * full;
                    return (full + (rest == 0 ? 0 : rest <= 148 ? 0.65 : 1)) * (cn.n_qv / 32 / (double)s + 18) + 14 * ((total + p - 1) / p - 1);
                  };
                  check(time(a.passes, n) <= 1.07 * time(1, default_splits(L, U)), "time against one launch per group");
                }
                if (!cap) continue;      // the next function divides by the grid
                const int grid = fill_split_args(L, cn, a, G / kChunk, false, n, 0);
                check(grid >= 1 && grid <= a.row_cap && a.n_splits <= grid, "grid rows");
                check(a.passes == 1 || grid < 1 << a.ticket_bits, "ticket field");
                check(a.passes * a.ticket_bits <= 32, "ticket word");
                check(a.tiles_q0 * grid + a.tiles_rem == a.n_tail_tiles && a.tiles_rem < grid, "tail tiles");
              }
          }
  std::printf("%lld calls, %lld failure(s)\n", calls, failures);
  return failures != 0;
}
