// Host check (no GPU, a fake of the CUDA runtime's calls) of when a decode merges in a cluster of CTAs, and of what it does
// where one cannot be placed: the device says so, or the launch is refused.  Prints one line per failed property and returns 1 if there were any.
#include <cstdio>
#include <vector>

#include "innerq_kernels.h"

namespace {
int device = 0, asked = 0;
}

extern "C" {
cudaError_t CUDARTAPI cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t CUDARTAPI cudaGetLastError(void) { return cudaSuccess; }
cudaError_t CUDARTAPI cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
// device 0 holds clusters of up to 8 CTAs, device 1 of any number; 5 CTAs: the question itself fails
cudaError_t CUDARTAPI cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* cfg) {
  ++asked;
  const unsigned ctas = cfg->numAttrs == 1 ? cfg->attrs[0].val.clusterDim.y : 0;
  if (ctas == 0 || ctas == 5 || cfg->dynamicSmemBytes != 1000) return cudaErrorInvalidValue;
  *n = device == 0 && ctas > 8 ? 0 : (int)(100 / ctas);
  return cudaSuccess;
}
}

int main() {
  using namespace iq;
  int failures = 0;
  auto check = [&](bool ok, const char* what) {
    if (!ok) { ++failures; std::printf("FAIL %s\n", what); }
  };
  void (*kernel)() = nullptr;
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = 1000;
  static ClusterRoom room;
  for (int again = 0; again < 2; ++again) {
    device = 0;
    check(room(kernel, cfg, 8) == 12 && room(kernel, cfg, 2) == 50, "what fits");
    check(room(kernel, cfg, 16) == 0 && room(kernel, cfg, 9) == 0, "what does not");
    check(room(kernel, cfg, 5) == 0 && room(kernel, cfg, 0) == 0 && room(kernel, cfg, 17) == 0, "no answer");
    device = 1;
    check(room(kernel, cfg, 16) == 6 && room(kernel, cfg, 8) == 12, "another device");
    check(asked == 7, "asked once per device and size");
  }
  // launches with and without a cluster; which of the two forms the device accepts
  for (int wanted = 0; wanted < 2; ++wanted)
    for (int takes_cluster = 0; takes_cluster < 2; ++takes_cluster)
      for (int takes_plain = 0; takes_plain < 2; ++takes_plain) {
        std::vector<bool> tried;
        const bool ok = launch_merging(wanted != 0, [&](bool in_cluster) {
          tried.push_back(in_cluster);
          return in_cluster ? takes_cluster != 0 : takes_plain != 0;
        });
        std::vector<bool> want;
        if (wanted) want.push_back(true);
        if (!wanted || !takes_cluster) want.push_back(false);
        check(tried == want && ok == ((wanted && takes_cluster) || takes_plain), "launch_merging");
      }
  // the rule's edges: {bits, clusters, CTAs of one, rows, chunks per warp, room} and whether they merge in the cluster
  const struct { int bits, n, grid_y, rows, chunks, room; bool want; } edges[] = {
      {4, 7, 16, 4, 2, 14, true}, {4, 8, 16, 4, 2, 14, false}, {4, 1, 17, 4, 2, 14, false}, {2, 16, 8, 3, 3, 33, true},
      {2, 17, 8, 3, 3, 33, false}, {2, 6, 8, 4, 6, 33, true}, {2, 5, 8, 4, 7, 33, true}, {2, 6, 8, 4, 7, 33, false},
      {4, 6, 8, 3, 2, 33, true}, {4, 6, 8, 3, 3, 33, false}, {4, 5, 8, 3, 3, 33, true}, {4, 148, 2, 3, 9, 148, true},                  // short and long
      {4, 148, 2, 4, 300, 148, true}, {4, 149, 2, 4, 1, 148, false}, {4, 48, 1, 4, 1, 296, true}, {4, 49, 1, 4, 1, 296, false},
      {2, 1, 2, 4, 1, 0, false}, {2, 1, 1, 1, 1, 0, false},                                                // no room at all
      {4, 2, 16, 1, 2, 14, true}, {4, 3, 16, 1, 2, 14, false}, {2, 5, 16, 1, 2, 14, true}, {2, 6, 16, 2, 1, 14, false},
      {2, 2, 16, 2, 7, 14, false}, {4, 48, 1, 2, 6, 296, true}, {4, 48, 1, 2, 7, 296, false},
      {4, 9, 8, 4, 2, 33, true}, {4, 10, 8, 4, 2, 33, false}, {4, 10, 9, 4, 2, 30, true},
      {2, 74, 2, 1, 1, 148, true}, {2, 75, 2, 1, 1, 148, false}, {2, 148, 2, 1, 1, 148, false},
      {2, 74, 2, 2, 4, 148, true}, {2, 99, 2, 2, 1, 148, false}, {2, 100, 2, 2, 8, 148, true}, {2, 100, 2, 2, 9, 148, false}};
  for (const auto& e : edges) {
    Layout L = {};
    L.k.bits = L.v.bits = e.bits;
    if (merges_in_cluster(L, e.n, e.grid_y, e.rows, e.chunks, e.room) != e.want) {
      ++failures;
      std::printf("FAIL rule: %d bits, %d clusters of %d, %d rows, %d chunks, room %d\n", e.bits, e.n, e.grid_y, e.rows, e.chunks, e.room);
    }
  }
  std::printf("%d failure(s)\n", failures);
  return failures != 0;
}
