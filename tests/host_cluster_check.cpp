// Host check (no GPU, a fake of the CUDA runtime's calls) of what a decode does where a cluster of CTAs cannot be placed: the
// device says so, or the launch is refused.  Prints one line per failed property and returns 1 if there were any.
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
  std::printf("%d failure(s)\n", failures);
  return failures != 0;
}
