// Host-callable launchers of the library's kernels (internal interface between the .cu files).
// Each returns the number of kernels it launched, or -1 on a CUDA error.
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "innerq_layout.h"
#include "innerq_split.h"

namespace iq {

// More than 48 KB of dynamic shared memory is an opt-in per kernel AND per device: `done` (one per kernel, a bit per
// device ordinal) remembers where it has been set, so a process that drives several GPUs sets it on each of them.
template <typename Kernel>
inline bool opt_in_dynamic_smem(Kernel kernel, int bytes, std::atomic<unsigned long long>& done, bool clusters = false) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  const unsigned long long bit = 1ull << dev;
  if (done.load(std::memory_order_acquire) & bit) return true;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) return false;
  // clusters of more than the portable 8 CTAs, where the device has them (see ClusterRoom)
  if (clusters && cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
  done.fetch_or(bit, std::memory_order_release);
  return true;
}

// How many clusters of a kernel the device holds at once, by their number of CTAs; 0: it cannot place one (few SMs per GPC, a
// share of the SMs only).  The question is put once per kernel (which has one of these), device and number; launches that are
// refused all the same (a stream with fewer SMs than the device) fall back in launch_merging.
struct ClusterRoom {
  std::atomic<uint16_t> known[64][kClusterCtas] = {};      // answer + 1
  template <typename Kernel> int operator()(Kernel kernel, const cudaLaunchConfig_t& like, int ctas) {
    int dev = -1;
    if (ctas < 1 || ctas > kClusterCtas || cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::atomic<uint16_t>& k = known[dev][ctas - 1];
    int n = (int)k.load(std::memory_order_relaxed) - 1;
    if (n < 0) {
      cudaLaunchConfig_t cfg = like;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = attr[0].val.clusterDim.z = 1;
      attr[0].val.clusterDim.y = ctas;
      cfg.attrs = attr; cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&n, reinterpret_cast<const void*>(kernel), &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
      n = std::min(std::max(n, 0), 65534);
      k.store((uint16_t)(n + 1), std::memory_order_relaxed);
    }
    return n;
  }
};

struct ExportPtrs {
  uint8_t *k_code, *v_code;
  uint16_t *k_scale, *k_zero, *v_scale, *v_zero;
  float* norm;
  uint16_t *k_sink, *v_sink, *k_recent, *v_recent;
};

int launch_prefill(const Layout& L, unsigned char* cache, unsigned char* ws, const __half* K, const __half* V, int N,
                   cudaStream_t st);
// Prefill of an inner-grouped cache (N > 0): two launches.  K, V: [U][N][128] fp16.
int launch_prefill_inner(const Layout& L, const Counts& cn, unsigned char* cache, unsigned char* ws, const __half* K,
                         const __half* V, cudaStream_t st);
// fp16 windows, counts and norms (1) of any cache: all that an empty or an unquantised cache needs.
int launch_prefill_windows(const Layout& L, const Counts& cn, unsigned char* cache, const __half* K, const __half* V,
                           cudaStream_t st);
int launch_append(const Layout& L, unsigned char* cache, const __half* k_new, const __half* v_new, int N_after,
                  cudaStream_t st, int late_wait = 0);
int launch_export(const Layout& L, const unsigned char* cache, int N, const ExportPtrs& e, cudaStream_t st);
// The inverse: fills the cache (packed records, windows, norms, counts) for N tokens from canonical arrays.
int launch_import(const Layout& L, unsigned char* cache, int N, const ExportPtrs& e, cudaStream_t st);

// Generic SIMT decode (any store kinds, bits, group sizes): split kernel + merge kernel.
int launch_decode_simt(const Layout& L, const unsigned char* cache, unsigned char* ws, int N, const __half* q,
                       __half* out, int n_splits, cudaStream_t st);

// Warp-MMA decode for the INNER layout.  Returns -2 if the configuration is not supported.
// pages_host: a paged cache's page list on the host (optional: saves the kernel its look-ups in device memory).
int launch_decode_mma(const Layout& L, const unsigned char* cache, unsigned char* ws, int N, const __half* q,
                      __half* out, int n_splits, cudaStream_t st, int n_q = 1, float* multi_partials = nullptr,
                      int N_safe = 0, const uint32_t* pages_host = nullptr, int n_pages_host = 0);
int launch_decode_mma_batched(const Layout& L, int n, const unsigned char* const* caches, unsigned char* const* wss,
                              const int* Ns, const int* Ns_safe, const __half* q, __half* out, int n_splits,
                              cudaStream_t st);
int launch_append_batched(const Layout& L, int n, unsigned char* const* caches, const int* Ns_after, const int* late_wait,
                          const __half* k_new, const __half* v_new, cudaStream_t st);
bool decode_mma_supported(const Layout& L);

// Warp-MMA decode over an unquantised fp16 cache (grouping = FP16).  Returns -2 for other layouts.
int launch_decode_fp16(const Layout& L, const unsigned char* cache, unsigned char* ws, int N, const __half* q,
                       __half* out, int n_splits, cudaStream_t st);
// Test support: a one-warp kernel whose bounded wait runs out and sets the workspace's error word.
int launch_wait_expiry_selftest(const Layout& L, unsigned char* ws, cudaStream_t st);
void decode_mma_set_chunks_per_iter(int n);   // tuning: 32-token chunks per loop iteration (1 or 2)
void decode_mma_set_ablation(int mask);       // timing experiments: bit 0 / 1 = no key-side / value-side work in the loop


}  // namespace iq
