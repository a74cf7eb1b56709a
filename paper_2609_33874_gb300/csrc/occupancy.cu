// What the launchers ask the current device: its SMs, and how many CTA pairs of a
// kernel it holds at once.
#include <algorithm>
#include <atomic>

#include "jet_internal.h"
#include "pair_cache.h"

namespace jet {

int sm_count() {
  static std::atomic<int> kept[64];
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return 0;
  if (dev < 64 && (n = kept[dev].load(std::memory_order_relaxed)) > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (dev < 64) kept[dev].store(n, std::memory_order_relaxed);
  return n;
}

int resident_pairs(const void* kernel, int threads, size_t smem) {
  static PairCache cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  const int n = cache.get(dev, kernel, smem, [&] {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(unsigned(threads));
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute cl{};
    cl.id = cudaLaunchAttributeClusterDimension;
    cl.val.clusterDim.x = 2;
    cl.val.clusterDim.y = 1;
    cl.val.clusterDim.z = 1;
    cfg.attrs = &cl;
    cfg.numAttrs = 1;
    int pairs = 0;
    if (cudaOccupancyMaxActiveClusters(&pairs, kernel, &cfg) == cudaSuccess) return pairs;
    cudaGetLastError();
    return 0;
  });
  return n > 0 ? n : std::max(1, sm_count() / 2);
}

}  // namespace jet
