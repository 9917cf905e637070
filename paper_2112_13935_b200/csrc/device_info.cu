// What the launch rules need to know about the current device: how many SMs it has, and how many clusters of one CTA per SM
// it runs at once.  Clusters do not straddle GPCs, and GPCs differ in the SMs they have left, so the second does not follow from the
// first: 148 SMs hold 74 clusters of two, 45 of three, 33 of four (not 37), 26 of five, 22 of six, and 15 of seven or eight (not 21 and 18); a launch of one more runs as two waves.
#include <cuda_runtime.h>

#include <atomic>

#include "aet_kernels.h"

namespace aet {
namespace {

constexpr int kMaxDevices = 64, kThreads = 512, kSmem = 200 * 1024;   // as the round kernels: nobody shares an SM

__global__ void __launch_bounds__(kThreads, 1) whole_sm_kernel(float* p) {   // never launched
  extern __shared__ float s[];
  if (p) p[threadIdx.x] = s[threadIdx.x];
}

// [device][CTAs], one more than the answer; 0: not asked yet.  Two host threads may ask at once and store the same value.
std::atomic<uint32_t> g_fit[kMaxDevices][9] = {};

cudaError_t at_once_on(int dev, uint32_t cluster, uint32_t* out) {
  std::atomic<uint32_t>* known = dev >= 0 && dev < kMaxDevices ? &g_fit[dev][cluster] : nullptr;
  uint32_t n = known ? known->load(std::memory_order_relaxed) : 0;
  if (!n) {
    int v = 0;
    cudaError_t e;
    if (cluster == 1) {
      e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    } else {
      e = cudaFuncSetAttribute(whole_sm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(cluster, 1, 1);
      cfg.blockDim = dim3(kThreads, 1, 1);
      cfg.dynamicSmemBytes = kSmem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = cluster;
      attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&v, whole_sm_kernel, &cfg);
    }
    if (e != cudaSuccess) return e;
    n = (uint32_t)(v > 0 ? v : 0) + 1;   // (a part of a device may have no place for a wide cluster at all)
    if (known) known->store(n, std::memory_order_relaxed);
  }
  *out = n - 1;
  return cudaSuccess;
}

}  // namespace

cudaError_t clusters_at_once(uint32_t cluster, uint32_t* out) {
  int dev = 0;
  if (cluster < 1 || cluster > 8) return cudaErrorInvalidValue;
  if (const cudaError_t e = cudaGetDevice(&dev)) return e;
  return at_once_on(dev, cluster, out);
}

cudaError_t clusters_at_once(uint32_t (&out)[9]) {
  int dev = 0;
  if (const cudaError_t e = cudaGetDevice(&dev)) return e;
  out[0] = 0;
  for (uint32_t cl = 1; cl <= 8; ++cl)
    if (const cudaError_t e = at_once_on(dev, cl, &out[cl])) return e;
  return cudaSuccess;
}

}  // namespace aet
