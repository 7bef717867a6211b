// Launch and occupancy of the fine tile kernel, included by the files that instantiate it.
#pragma once

#include <algorithm>
#include <map>
#include <mutex>

#include "fine_tile.cuh"

namespace bsp {

constexpr size_t kFineSpreadSmem = 120 * 1024;   // above half an SM's shared memory

template <int TC, int TR>
static int fine_tile_config(int C, bool spread, cudaLaunchConfig_t& cfg, cudaLaunchAttribute& attr) {
  const size_t b = FineShape<TC, TR>::BYTES, smem = spread ? std::max(b, kFineSpreadSmem) : b;
  auto kern = fine_tile_kernel<TC, TR>;
  BS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::max(b, kFineSpreadSmem)));
  if (C > 8) BS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  cfg = {};
  cfg.gridDim = dim3(C, 1, 1);
  cfg.blockDim = dim3(kFineThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = C;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return BS_OK;
}

template <int TC, int TR>
int fine_tile_launch(const FineBatch& fb, const FineLaunch& fl, bool spread, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  int rc = fine_tile_config<TC, TR>(fb.C, spread, cfg, attr);
  if (rc) return rc;
  cfg.gridDim = dim3(fb.C, fb.ntx * fb.nty, fb.n);
  cfg.stream = s;
  BS_CUDA_TRY(cudaLaunchKernelEx(&cfg, fine_tile_kernel<TC, TR>, fb, fl));
  return BS_OK;
}

// Measured once per device and cluster size through the occupancy API.
template <int TC, int TR>
int fine_tile_capacity(int C) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find({dev, C});
  if (it != cache.end()) return it->second;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  int n = 0;
  if (fine_tile_config<TC, TR>(C, false, cfg, attr) != BS_OK ||
      cudaOccupancyMaxActiveClusters(&n, fine_tile_kernel<TC, TR>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  cache[{dev, C}] = n;
  return n;
}

#define BS_FINE_INSTANCE(TC, TR)                                                            \
  template int fine_tile_launch<TC, TR>(const FineBatch&, const FineLaunch&, bool, cudaStream_t); \
  template int fine_tile_capacity<TC, TR>(int);

}  // namespace bsp
