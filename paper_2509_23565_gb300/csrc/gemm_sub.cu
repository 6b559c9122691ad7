// The product kernel (gemm_kernel.cuh) with the C update C <- C - D (the Schur update).
#include <map>
#include <mutex>
#include <utility>

#include "gemm_kernel.cuh"

namespace emul {

cudaError_t launch_gemm_sub(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                        const GemmArgs& args, int grid, int stages, size_t smem_bytes) {
  return launch_upd<kSub>(st, cfg, tmA, tmB, args, grid, stages, smem_bytes);
}

// CTA pairs of the product kernel that can be resident at once with this much
// shared memory (0: none, e.g. on a partition without two free SMs side by side).
int gemm_pair_capacity(size_t smem_bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, size_t>, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  const auto key = std::make_pair(dev, smem_bytes);
  const auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  auto kern = gemm_kernel<false, 128, kSub, true, false>;
  int pairs = 0;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem) == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem_bytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&pairs, kern, &cfg) != cudaSuccess) pairs = 0;
  }
  cudaGetLastError();   // a failed query leaves no error behind
  cache[key] = pairs;
  return pairs;
}

}  // namespace emul
