// The product kernel (gemm_kernel.cuh) with the C update C <- D.
#include "gemm_kernel.cuh"

namespace emul {

cudaError_t launch_gemm_set(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                        const GemmArgs& args, int grid, int stages, size_t smem_bytes) {
  return launch_upd<kSet>(st, cfg, tmA, tmB, args, grid, stages, smem_bytes);
}

}  // namespace emul
