// The product kernel (gemm_kernel.cuh) with the C update C <- alpha D + beta C.
#include "gemm_kernel.cuh"

namespace emul {

cudaError_t launch_gemm_general(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                        const GemmArgs& args, int grid, int stages, size_t smem_bytes) {
  return launch_upd<kGeneral>(st, cfg, tmA, tmB, args, grid, stages, smem_bytes);
}

}  // namespace emul
