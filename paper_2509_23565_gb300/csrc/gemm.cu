// Launch configuration of the product kernel: shared-memory ring and dispatch
// over the update modes of C (each compiled in its own source file).
#include <cstddef>

#include "emul_internal.h"

namespace emul {

// Ring stages of a launch and its shared-memory bytes.  A stage holds s tiles
// of A (128 rows x kBK) and s of B (bn rows, half of them in a CTA pair); 1 KB
// aligns the ring, 2 KB are left for the static arrays, and `stash` takes two
// bytes per entry of the CTA's 128 x bn tile.
int gemm_stages(const GemmConfig& cfg, int s, size_t* smem_bytes) {
  const size_t b_rows = cfg.var == Variant::kPair ? cfg.bn / 2 : cfg.bn;
  const size_t stage = static_cast<size_t>(s) * (128 + b_rows) * kBK * 2;
  const size_t stash = cfg.stash ? static_cast<size_t>(128) * cfg.bn * 2 : 0;
  int stages = static_cast<int>((232448 - 1024 - 2048 - stash) / stage);
  if (stages > kMaxStagesCfg) stages = kMaxStagesCfg;
  if (smem_bytes) *smem_bytes = stages * stage + stash + 1024;
  return stages;
}

cudaError_t launch_gemm(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                        const GemmArgs& args, int grid, int stages, size_t smem_bytes) {
  if (args.alpha == -1.0 && args.beta == 1.0) return launch_gemm_sub(st, cfg, tmA, tmB, args, grid, stages, smem_bytes);
  if (args.alpha == 1.0 && args.beta == 0.0) return launch_gemm_set(st, cfg, tmA, tmB, args, grid, stages, smem_bytes);
  return launch_gemm_general(st, cfg, tmA, tmB, args, grid, stages, smem_bytes);
}

}  // namespace emul
