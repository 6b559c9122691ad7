// Launch of a kernel that may start before the one ahead of it in the stream has
// ended (programmatic stream serialization).  The kernel calls grid_wait()
// (ptx.cuh) before its first access to global memory, so the order of the work
// is that of the stream; what overlaps is the launch itself and the kernel's
// set-up.  Dependent kernels launched the plain way end on a grid of 2.05 us
// (every chain of 4 to 120 us kernels measured here took a multiple of 2.048 us
// per kernel), and the panels of the factorizations are chains of such kernels:
// a product of 64 x 64 x 64 in a loop took 14.3 us that way and takes 11.8, LU at
// n = 4001 17.8 ms and 17.2, Cholesky at 12000 36.6 and 35.9, LU without pivoting
// at 6144 23.9 and 22.5.  Cooperative kernels are launched the plain way.
#pragma once
#include <utility>

#include <cuda_runtime.h>

namespace emul {

// dependent = false launches the same kernel the plain way: on the second stream,
// whose kernels with the attribute did not overlap the first stream's (Cholesky at
// 12000 with its diagonal blocks there 32.8 ms, and 27.3 with plain launches).
template <typename... Params, typename... Args>
cudaError_t launch_chained(bool dependent, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem,
                           cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}

template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                             Args&&... args) {
  return launch_chained(true, kernel, grid, block, smem, st, std::forward<Args>(args)...);
}

}  // namespace emul
