// Scale extraction and slicing of GEMM operands (arXiv 2509.23565, Section 2,
// Eq. 1-4): per row r of a rows x k operand,
//   e_r = smallest e with max_c |x(r,c)| < 2^e   (0 for a zero row, NONFINITE for Inf/NaN),
//   N   = trunc(x * 2^(7s - e_r)),  |N| < 2^(7s),
//   slice p (0 = most significant) = sign(x) * ((|N| >> 7(s-1-p)) & 127).
// Everything is integer arithmetic on the IEEE-754 bit fields; no FP64
// instruction is issued.  Slices are stored as BF16 bit patterns (every
// integer in [-127, 127] is exact in BF16), plane-major and K-contiguous:
//   out[(p*rows + r)*ldk + c], the layout the TMA loads of the product read.
#include <cstdint>
#include <cuda_runtime.h>

#include "emul_internal.h"
#include "launch.h"
#include "ptx.cuh"
#include "slice.cuh"

namespace emul {
namespace {

constexpr int kSplitThreads = 256;
constexpr int kSplitRows = 8;            // rows per block

struct SplitArgs {
  const double* X;
  long rs, cs;
  int rows, k;
  int32_t* exps;
  uint16_t* out;
  long ldk;
  int blocks;       // blocks of this operand
};

// One block slices eight rows.  Rows contiguous in memory (rs = 1): a warp
// covers the 8 rows x 4 groups of eight k, so a column of the tile is one 64-byte
// piece and the four groups of a row are 64 bytes of a plane; k contiguous: a
// warp takes one row, 32 groups at a time.  KEEP: all of K fits in one pass, the elements
// stay in registers between the maximum and the digits; otherwise the second
// pass reads them again (from L2).  Bound by memory for tall operands
// (8 B read, 2s B written per element), by latency for small ones; the blocks
// are small so that a 256-row operand already fills 32 SMs, and both operands
// of a product go in one launch.
template <int S, bool KEEP>
__global__ void __launch_bounds__(kSplitThreads) split_kernel(const SplitArgs a0, const SplitArgs a1) {
  __shared__ uint32_t up_s[kSplitThreads / 32][kSplitRows];
  __shared__ unsigned long long full_s[kSplitRows];
  grid_launch();
  grid_wait();
  const bool second = static_cast<int>(blockIdx.x) >= a0.blocks;
  const SplitArgs& a = second ? a1 : a0;
  const int r0 = (static_cast<int>(blockIdx.x) - (second ? a0.blocks : 0)) * kSplitRows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool by_rows = a.rs == 1;
  const int rl = by_rows ? lane & 7 : warp;                       // row within the block
  const int g0 = by_rows ? warp * 4 + (lane >> 3) : lane;         // first K group of this thread
  constexpr int gstep = 32;
  const int groups = static_cast<int>(a.ldk >> 3);
  const int r = r0 + rl;
  const bool row_ok = r < a.rows;
  const uint64_t* row = reinterpret_cast<const uint64_t*>(a.X) + r * a.rs;
  auto load = [&](int g, uint64_t (&u)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = 8 * g + j;
      u[j] = row_ok && c < a.k ? row[c * a.cs] : 0ull;
    }
  };
  // the maximum over the threads that share a row: lanes 8 and 16 apart, then
  // the warps (rows contiguous), or the warp (k contiguous)
  uint64_t u[8];
  uint32_t up = 0;
  if (KEEP) {
    load(g0, u);
    up = max_upper8(u);
  } else {
    for (int g = g0; g < groups; g += gstep) {
      load(g, u);
      up = max(up, max_upper8(u));
    }
  }
  if (by_rows) {
    up = max(up, __shfl_xor_sync(0xFFFFFFFFu, up, 8));
    up = max(up, __shfl_xor_sync(0xFFFFFFFFu, up, 16));
    if (lane < kSplitRows) up_s[warp][lane] = up;
  } else {
    up = __reduce_max_sync(0xFFFFFFFFu, up);
  }
  if (threadIdx.x < kSplitRows) full_s[threadIdx.x] = 0;
  __syncthreads();
  if (by_rows) {
#pragma unroll
    for (int w = 0; w < kSplitThreads / 32; ++w) up = max(up, up_s[w][rl]);
  }
  int e = exponent_of_upper(up);
  if (__syncthreads_or(row_ok && needs_full_max(up))) {
    // some row is all zeros and subnormals: the full patterns decide
    if (row_ok && needs_full_max(up)) {
      uint64_t mx = 0;
      if (KEEP) {
        mx = max_bits8(u);
      } else {
        for (int g = g0; g < groups; g += gstep) {
          load(g, u);
          const uint64_t v = max_bits8(u);
          mx = v > mx ? v : mx;
        }
      }
      atomicMax(&full_s[rl], static_cast<unsigned long long>(mx));
    }
    __syncthreads();
    if (needs_full_max(up)) e = exponent_of_maxbits(full_s[rl]);
  }
  if (!row_ok) return;
  if (g0 == 0) a.exps[r] = e;
  if (KEEP) {
    if (g0 < groups)
      slice8<S>(u, e, [&](int p, uint4 w) {
        *reinterpret_cast<uint4*>(a.out + (static_cast<long>(p) * a.rows + r) * a.ldk + 8 * g0) = w;
      });
  } else {
    for (int g = g0; g < groups; g += gstep) {
      load(g, u);
      slice8<S>(u, e, [&](int p, uint4 w) {
        *reinterpret_cast<uint4*>(a.out + (static_cast<long>(p) * a.rows + r) * a.ldk + 8 * g) = w;
      });
    }
  }
}

template <int S>
cudaError_t launch_s(cudaStream_t st, const SplitArgs& a, const SplitArgs& b) {
  const int grid = a.blocks + b.blocks;
  const long ldk = a.ldk > b.ldk ? a.ldk : b.ldk;
  if (ldk <= 256)
    return launch_dependent(split_kernel<S, true>, dim3(grid), dim3(kSplitThreads), 0, st, a, b);
  return launch_dependent(split_kernel<S, false>, dim3(grid), dim3(kSplitThreads), 0, st, a, b);
}

SplitArgs make_args(int rows, int k, const double* X, long rs, long cs, int32_t* exps, uint16_t* out, long ldk) {
  return SplitArgs{X, rs, cs, rows, k, exps, out, ldk, rows > 0 ? (rows + kSplitRows - 1) / kSplitRows : 0};
}

cudaError_t dispatch(cudaStream_t st, int s, const SplitArgs& a, const SplitArgs& b) {
  if (a.blocks + b.blocks == 0) return cudaSuccess;
  switch (s) {
    case 1: return launch_s<1>(st, a, b);
    case 2: return launch_s<2>(st, a, b);
    case 3: return launch_s<3>(st, a, b);
    case 4: return launch_s<4>(st, a, b);
    case 5: return launch_s<5>(st, a, b);
    case 6: return launch_s<6>(st, a, b);
    case 7: return launch_s<7>(st, a, b);
    case 8: return launch_s<8>(st, a, b);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_split(cudaStream_t st, int rows, int k, const double* X, long rs, long cs, int s, int32_t* exps,
                         uint16_t* out, long ldk) {
  return dispatch(st, s, make_args(rows, k, X, rs, cs, exps, out, ldk), make_args(0, k, X, rs, cs, exps, out, 0));
}

cudaError_t launch_split2(cudaStream_t st, int k, int s, long ldk, int rows_a, const double* A, long ars, long acs,
                          int32_t* ea, uint16_t* sa, int rows_b, const double* B, long brs, long bcs, int32_t* fb,
                          uint16_t* sb) {
  return dispatch(st, s, make_args(rows_a, k, A, ars, acs, ea, sa, ldk), make_args(rows_b, k, B, brs, bcs, fb, sb, ldk));
}

}  // namespace emul
