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
constexpr int kSplitRows = 8;            // rows per block, with 32 groups of eight k at a time
constexpr int kSplitTall = 32;           // the same with 8 groups, for k <= 64 and
constexpr int kSplitTallRows = 32768;    // at least so many rows in the launch

struct SplitArgs {
  const double* X;
  long rs, cs;
  int rows, k;
  int32_t* exps;
  uint16_t* out;
  long ldk;
  int blocks;       // blocks of this operand
};

// One block slices eight rows (R; 32 of a tall operand with k <= 64, where a row has
// at most 8 groups of eight k for its threads: 100000 x 8 at s = 3 7.3 us, 23.7 with
// eight, 50000 x 64 at s = 7 16.8 and 21.1; 256 x 64 3.0 and 2.2; between, where the
// slicing alone gains a microsecond or two, the product that follows loses as much as
// often as not: 2421 x 8184 x 54 at s = 3 237 and 234, 16384 x 16384 x 64 2728 and 2736).
// Rows contiguous in memory (rs = 1): a warp covers the 8 rows x 4 groups, so a
// column of the tile is one 64-byte piece and the four groups of a row are 64 bytes of
// a plane (R = 32: 32 rows of one group); k contiguous: a warp takes one row, 32
// groups at a time (R = 32: four rows).  KEEP: all of K fits in one pass, the elements
// stay in registers between the maximum and the digits; otherwise the second pass
// reads them again (from L2).  Bound by memory for tall operands (8 B read, 2s B
// written per element), by latency for small ones; the blocks are small so that a
// 256-row operand already fills 32 SMs, and both operands of a product go in one
// launch.
template <int S, bool KEEP, int R>
__global__ void __launch_bounds__(kSplitThreads) split_kernel(const SplitArgs a0, const SplitArgs a1) {
  constexpr int gstep = kSplitThreads / R;      // groups of a row taken at once
  __shared__ uint32_t up_s[kSplitThreads / 32][R];
  __shared__ unsigned long long full_s[R];
  grid_launch();
  grid_wait();
  const bool second = static_cast<int>(blockIdx.x) >= a0.blocks;
  const SplitArgs& a = second ? a1 : a0;
  const int r0 = (static_cast<int>(blockIdx.x) - (second ? a0.blocks : 0)) * R;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool by_rows = a.rs == 1;
  const int tid = threadIdx.x;
  const int rl = by_rows ? tid % R : tid / gstep;                 // row within the block
  const int g0 = by_rows ? tid / R : tid % gstep;                 // first K group of this thread
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
  // the maximum over the threads that share a row: lanes R apart, then the warps
  // (rows contiguous), or gstep neighbouring lanes (k contiguous)
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
#pragma unroll
    for (int o = R; o < 32; o *= 2) up = max(up, __shfl_xor_sync(0xFFFFFFFFu, up, o));
    if (lane < R) up_s[warp][lane] = up;
  } else if (gstep == 32) {
    up = __reduce_max_sync(0xFFFFFFFFu, up);
  } else {
#pragma unroll
    for (int o = 1; o < gstep; o *= 2) up = max(up, __shfl_xor_sync(0xFFFFFFFFu, up, o));
  }
  if (tid < R) full_s[tid] = 0;
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
cudaError_t launch_s(cudaStream_t st, SplitArgs a, SplitArgs b) {
  const long ldk = a.ldk > b.ldk ? a.ldk : b.ldk;
  const bool tall = ldk <= kSplitThreads / kSplitTall * 8 && a.rows + b.rows >= kSplitTallRows;
  const int R = tall ? kSplitTall : kSplitRows;
  a.blocks = (a.rows + R - 1) / R;
  b.blocks = (b.rows + R - 1) / R;
  const dim3 grid(a.blocks + b.blocks), block(kSplitThreads);
  if (tall) return launch_dependent(split_kernel<S, true, kSplitTall>, grid, block, 0, st, a, b);
  if (ldk <= 256) return launch_dependent(split_kernel<S, true, kSplitRows>, grid, block, 0, st, a, b);
  return launch_dependent(split_kernel<S, false, kSplitRows>, grid, block, 0, st, a, b);
}

SplitArgs make_args(int rows, int k, const double* X, long rs, long cs, int32_t* exps, uint16_t* out, long ldk) {
  return SplitArgs{X, rs, cs, rows > 0 ? rows : 0, k, exps, out, ldk, 0};
}

cudaError_t dispatch(cudaStream_t st, int s, const SplitArgs& a, const SplitArgs& b) {
  if (a.rows + b.rows == 0) return cudaSuccess;
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
