// LU without pivoting whose every third-order step runs through the emulated
// product: the Level-3-only factorization arXiv 2509.23565 times for blocking
// factors 256 to 2048 (Section 8), with the Schur update of Eq. 7.
//
// Step j0 (right-looking, block nb):
//   1. the panel A[j0:n, j0:j0+jb] is factored by recursive halving.  A leaf
//      (<= 64 columns) factors its diagonal block in FP64 on one cluster of eight
//      CTAs and forms the inverses of both triangular factors, a warp per column;
//      its rows below become L21 = A21 U11^-1 through the emulated product.  An inner node
//      forms U12 = L11^-1 A12 and the Schur update of the rows below with the
//      emulated product, recurses into its right half, and joins the two
//      halves' unit-lower inverses, X21 = -X22 (L21 X11);
//   2. U12 = X A12 with X = L11^-1 of the whole block (emulated product);
//   3. A22 <- A22 - L21 U12 (emulated product, alpha = -1, beta = 1).
// The Schur updates and U12 run as products over K chunks of at most 1024
// (see gemm_kchunks).
// No row is ever exchanged, so the factorization is stable only for matrices
// that need no pivoting (diagonally dominant, SPD).
#include <cuda_runtime.h>

#include "handle.h"
#include "launch.h"
#include "ptx.cuh"

namespace emul {
namespace {

constexpr int kNpLeaf = 64;           // widest diagonal block factored in one launch
constexpr int kNpWarps = 8;           // the leaf's warps, columns dealt round
constexpr int kNpChunk = 1024;        // K of one emulated product in the Schur updates
constexpr size_t kNpAl = 256;

inline size_t np_al(size_t x) { return (x + kNpAl - 1) / kNpAl * kNpAl; }

// The w x w diagonal block at A[d.., d..] (w <= 64) is factored in place
// without pivoting, A = L U (L unit lower).  A zero pivot leaves its column
// unscaled and records its 1-based index in *info unless an earlier one is
// there.
//
// FP64 retires 1.68 FMA per clock per SM, a warp's DFMA occupies its
// sub-partition for 64-76 cycles and a division takes 560, so what counts is the
// chain from pivot to pivot and that no FP64 instruction is wasted.  np_factor:
// eight warps of a CTA hold 32 columns in registers, warp g the columns g, g + 8,
// ..., rows across the lanes, so a pivot column lies in one warp: its owner
// updates it first, takes the reciprocal, scales, publishes the multipliers in
// shared memory (a place of its own for each pivot) and arrives at the step's
// barrier before it updates its other columns; the other warps meet it there after
// theirs.  The pivot row comes by shuffles.
//
// The left 32 columns and then the lower right 32 x 32 are factored that way by
// CTA 0 of a cluster.  In between the right 32 columns take the left ones'
// pivots on all eight CTAs, a warp per column, with the multipliers and the
// results carried through distributed shared memory: on one SM these updates kept
// its FP64 units busy for 1000 to 2000 cycles a pivot, twice the chain's length
// (57 us for 64 x 64 that way, 47 here).  Every entry sees the same operations in the
// same order as in a plain right-looking elimination.
__device__ __noinline__ double np_recip(double p) { return 1.0 / p; }
// x == 0 by the bits (an FP64 comparison would take a DFMA's 64 cycles)
__device__ __forceinline__ bool np_zero(double x) {
  return (static_cast<unsigned long long>(__double_as_longlong(x)) << 1) == 0;
}

constexpr int kNpHalf = kNpLeaf / 2;
constexpr int kNpCluster = 8;                              // CTAs of a leaf
constexpr int kNpRight = kNpHalf / kNpCluster;             // right columns of each
constexpr int kNpCols = kNpHalf / kNpWarps;

// Factors the 32 H x 32 columns v (v[s][h]: row lane + 32 h of column g + 8 s), of
// which the leading w count; pivot k's multipliers go to M[k].  `first` is the
// global index of the first pivot.
template <int H>
__device__ __forceinline__ void np_factor(double (&v)[kNpCols][H], int g, int lane, int w, double (*M)[kNpLeaf],
                                          int first, int32_t* info) {
  // multipliers of pivot k from its column (in registers c of the owner)
  auto scale = [&](int k, double (&c)[H]) {
    const double p = __shfl_sync(0xFFFFFFFFu, c[0], k);
    const double r = np_zero(p) ? 0.0 : np_recip(p);
    if (np_zero(p) && lane == 0) atomicCAS(info, 0, first + k + 1);
    if (!np_zero(r)) {
      if (lane > k) c[0] *= r;
      if (H == 2) c[H - 1] *= r;
    }
    M[k][lane] = lane > k ? c[0] : 0.0;
    if (H == 2) M[k][lane + 32] = c[H - 1];
    // barriers 1 and 2 in turn; the owner has published and does not wait
    __syncwarp();
    if (k + 1 < w) asm volatile("bar.arrive %0, %1;" ::"r"(1 + (k & 1)), "n"(32 * kNpWarps) : "memory");
  };
  if (g == 0) scale(0, v[0]);
  // pivots k = 8 so + kk; the inner loop stays rolled (32 copies of a step would
  // run from the instruction cache's misses)
#pragma unroll
  for (int so = 0; so < kNpCols; ++so) {
#pragma unroll 1
    for (int kk = 0; kk < kNpWarps; ++kk) {
      const int k = kNpWarps * so + kk;
      if (k + 1 >= w) break;
      if (g != kk) asm volatile("bar.sync %0, %1;" ::"r"(1 + (k & 1)), "n"(32 * kNpWarps) : "memory");
      const double l0 = M[k][lane], l1 = H == 2 ? M[k][lane + 32] : 0.0;
      auto update = [&](double (&c)[H]) {
        const double u = __shfl_sync(0xFFFFFFFFu, c[0], k);
        if (lane > k) c[0] = fma(-l0, u, c[0]);
        if (H == 2) c[H - 1] = fma(-l1, u, c[H - 1]);
      };
      // the next pivot's column first, and its multipliers
      const bool mine = g == (kk + 1) % kNpWarps;
      if (mine) {
        if (kk + 1 < kNpWarps) {
          update(v[so]);
          scale(k + 1, v[so]);
        } else if (so + 1 < kNpCols) {
          update(v[so + 1 < kNpCols ? so + 1 : so]);
          scale(k + 1, v[so + 1 < kNpCols ? so + 1 : so]);
        }
      }
      const int snext = kk + 1 < kNpWarps ? so : so + 1;
#pragma unroll
      for (int s = so; s < kNpCols; ++s)
        if ((s > so || g > kk) && !(mine && s == snext)) update(v[s]);
    }
  }
}

__global__ void __cluster_dims__(kNpCluster, 1, 1) __launch_bounds__(32 * kNpWarps, 1)
    np_leaf_kernel(double* A, long lda, int d, int w, int32_t* info) {
  __shared__ double M[kNpHalf][kNpLeaf];       // multipliers of the left columns' pivots
  __shared__ double S[kNpHalf][kNpHalf];       // CTA 0: S[j][i], the lower right block
  grid_launch();
  grid_wait();
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int b = static_cast<int>(cluster_rank());
  if (w <= kNpHalf && b != 0) return;          // (no cluster barrier then)
  double* D = A + d + static_cast<long>(d) * lda;
  // beyond w the block is the identity: nothing there changes or is stored
  auto load = [&](int i, int j) { return i < w && j < w ? D[i + static_cast<long>(j) * lda] : (i == j ? 1.0 : 0.0); };
  const int jr = kNpHalf + kNpRight * b + g;   // this warp's right column
  double c0 = 0.0, c1 = 0.0;
  if (w > kNpHalf && g < kNpRight) {
    c0 = load(lane, jr);
    c1 = load(lane + 32, jr);
  }
  if (b == 0) {
    double v[kNpCols][2];
#pragma unroll
    for (int s = 0; s < kNpCols; ++s)
#pragma unroll
      for (int h = 0; h < 2; ++h) v[s][h] = load(lane + 32 * h, g + kNpWarps * s);
    np_factor<2>(v, g, lane, w < kNpHalf ? w : kNpHalf, M, d, info);
#pragma unroll
    for (int s = 0; s < kNpCols; ++s)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h, j = g + kNpWarps * s;
        if (i < w && j < w) D[i + static_cast<long>(j) * lda] = v[s][h];
      }
  }
  if (w <= kNpHalf) return;
  cluster_sync();                              // CTA 0's multipliers stand
  if (b != 0) {
    const uint32_t from = mapa_addr(smem_u32(&M[0][0]), 0) + 8u * threadIdx.x;
    constexpr int kEach = kNpHalf * kNpLeaf / (32 * kNpWarps);
    double x[kEach];
#pragma unroll
    for (int q = 0; q < kEach; ++q) x[q] = ld_cluster_f64(from + 8u * 32 * kNpWarps * q);
#pragma unroll
    for (int q = 0; q < kEach; ++q) (&M[0][0])[threadIdx.x + 32 * kNpWarps * q] = x[q];
    __syncthreads();
  }
  if (g < kNpRight) {
#pragma unroll 4
    for (int k = 0; k < kNpHalf; ++k) {
      const double u = __shfl_sync(0xFFFFFFFFu, c0, k);
      if (lane > k) c0 = fma(-M[k][lane], u, c0);
      c1 = fma(-M[k][lane + 32], u, c1);
    }
    if (jr < w) D[lane + static_cast<long>(jr) * lda] = c0;
    st_cluster_f64(mapa_addr(smem_u32(&S[jr - kNpHalf][lane]), 0), c1);
  }
  cluster_sync();                              // the lower right block stands in CTA 0
  if (b != 0) return;
  double v[kNpCols][1];
#pragma unroll
  for (int s = 0; s < kNpCols; ++s) v[s][0] = S[g + kNpWarps * s][lane];
  np_factor<1>(v, g, lane, w - kNpHalf, M, d + kNpHalf, info);
#pragma unroll
  for (int s = 0; s < kNpCols; ++s) {
    const int i = kNpHalf + lane, j = kNpHalf + g + kNpWarps * s;
    if (i < w && j < w) D[i + static_cast<long>(j) * lda] = v[s][0];
  }
}

// Inverses of the leaf's factors: X <- L^-1 (ld ldx, zeros above the diagonal)
// and Y <- U^-1 (ld w, zeros below; an infinite reciprocal for a zero pivot).
// One warp per column of X or Y and four columns per block, so every warp has a
// sub-partition's FP64 unit to itself: a step is a shuffle and one or two DFMAs.
// Row k of a column, once final, is broadcast; column j of X starts at row j, of Y
// at row j and goes up.
constexpr int kInvCols = 4;
__global__ void __launch_bounds__(32 * kInvCols) np_inverse_kernel(const double* A, long lda, int d, int w, double* X,
                                                                  long ldx, double* Y) {
  __shared__ double S[kNpLeaf][kNpLeaf + 1];      // S[k][i] = (L\U)(i, k)
  __shared__ double rdiag[kNpLeaf];
  grid_launch();
  grid_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double* D = A + d + static_cast<long>(d) * lda;
  // sixteen loads in flight per thread
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    double v[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int e = threadIdx.x + (16 * h + q) * 32 * kInvCols, i = e & (kNpLeaf - 1), k = e / kNpLeaf;
      v[q] = i < w && k < w ? D[i + static_cast<long>(k) * lda] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 16; ++q) {
      const int e = threadIdx.x + (16 * h + q) * 32 * kInvCols;
      S[e / kNpLeaf][e & (kNpLeaf - 1)] = v[q];
    }
  }
  __syncthreads();
  const bool lower = blockIdx.y == 0;
  if (!lower) {
    if (threadIdx.x < w) {
      const double p = S[threadIdx.x][threadIdx.x];
      const double r = p != 0.0 ? 1.0 / p : 0.0;
      rdiag[threadIdx.x] = r != 0.0 ? r : __longlong_as_double(0x7FF0000000000000ll);
    }
    __syncthreads();
  }
  const int j = blockIdx.x * kInvCols + warp;
  if (j >= w) return;
  // x0, x1: rows lane and lane + 32 of the column; r0, r1: their final values,
  // kept aside (a finished row, updated with zeros from then on, may meet an infinity)
  double x0 = lane == j ? 1.0 : 0.0, x1 = lane + 32 == j ? 1.0 : 0.0, r0 = 0.0, r1 = 0.0;
  if (lower) {
    const int n0 = w < 32 ? w : 32;
    for (int k = j; k < n0; ++k) {
      const double xk = __shfl_sync(0xFFFFFFFFu, x0, k);
      if (lane == k) r0 = x0;
      x0 = fma(lane > k ? -S[k][lane] : 0.0, xk, x0);
      x1 = fma(-S[k][lane + 32], xk, x1);
    }
    for (int k = j > 32 ? j : 32; k < w; ++k) {
      const double xk = __shfl_sync(0xFFFFFFFFu, x1, k - 32);
      if (lane == k - 32) r1 = x1;
      x1 = fma(lane > k - 32 ? -S[k][lane + 32] : 0.0, xk, x1);
    }
    if (lane < w) X[lane + static_cast<long>(j) * ldx] = r0;
    if (lane + 32 < w) X[lane + 32 + static_cast<long>(j) * ldx] = r1;
  } else {
    const double d0 = lane < w ? rdiag[lane] : 1.0, d1 = lane + 32 < w ? rdiag[lane + 32] : 1.0;
    for (int k = j; k >= 32; --k) {
      const double xv = x1 * d1;
      const double xk = __shfl_sync(0xFFFFFFFFu, xv, k - 32);
      if (lane == k - 32) r1 = xv;
      x0 = fma(-S[k][lane], xk, x0);
      x1 = fma(lane < k - 32 ? -S[k][lane + 32] : 0.0, xk, x1);
    }
    for (int k = j < 31 ? j : 31; k >= 0; --k) {
      const double xv = x0 * d0;
      const double xk = __shfl_sync(0xFFFFFFFFu, xv, k);
      if (lane == k) r0 = xv;
      x0 = fma(lane < k ? -S[k][lane] : 0.0, xk, x0);
    }
    if (lane < w) Y[lane + static_cast<long>(j) * w] = r0;
    if (lane + 32 < w) Y[lane + 32 + static_cast<long>(j) * w] = r1;
  }
}

struct NpBufs {
  double* X;     // jb x jb, ld nb: L11^-1 of the current block
  double* Y;     // 64 x 64: U^-1 of the current leaf
  double* T;     // scratch for the inverse join, up to nb x nb
  double* U;     // U12 of the current block, jb x (n - j0 - jb), ld jb
  long ldx;
};

// C <- beta C + alpha A B as consecutive emulated products over K chunks of at
// most kNpChunk; C must not overlap A or B, and is read and written once per chunk.
// Each chunk is rounded once, and these roundings are part of the result, so the
// chunks are the same for every m.  The one-CTA variants (at most 128 rows) need them
// for speed: up to 1024 level 2 is one accumulator job (1040 products of 127^2 per
// FP32 accumulator); the CTA pairs would take any K at s <= 7.
int gemm_kchunks(emul_handle_t h, int m, int n, int k, double alpha, Operand A, Operand B, double beta, double* C,
                 long ldc, int s) {
  for (int c0 = 0; c0 < k; c0 += kNpChunk) {
    const int kc = k - c0 < kNpChunk ? k - c0 : kNpChunk;
    const int rc = gemm_run(h, m, n, kc, alpha, Operand{A.ptr + c0 * A.cs, A.rs, A.cs},
                            Operand{B.ptr + c0 * B.cs, B.rs, B.cs}, c0 == 0 ? beta : 1.0, C, ldc, s, false, 0,
                            nullptr, 0, 0);
    if (rc) return rc;
  }
  return EMUL_OK;
}

// Split of a w-column panel: the left part a multiple of 16 near w/2.
inline int np_split(int w) {
  const int w1 = (w / 2 + 15) / 16 * 16;
  return w1 < w ? w1 : w / 2;
}

// Factor the panel A[d:n, d:d+w] (no pivoting) and leave L^-1 of its diagonal
// block in X at (d - j0, d - j0), unless the panel is the matrix's last.
int np_panel(emul_handle_t h, double* A, long lda, int n, int j0, int d, int w, int s, int32_t* info,
             const NpBufs& B) {
  double* Xd = B.X + (d - j0) + static_cast<long>(d - j0) * B.ldx;
  if (w <= kNpLeaf) {
    launch_dependent(np_leaf_kernel, dim3(kNpCluster), dim3(32 * kNpWarps), 0, h->stream, A, lda, d, w, info);
    h->launches++;
    const int mb = n - d - w;
    if (mb > 0) {                 // (no row and no column is left to use the last leaf's inverses)
      launch_dependent(np_inverse_kernel, dim3((w + kInvCols - 1) / kInvCols, 2), dim3(32 * kInvCols), 0, h->stream,
                       A, lda, d, w, Xd, B.ldx, B.Y);
      h->launches++;
    }
    int rc = check_cuda(h, cudaGetLastError(), "no-pivot leaf");
    if (rc || mb <= 0) return rc;
    double* A21 = A + (d + w) + static_cast<long>(d) * lda;
    // L21 = A21 U11^-1, written over A21 (both operands are sliced before the product writes)
    return gemm_run(h, mb, w, w, 1.0, Operand{A21, 1, lda}, Operand{B.Y, w, 1}, 0.0, A21, lda, s, false, 0,
                    nullptr, 0, 0);
  }
  const int w1 = np_split(w), w2 = w - w1;
  int rc = np_panel(h, A, lda, n, j0, d, w1, s, info, B);
  if (rc) return rc;
  double* A12 = A + d + static_cast<long>(d + w1) * lda;
  // U12 = L11^-1 A12 (w1 x w2), over A12
  rc = gemm_run(h, w1, w2, w1, 1.0, Operand{Xd, 1, B.ldx}, Operand{A12, lda, 1}, 0.0, A12, lda, s, false, 0, nullptr,
                0, 0);
  if (rc) return rc;
  // Schur update of the right half, every row below the left half's diagonal block
  const double* L21 = A + (d + w1) + static_cast<long>(d) * lda;
  double* A22 = A + (d + w1) + static_cast<long>(d + w1) * lda;
  rc = gemm_kchunks(h, n - d - w1, w2, w1, -1.0, Operand{L21, 1, lda}, Operand{A12, lda, 1}, 1.0, A22, lda, s);
  if (rc) return rc;
  rc = np_panel(h, A, lda, n, j0, d + w1, w2, s, info, B);
  if (rc || d + w == n) return rc;
  // join the inverses: X21 = -X22 (L21 X11), L21 the w2 x w1 block below the left diagonal block
  double* X22 = Xd + w1 + static_cast<long>(w1) * B.ldx;
  double* X21 = Xd + w1;
  rc = gemm_run(h, w2, w1, w1, 1.0, Operand{L21, 1, lda}, Operand{Xd, B.ldx, 1}, 0.0, B.T, w2, s, false, 0, nullptr,
                0, 0);
  if (rc) return rc;
  return gemm_run(h, w2, w1, w2, -1.0, Operand{X22, 1, B.ldx}, Operand{B.T, w2, 1}, 0.0, X21, B.ldx, s, false, 0,
                  nullptr, 0, 0);
}

}  // namespace
}  // namespace emul

extern "C" {

int emul_dgetrf_nopiv(emul_handle_t h, int n, double* A, int lda, int nb, int slices, int32_t* info,
                      emul_stats* stats) {
  using namespace emul;
  if (!h) return EMUL_INVALID_ARG;
  if (nb == 0) nb = 1024;
  if (n < 0 || lda < (n > 1 ? n : 1) || nb < 16 || nb > 4096 || slices < 1 || slices > kMaxSlices ||
      (n > 0 && (!A || !info)))
    return set_error(h, EMUL_INVALID_ARG, "emul_dgetrf_nopiv: invalid argument");
  if (stats) *stats = emul_stats{0, slices, slices, 0, 0.0, static_cast<double>(slices)};
  if (n == 0) return EMUL_OK;
  int rc = check_cuda(h, cudaMemsetAsync(info, 0, sizeof(int32_t), h->stream), "info reset");
  if (rc) return rc;
  const int nbe = nb < n ? nb : n;
  // [product workspace | X (nbe x nbe) | Y (64 x 64) | T (nbe x nbe) | U (nbe x n)]
  const size_t gw = np_al(gemm_workspace_bytes(n, n, nbe, slices, false));
  const size_t xb = np_al(8ull * nbe * nbe), yb = np_al(8ull * kNpLeaf * kNpLeaf);
  rc = reserve_workspace(h, gw + 2 * xb + yb + np_al(8ull * nbe * n));
  if (rc) return rc;
  uint8_t* base = static_cast<uint8_t*>(h->ws);
  const NpBufs B{reinterpret_cast<double*>(base + gw), reinterpret_cast<double*>(base + gw + xb),
                 reinterpret_cast<double*>(base + gw + xb + yb), reinterpret_cast<double*>(base + gw + 2 * xb + yb),
                 nbe};
  for (int j0 = 0; j0 < n; j0 += nb) {
    const int jb = nb < n - j0 ? nb : n - j0;
    int ph = phase_begin(h, EMUL_PHASE_PANEL);
    // the blocks of X above the diagonal are never written: zero them
    rc = check_cuda(h, cudaMemsetAsync(B.X, 0, 8ull * nbe * jb, h->stream), "inverse reset");
    if (rc) return rc;
    rc = np_panel(h, A, lda, n, j0, j0, jb, slices, info, B);
    phase_end(h, ph);
    if (rc) return rc;
    const int m2 = n - j0 - jb;
    if (m2 > 0) {
      ph = phase_begin(h, EMUL_PHASE_U12);
      double* A12 = A + j0 + static_cast<long>(j0 + jb) * lda;
      // U12 = X A12 into U, by K chunks; X is lower triangular, so chunk c only
      // reaches the rows from c on
      for (int c0 = 0; c0 < jb && !rc; c0 += kNpChunk) {
        const int kc = jb - c0 < kNpChunk ? jb - c0 : kNpChunk;
        rc = gemm_run(h, jb - c0, m2, kc, 1.0, Operand{B.X + c0 + static_cast<long>(c0) * B.ldx, 1, B.ldx},
                      Operand{A12 + c0, lda, 1}, c0 == 0 ? 0.0 : 1.0, B.U + c0, jb, slices, false, 0, nullptr, 0, 0);
      }
      if (!rc)
        rc = check_cuda(h, cudaMemcpy2DAsync(A12, 8ull * lda, B.U, 8ull * jb, 8ull * jb, m2, cudaMemcpyDeviceToDevice,
                                             h->stream), "U12 copy");
      phase_end(h, ph);
      if (rc) return rc;
      ph = phase_begin(h, EMUL_PHASE_UPDATE);
      const double* L21 = A + (j0 + jb) + static_cast<long>(j0) * lda;
      double* A22 = A + (j0 + jb) + static_cast<long>(j0 + jb) * lda;
      rc = gemm_kchunks(h, m2, m2, jb, -1.0, Operand{L21, 1, lda}, Operand{B.U, jb, 1}, 1.0, A22, lda, slices);
      phase_end(h, ph);
      if (rc) return rc;
    }
    if (stats) stats->steps++;
  }
  return EMUL_OK;
}

}  // extern "C"
