// Products with a short inner dimension and few tiles, in one launch: slicing,
// slice-pair products, exact recombination and the update of C (arXiv
// 2509.23565, Section 2, Eq. 1-4; Section 4, Eq. 7) in one block per 128 x 32
// tile of C.
//
// Such a product is bound by latency, not by any unit: two slicing launches
// and a one-tile launch of the persistent kernel took 5 + 5 + 27 us for a 64^3
// product (the persistent kernel drains its level sums through four slots one
// after another, in code unrolled for 32 columns a thread that runs once).
// Here the operands are read once, straight into registers; row maxima,
// digits and the swizzled shared-memory tiles follow without touching global
// memory; every level has an accumulator of its own in tensor memory (s levels
// x 32 columns), so all MMAs are issued back to back and drained together; a
// thread rounds 8 entries.
//
// The digits of A are formed again for each 32 columns of C and those of B for
// each 128 rows, so the kernel is for grids that fit the device at once.
#include <atomic>
#include <cstdint>

#include "emul_internal.h"
#include "launch.h"
#include "ptx.cuh"
#include "round.cuh"
#include "slice.cuh"

namespace emul {
namespace {

constexpr int kSmThreads = 512;
constexpr int kSmBM = 128, kSmBN = 32;     // tile of C
constexpr int kSmHalf = 64;                // K elements staged at a time
constexpr int kSmMaxK = 128;               // s k <= 1040 keeps every level sum exact in FP32 for s <= 8
constexpr uint32_t kSmATile = kSmBM * 64;  // one plane of one 32-wide K chunk: 64-byte rows
constexpr uint32_t kSmBTile = kSmBN * 64;
constexpr int kSmTimeout = -4;             // EMUL_TIMEOUT
constexpr uint32_t kSmTmemCols = 256;      // 8 levels x 32 columns

struct SmallArgs {
  int M, N, K, s;
  const double* A;
  long ars, acs;
  const double* B;
  long brs, bcs;
  double alpha, beta;
  double* C;
  long ldc;
  int* status;
  long long wait_limit;
};

// Eight elements of row r (k from k0 on), zero outside the operand.
__device__ __forceinline__ void load8(const double* X, long rs, long cs, int r, int rows, int k0, int k,
                                      uint64_t (&u)[8]) {
  const uint64_t* p = reinterpret_cast<const uint64_t*>(X) + r * rs + k0 * cs;
#pragma unroll
  for (int j = 0; j < 8; ++j) u[j] = (r < rows && k0 + j < k) ? p[j * cs] : 0ull;
}

// Shared-memory offset of the 16-byte piece `piece` (8 K elements) of row r in a
// tile of 64-byte rows with the 64-byte swizzle.
__device__ __forceinline__ uint32_t swz(int r, int piece) {
  return static_cast<uint32_t>(r * 64 + ((piece ^ ((r >> 1) & 3)) << 4));
}

// Thread layout: slicing A, thread t holds row t & 127 and the K groups of eight
// (t >> 7) + 4 i, i = 0..3; slicing B, one group of one row, rows across lanes
// or groups across lanes by the operand's stride.  After the MMAs warp w holds
// the 32 rows of TMEM quarter w & 3 and columns 8 (w >> 2) .. + 7.
template <int S>
__global__ void __launch_bounds__(kSmThreads, 1) small_product_kernel(const SmallArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ uint32_t part_a[4][kSmBM], part_b[kSmMaxK / 8][kSmBN + 1];
  __shared__ unsigned long long full_a[kSmBM], full_b[kSmBN];
  __shared__ int ea[kSmBM], fb[kSmBN];
  __shared__ __align__(8) uint64_t done;
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.x * kSmBM, n0 = blockIdx.y * kSmBN;
  constexpr int s = S;
  uint8_t* sA = smem;                                       // [s][2 chunks][128 rows x 64 B]
  uint8_t* sB = smem + static_cast<size_t>(s) * 2 * kSmATile;   // [s][2 chunks][32 rows x 64 B]

  if (tid == 0) {
    mbar_init(&done, 1);
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc(&tmem_base, kSmTmemCols);
  grid_wait();
  // operands into registers (all loads in flight together)
  const int ar = tid & 127, ag = tid >> 7;
  const bool b_rows = a.brs == 1;
  const int br = b_rows ? tid & 31 : tid >> 4, bg = b_rows ? tid >> 5 : tid & 15;
  uint64_t ua[4][8], ub[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) load8(a.A, a.ars, a.acs, m0 + ar, a.M, 8 * (ag + 4 * i), a.K, ua[i]);
  load8(a.B, a.brs, a.bcs, n0 + br, a.N, 8 * bg, a.K, ub);

  {
    uint32_t up = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) up = max(up, max_upper8(ua[i]));
    part_a[ag][ar] = up;
    part_b[bg][br] = max_upper8(ub);
  }
  if (tid < kSmBM) full_a[tid] = 0;
  if (tid < kSmBN) full_b[tid] = 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  grid_launch();
  bool full = false;        // an existing row of zeros and subnormals only
  if (tid < kSmBM) {
    uint32_t up = part_a[0][tid];
#pragma unroll
    for (int p = 1; p < 4; ++p) up = max(up, part_a[p][tid]);
    ea[tid] = exponent_of_upper(up);
    full = m0 + tid < a.M && needs_full_max(up);
  } else if (tid < kSmBM + kSmBN) {
    const int r = tid - kSmBM;
    uint32_t up = 0;
#pragma unroll
    for (int p = 0; p < kSmMaxK / 8; ++p) up = max(up, part_b[p][r]);
    fb[r] = exponent_of_upper(up);
    full = n0 + r < a.N && needs_full_max(up);
  }
  if (__syncthreads_or(full)) {
#pragma unroll
    for (int i = 0; i < 4; ++i) atomicMax(&full_a[ar], static_cast<unsigned long long>(max_bits8(ua[i])));
    atomicMax(&full_b[br], static_cast<unsigned long long>(max_bits8(ub)));
    __syncthreads();
    if (tid < kSmBM)
      ea[tid] = exponent_of_maxbits(full_a[tid]);
    else if (tid < kSmBM + kSmBN)
      fb[tid - kSmBM] = exponent_of_maxbits(full_b[tid - kSmBM]);
    __syncthreads();
  }
  const uint32_t tmem = tmem_base;

  bool ok = true;
  uint32_t acc = 0;
#pragma unroll
  for (int h = 0; h < kSmMaxK / kSmHalf; ++h) {
    if (h * kSmHalf >= a.K || !ok) break;                   // uniform over the block
    const int kh = a.K - h * kSmHalf < kSmHalf ? a.K - h * kSmHalf : kSmHalf;
    const int chunks = (kh + 31) / 32;
    // digits of this half's K groups into the tiles of their chunk
#pragma unroll
    for (int i = 2 * h; i < 2 * h + 2; ++i) {
      const int g = ag + 4 * i - 8 * h;                     // group within the half: chunk g / 4, piece g % 4
      if (g >= 4 * chunks) continue;
      uint8_t* base = sA + (g >> 2) * kSmATile + swz(ar, g & 3);
      slice8<S>(ua[i], ea[ar], [&](int p, uint4 w) { *reinterpret_cast<uint4*>(base + p * 2 * kSmATile) = w; });
    }
    {
      const int g = bg - 8 * h;
      if (g >= 0 && g < 4 * chunks) {
        uint8_t* base = sB + (g >> 2) * kSmBTile + swz(br, g & 3);
        slice8<S>(ub, fb[br], [&](int p, uint4 w) { *reinterpret_cast<uint4*>(base + p * 2 * kSmBTile) = w; });
      }
    }
    fence_async_smem();                                     // the MMAs read shared memory through the async proxy
    __syncthreads();
    if (warp == 0) {
      constexpr uint32_t idesc = idesc_bf16_f32(kSmBM, kSmBN);
      const uint32_t tm = __shfl_sync(0xFFFFFFFFu, tmem, 0);
      const uint64_t dA = umma_desc(smem_u32(sA), 64, 4), dB = umma_desc(smem_u32(sB), 64, 4);
      const uint32_t hi = static_cast<uint32_t>(dA >> 32);
      for (int L = s + 1; L >= 2; --L)
        for (int c = 0; c < chunks; ++c)
          for (int p = 1; p < L; ++p)
            mma_bf16_k32_elect<false>(tm + (uint32_t)((L - 2) * kSmBN),
                                      (uint32_t)dA + (uint32_t)((2 * (p - 1) + c) * (int)(kSmATile >> 4)),
                                      (uint32_t)dB + (uint32_t)((2 * (L - p - 1) + c) * (int)(kSmBTile >> 4)), hi,
                                      idesc, acc | (uint32_t)(c | (p - 1)));
      mma_commit_elect(&done);
    }
    acc = 1;
    ok = mbar_wait(&done, (uint32_t)(h & 1), a.wait_limit);
    if (!ok) atomicExch(a.status, kSmTimeout);
    ok = __syncthreads_and(ok) != 0;
  }
  tc_fence_after();

  if (ok) {
    // T = hi 2^28 + lo: the four highest levels (weights 2^0 .. 2^21) in lo, the
    // others in hi; two adjacent levels in one 32-bit word first.  Below 2^22 a
    // level sum becomes an integer by an FP32 add (see gemm_kernel.cuh).
    const int quarter = warp & 3, cg = warp >> 2;
    const uint32_t ta = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + (uint32_t)(cg * 8);
    long long lo[8], hi[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) lo[c] = hi[c] = 0;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      // four levels' loads in flight together
      uint32_t r[4][8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int L = s + 1 - 4 * q - i;
        if (L >= 2) tmem_ld8(ta + (uint32_t)((L - 2) * kSmBN), r[i]);
      }
      tmem_ld_wait();
      float mx = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (s + 1 - 4 * q - i >= 2) {
#pragma unroll
          for (int c = 0; c < 8; ++c) mx = fmaxf(mx, fabsf(__uint_as_float(r[i][c])));
        }
      const bool quick = mx < 4194304.0f;
#pragma unroll
      for (int i = 0; i < 4; i += 2) {
        if (s + 1 - 4 * q - i < 2) continue;
        const bool two = s + 1 - 4 * q - i - 1 >= 2;
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          long long v;
          if (quick) {
            int w = __float_as_int(__uint_as_float(r[i][c]) + 12582912.0f) - 0x4B400000;
            if (two) w += (__float_as_int(__uint_as_float(r[two ? i + 1 : i][c]) + 12582912.0f) - 0x4B400000) * 128;
            v = w;
          } else {
            v = __float2int_rn(__uint_as_float(r[i][c]));
            if (two) v += (long long)__float2int_rn(__uint_as_float(r[two ? i + 1 : i][c])) * 128;
          }
          if (q == 0)
            lo[c] += v << (7 * i);
          else
            hi[c] += v << (7 * i);
        }
      }
    }
    const int row = m0 + quarter * 32 + lane;
    if (row < a.M) {
      const int e = ea[quarter * 32 + lane];
      const bool sub = a.alpha == -1.0 && a.beta == 1.0, set = a.alpha == 1.0 && a.beta == 0.0;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int col = n0 + cg * 8 + c;
        if (col >= a.N) break;
        const int f = fb[cg * 8 + c];
        double D;
        const int sh0 = -7 * (s + 1);
        if (e == kNonFinite || f == kNonFinite) {
          D = __longlong_as_double(0x7FF8000000000000ll);
        } else {
          const int sh = e + f + sh0;
          if (sh < -1022 || sh > 944) {
            D = rn_scaled(((__int128)hi[c] << 28) + (__int128)lo[c], sh);
          } else if (S <= 6 || (S == 7 && a.K <= 64)) {   // |T| < 1.02 2^(14 + 35) k, 2^(14 + 42) k: 64 bits hold it
            D = rn_x64((hi[c] << 28) + lo[c], sh);
          } else {
            D = rn_x80((hi[c] << 12) + (lo[c] >> 16), (uint32_t)lo[c] & 0xFFFFu, sh);
          }
        }
        double* cp = a.C + row + static_cast<long>(col) * a.ldc;
        if (sub)
          red_add_f64(cp, neg_d(D));
        else if (set)
          *cp = D;
        else
          *cp = a.beta == 0.0 ? __dmul_rn(a.alpha, D)
                              : __dadd_rn(__dmul_rn(a.alpha, D), __dmul_rn(a.beta, *cp));
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kSmTmemCols);
  }
}

}  // namespace

// Whether the one-launch product takes this shape: K and the level sums within
// its limits, and one block per SM at most.  Both sides of the line in us (this
// kernel / slicing kernel and persistent kernel, s = 7): 64^3 11.9 / 21.3, 128^3
// 18.6 / 26.6, 4000 x 64 x 64 12.4 / 16.1, 600 x 960 x 64 (150 tiles) 12.6 / 18.3;
// with a second block on some SMs 1000 x 1000 x 64 24.3 / 19.0, 8192 x 128 x 128
// 37.3 / 23.2 (at s = 3 17.4 / 16.5 and 24.0 / 17.2).
bool small_product_fits(int m, int n, int k, int s, int nsm) {
  const long tiles = static_cast<long>((m + kSmBM - 1) / kSmBM) * ((n + kSmBN - 1) / kSmBN);
  return k >= 1 && k <= kSmMaxK && s * k <= kExactBudget && s <= kMaxSlices && tiles <= nsm;
}

template <int S>
cudaError_t launch_small_s(cudaStream_t st, const SmallArgs& a) {
  constexpr int smem = S * 2 * static_cast<int>(kSmATile + kSmBTile) + 1024;
  static std::atomic<bool> ready[64];      // the limit is raised once per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !ready[dev].load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(small_product_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    if (dev < 64) ready[dev].store(true, std::memory_order_release);
  }
  const dim3 grid((a.M + kSmBM - 1) / kSmBM, (a.N + kSmBN - 1) / kSmBN);
  return launch_dependent(small_product_kernel<S>, grid, kSmThreads, smem, st, a);
}

cudaError_t launch_small_product(cudaStream_t st, int m, int n, int k, double alpha, const double* A, long ars,
                                 long acs, const double* B, long brs, long bcs, double beta, double* C, long ldc,
                                 int s, int* status, long long wait_limit) {
  const SmallArgs a{m, n, k, s, A, ars, acs, B, brs, bcs, alpha, beta, C, ldc, status, wait_limit};
  switch (s) {
    case 1: return launch_small_s<1>(st, a);
    case 2: return launch_small_s<2>(st, a);
    case 3: return launch_small_s<3>(st, a);
    case 4: return launch_small_s<4>(st, a);
    case 5: return launch_small_s<5>(st, a);
    case 6: return launch_small_s<6>(st, a);
    case 7: return launch_small_s<7>(st, a);
    case 8: return launch_small_s<8>(st, a);
  }
  return cudaErrorInvalidValue;
}

}  // namespace emul
