// Blocked LU with partial pivoting and blocked Cholesky whose third-order work
// runs through the emulated product (arXiv 2509.23565, Section 4, Eq. 5-7),
// the triangular solves that use the factors, and the residual of Eq. 8.
//
// LU step (right-looking, block nb):
//   1. panel [A11; A21] factored with partial pivoting: recursive halving; the
//      inner Schur updates use the emulated product, the leaves (<= 32 columns)
//      run an FP64 kernel over many blocks (pivot search on the IEEE bit
//      patterns, one bounded exchange per column: through a cluster's shared
//      memory, or through L2 above 2048 rows);
//   2. the panel's row interchanges applied to the columns left and right of it;
//   3. U12 = L11^-1 A12: L11^-1 formed in FP64 (unit lower, nb x nb), the
//      product by the emulated GEMM;
//   4. A22 <- A22 - L21 U12 by the emulated GEMM (alpha = -1, beta = 1).
// Cholesky step (lower): FP64 diagonal block, L21 = A21 L11^-T through an FP64
// L11^-1 and the emulated GEMM, then A22 <- A22 - L21 L21^T on lower tiles only,
// with one slice set serving both operands; the next diagonal block is factored
// beside the update where that is long enough.
#include <cmath>
#include <cstdio>
#include <map>
#include <mutex>
#include <set>
#include <utility>

#include <cuda_runtime.h>

#include "handle.h"
#include "launch.h"
#include "ptx.cuh"

namespace emul {

namespace {

constexpr int kLeaf = 32;           // widest panel handled by the leaf kernel
constexpr int kLeafThreads = 256;
constexpr int kStatusTimeout = -4;
constexpr size_t kAl = 256;
inline size_t al(size_t x) { return (x + kAl - 1) / kAl * kAl; }

// Pivot exchange of the leaf: every block publishes its candidate as 8-byte
// words {32-bit payload, 32-bit epoch}; an aligned 64-bit store is
// single-copy atomic, so a reader that sees the epoch of the current column in
// a word also sees that word's payload, and no fence or counter is needed.
// Record of block b for column parity par: words [0, 4) = |value| low and high
// halves, candidate row, unused; words [4, 4 + 2w) = the candidate row, each
// double as its low and high halves; words [4 + 2 kLeaf, 6 + 2 kLeaf) = the
// reciprocal of the candidate.  Epoch = salt * 32 + column (salt > 0,
// distinct per leaf launch, records cleared before a factorization).
constexpr int kRecWords = 4 + 2 * kLeaf + 2;

__device__ __forceinline__ void put_word(uint64_t* p, uint32_t payload, uint32_t epoch) {
  *reinterpret_cast<volatile uint64_t*>(p) = (static_cast<uint64_t>(epoch) << 32) | payload;
}
// Two adjacent words (16-byte aligned) in one load; each stays single-copy atomic.
__device__ __forceinline__ void get_pair(const uint64_t* p, uint64_t& a, uint64_t& b) {
  asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
}
__device__ __forceinline__ bool has_epoch(uint64_t v, uint32_t epoch) { return static_cast<uint32_t>(v >> 32) == epoch; }
// Poll a pair of words until both carry `epoch` (bounded); the double they
// hold (low half first) is returned in x.  False on timeout.
__device__ __forceinline__ bool wait_pair(const uint64_t* p, uint32_t epoch, double& x, long long limit) {
  uint64_t a, b;
  get_pair(p, a, b);
  if (!(has_epoch(a, epoch) && has_epoch(b, epoch))) {
    const long long t0 = clock64();
    do {
      if (clock64() - t0 > limit) return false;
      get_pair(p, a, b);
    } while (!(has_epoch(a, epoch) && has_epoch(b, epoch)));
  }
  x = __longlong_as_double(static_cast<long long>((b << 32) | (a & 0xFFFFFFFFull)));
  return true;
}
constexpr int kMaxRecPerLane = 8;   // records polled by one lane: the leaf runs at most 256 blocks

__device__ __forceinline__ uint64_t absbits(double x) {
  return static_cast<uint64_t>(__double_as_longlong(x)) & 0x7FFFFFFFFFFFFFFFull;
}

// (value, row) pair ordering of the pivot search: larger |value| wins, ties
// go to the smaller row (the first maximal index, as LAPACK's idamax).
__device__ __forceinline__ bool better(uint64_t v1, int r1, uint64_t v2, int r2) {
  return v1 > v2 || (v1 == v2 && r1 < r2);
}

// The best of a warp's (value, row) pairs (better() above), in every lane, by
// three warp reductions on 32-bit words.
__device__ __forceinline__ void warp_best(uint64_t& v, int& r) {
  const uint32_t hi = static_cast<uint32_t>(v >> 32), mh = __reduce_max_sync(0xFFFFFFFFu, hi);
  const uint32_t lo = hi == mh ? static_cast<uint32_t>(v) : 0u, ml = __reduce_max_sync(0xFFFFFFFFu, lo);
  const bool top = hi == mh && static_cast<uint32_t>(v) == ml;
  r = __reduce_min_sync(0xFFFFFFFFu, top ? r : 0x7FFFFFFF);
  v = (static_cast<uint64_t>(mh) << 32) | ml;
}

// row[cc ld] -= l pv[cc] for cc = c0, c0 + step, ... < w, four at a time so that
// their loads do not wait for the stores before them.
__device__ __forceinline__ void rank1_row(double* row, int ld, double l, const double* pv, int c0, int w, int step) {
  int cc = c0;
  for (; cc + 3 * step < w; cc += 4 * step) {
    double v[4], u[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = row[(cc + q * step) * ld];
      u[q] = pv[cc + q * step];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) row[(cc + q * step) * ld] = fma(-l, u[q], v[q]);
  }
  for (; cc < w; cc += step) row[cc * ld] = fma(-l, pv[cc], row[cc * ld]);
}

// A column outside the leaf that follows its interchanges in global memory.  One
// thread owns it for the whole launch, so successive interchanges of one element
// stay in program order; the stores of an interchange are put off to the next
// one, when its loads have long arrived.
struct OutsideColumn {
  double* col;
  long r0 = -1, r1 = -1;
  double x0 = 0.0, x1 = 0.0;
  __device__ __forceinline__ void flush() {
    if (col && r0 >= 0) {
      col[r0] = x1;
      col[r1] = x0;
      r0 = -1;
    }
  }
  __device__ __forceinline__ void swap(long a, long b) {
    if (!col) return;
    flush();
    r0 = a;
    r1 = b;
    x0 = col[a];
    x1 = col[b];
  }
};

// Leaf panel: rows d0..n-1, columns d0..d0+w-1 of A, factored in place with
// partial pivoting.  Block b keeps panel rows [b*R, b*R+R) in shared memory.
//
// Column c: (1) pivot search on column c over the block's rows, (2) the
// block's candidate (|value|, row, the row itself) and, from the block owning
// it, row c published as epoch-tagged words, (3) warp 0 collects the G
// candidates and fetches the winner's row, the last warp fetches row c, while
// warps 1-6 apply the rank-1 update of pivot c-1 to columns c+1..w-1,
// (4) row interchange, (5) multipliers of column c and the update of column
// c+1 only, so that the next pivot search can start.  Each entry receives the
// same FMAs in the same order as in a plain right-looking elimination; the
// published rows get the deferred update of pivot c-1 applied on the fly (the
// same FMA).  The exchange needs no grid barrier: a block cannot publish
// column c+2 into the slot of column c before every block has published
// column c+1, which each does only after reading column c.
//
// Every interchange is also applied to the columns [pc0, d0) and [d0+w, pc1) of
// the enclosing panel, which live in global memory: the outside column q
// (0-based over both ranges) belongs to one thread of block q % G for the whole
// launch, so successive interchanges of one element stay in program order: to the
// (q / G)-th of the block's 256 threads, counted from warp 1 to warp 6 first, then
// warps 0 and 7, which run the exchange and interchange after it.  A column's loads
// are issued when the pivot is known, its stores when the next pivot is known, off
// the critical path.  At most 248 outside columns exist (panel <= 256 wide, leaf
// >= 8 wide).  The candidate's value and row are published by the first lane of
// warp 7, its reciprocal by the first lane of warp 6.
__global__ void __launch_bounds__(kLeafThreads) getf2_leaf_kernel(double* A, long lda, int n, int d0, int w, int R,
                                                                 int pc0, int pc1, int32_t* ipiv, int32_t* info,
                                                                 uint64_t* recs, uint64_t* drec, uint32_t salt,
                                                                 int* status, long long limit) {
  extern __shared__ double P[];   // P[c*ld + lr], ld odd: rows are read and written across banks
  const int ld = R | 1;
  __shared__ double prow[2][kLeaf], crow[kLeaf];
  __shared__ double rcp_s;
  __shared__ uint64_t red_v[kLeafThreads / 32];
  __shared__ int red_r[kLeafThreads / 32];
  __shared__ int win_s, ok_s, ok7_s;
  constexpr int kRowTid = kLeafThreads - 32;   // first lane of the last warp: publisher, row-c reader
  constexpr int kRcpTid = kLeafThreads - 64;   // first lane of warp 6: the candidate's reciprocal
  const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int mp = n - d0;
  const int r0 = b * R;
  const int rcount = mp - r0 < R ? (mp - r0 > 0 ? mp - r0 : 0) : R;
  const int nleft = d0 - pc0;
  const int nout = nleft + (pc1 - d0 - w);
  // outside columns go to the threads of warps 1-6 first: warps 0 and 7 run the exchange
  const int ot = tid >= 32 && tid < kRowTid ? tid - 32 : (tid < 32 ? kLeafThreads - 64 + tid : tid);
  const int q = ot * G + b;
  OutsideColumn out{q < nout ? A + static_cast<long>(q < nleft ? pc0 + q : d0 + w + (q - nleft)) * lda : nullptr};
  int p_last = -1;             // pivot row of column c-1
  bool pend = false;           // pivot c-1 was nonzero: its update of columns > c is pending
  // stage the rows: 16 loads in flight per thread before their stores
  for (int lr = tid; lr < rcount; lr += blockDim.x) {
    const double* src = A + (d0 + r0 + lr) + static_cast<long>(d0) * lda;
    for (int c0 = 0; c0 < w; c0 += 16) {
      double v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = c0 + j < w ? src[static_cast<long>(c0 + j) * lda] : 0.0;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (c0 + j < w) P[(c0 + j) * ld + lr] = v[j];
    }
  }
  __syncthreads();

  for (int c = 0; c < w; ++c) {
    const int par = c & 1;
    const uint32_t ep = (salt << 5) | static_cast<uint32_t>(c);
    const double* pv = prow[par ^ 1];   // pivot row of column c-1
    uint64_t* rec_all = recs + static_cast<long>(par) * G * kRecWords;
    uint64_t* my = rec_all + static_cast<long>(b) * kRecWords;
    uint64_t* drow = drec + par * 2 * kLeaf;
    // (1) local candidate for column c over own rows with panel row >= c
    uint64_t bv = 0;
    int br = 0x7FFFFFFF;
    for (int lr = tid; lr < rcount; lr += blockDim.x) {
      const int pr = r0 + lr;
      if (pr < c) continue;
      const uint64_t v = absbits(P[c * ld + lr]);
      if (better(v, pr, bv, br)) {
        bv = v;
        br = pr;
      }
    }
    warp_best(bv, br);
    if (lane == 0) {
      red_v[warp] = bv;
      red_r[warp] = br;
    }
    __syncthreads();
    bv = red_v[lane & (kLeafThreads / 32 - 1)];
    br = red_r[lane & (kLeafThreads / 32 - 1)];
    warp_best(bv, br);
    if (tid == kRowTid) {
      put_word(my + 0, static_cast<uint32_t>(bv), ep);
      put_word(my + 1, static_cast<uint32_t>(bv >> 32), ep);
      put_word(my + 2, static_cast<uint32_t>(br), ep);
    }
    // (2) publish the candidate row and row c, current through pivot c-1
    {
      const int pr = br;
      if (tid < 2 * w) {
        const int cc = tid >> 1;
        if (pr != 0x7FFFFFFF) {
          const int lr = pr - r0;
          double v = P[cc * ld + lr];
          if (pend && cc > c) v = fma(-P[(c - 1) * ld + lr], pv[cc], v);
          const uint64_t bits = static_cast<uint64_t>(__double_as_longlong(v));
          put_word(my + 4 + tid, static_cast<uint32_t>(tid & 1 ? bits >> 32 : bits), ep);
        }
        if (c >= r0 && c < r0 + rcount) {
          const int lr = c - r0;
          double v = P[cc * ld + lr];
          if (pend && cc > c) v = fma(-P[(c - 1) * ld + lr], pv[cc], v);
          const uint64_t bits = static_cast<uint64_t>(__double_as_longlong(v));
          put_word(drow + tid, static_cast<uint32_t>(tid & 1 ? bits >> 32 : bits), ep);
        }
      }
    }
    __syncthreads();
    // (3) exchange (warp 0: candidates and pivot row; last warp: row c) while
    // warps 1-6 apply the deferred update of pivot c-1
    if (warp == 0) {
      // every lane loads all of its records at once, then re-polls the late ones
      uint64_t w0[kMaxRecPerLane], w1[kMaxRecPerLane], w2[kMaxRecPerLane];
      unsigned pending = 0;
#pragma unroll
      for (int k = 0; k < kMaxRecPerLane; ++k)
        if (lane + 32 * k < G) pending |= 1u << k;
      bool ok = true;
      const long long t0 = clock64();
      while (true) {
#pragma unroll
        for (int k = 0; k < kMaxRecPerLane; ++k)
          if (pending >> k & 1u) {
            const uint64_t* r = rec_all + static_cast<long>(lane + 32 * k) * kRecWords;
            uint64_t unused;
            get_pair(r, w0[k], w1[k]);
            get_pair(r + 2, w2[k], unused);
          }
#pragma unroll
        for (int k = 0; k < kMaxRecPerLane; ++k)
          if ((pending >> k & 1u) && has_epoch(w0[k], ep) && has_epoch(w1[k], ep) && has_epoch(w2[k], ep))
            pending &= ~(1u << k);
        if (__all_sync(0xFFFFFFFFu, pending == 0)) break;
        if (__any_sync(0xFFFFFFFFu, clock64() - t0 > limit)) {
          ok = false;
          break;
        }
      }
      uint64_t gv = 0;
      int gr = 0x7FFFFFFF, gbk = 0;
#pragma unroll
      for (int k = 0; k < kMaxRecPerLane; ++k) {
        if (lane + 32 * k >= G) continue;
        const uint64_t v = ((w1[k] & 0xFFFFFFFFull) << 32) | (w0[k] & 0xFFFFFFFFull);
        const int rr = static_cast<int>(static_cast<uint32_t>(w2[k]));
        if (better(v, rr, gv, gr)) {
          gv = v;
          gr = rr;
          gbk = lane + 32 * k;
        }
      }
      {
        const uint64_t own_v = gv;
        const int own_r = gr;
        warp_best(gv, gr);
        const int src = __ffs(__ballot_sync(0xFFFFFFFFu, own_v == gv && own_r == gr)) - 1;
        gbk = __shfl_sync(0xFFFFFFFFu, gbk, src);
      }
      // the winner's row and, in flight with it, the reciprocal
      const uint64_t* rp = rec_all + static_cast<long>(gbk) * kRecWords + 4 + 2 * kLeaf;
      uint64_t ra = 0, rb = 0;
      if (ok && lane == 0) get_pair(rp, ra, rb);
      if (ok && lane < w) {
        double pvv = 0.0;
        ok = wait_pair(rec_all + static_cast<long>(gbk) * kRecWords + 4 + 2 * lane, ep, pvv, limit);
        prow[par][lane] = pvv;
      }
      if (ok && lane == 0) {
        double r = __longlong_as_double(static_cast<long long>((rb << 32) | (ra & 0xFFFFFFFFull)));
        if (!(has_epoch(ra, ep) && has_epoch(rb, ep))) ok = wait_pair(rp, ep, r, limit);
        rcp_s = r;
      }
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (lane == 0) {
        win_s = gr;
        ok_s = ok;
        if (!ok) atomicExch(status, kStatusTimeout);
        if (ok && b == 0) {
          ipiv[d0 + c] = d0 + gr + 1;
          if (gv == 0) atomicCAS(info, 0, d0 + c + 1);
        }
      }
    } else if (warp == kLeafThreads / 32 - 1) {
      bool ok = true;
      if (lane < w) {
        double x = 0.0;
        ok = wait_pair(drow + 2 * lane, ep, x, limit);
        crow[lane] = x;
      }
      ok = __all_sync(0xFFFFFFFFu, ok);
      if (lane == 0) {
        ok7_s = ok;
        if (!ok) atomicExch(status, kStatusTimeout);
      }
    } else {
      if (tid == kRcpTid) {
        // the block's candidate is the pivot of the whole panel for one block:
        // its reciprocal is ready when the winner is known
        const double r = br != 0x7FFFFFFF ? 1.0 / P[c * ld + (br - r0)] : 0.0;
        const uint64_t bits = static_cast<uint64_t>(__double_as_longlong(r));
        put_word(my + 4 + 2 * kLeaf, static_cast<uint32_t>(bits), ep);
        put_word(my + 5 + 2 * kLeaf, static_cast<uint32_t>(bits >> 32), ep);
      }
      if (c > 0 && p_last != c - 1) out.swap(d0 + c - 1, d0 + p_last);
      if (pend && c + 1 < w) {
        // eight shares of the columns, two for each sub-partition's FP64 unit:
        // warps 3 and 4, alone beside warps 7 and 0 of the exchange, take two each
        const int s0 = warp == 3 ? 4 : (warp == 4 ? 6 : (warp < 3 ? warp - 1 : warp - 3));
        const int s1 = warp == 3 || warp == 4 ? s0 + 2 : s0 + 1;
        for (int lr = lane; lr < rcount; lr += 32) {
          if (r0 + lr <= c - 1) continue;
          const double l = P[(c - 1) * ld + lr];
          for (int s = s0; s < s1; ++s) rank1_row(P + lr, ld, l, pv, c + 1 + s, w, 8);
        }
      }
    }
    if ((warp == 0 || warp == kLeafThreads / 32 - 1) && c > 0 && p_last != c - 1) out.swap(d0 + c - 1, d0 + p_last);
    __syncthreads();
    if (!ok_s || !ok7_s) return;
    const int p = win_s;
    p_last = p;
    const double piv = prow[par][c];
    pend = absbits(piv) != 0;           // (an FP64 comparison takes 64 cycles)
    if (pend) {
      // (4) interchange rows c and p (both current through pivot c-1); columns
      // c and c+1 of row p are left to the thread that has row p in (5)
      if (p != c) {
        if (c >= r0 && c < r0 + rcount)
          for (int cc = tid; cc < w; cc += blockDim.x) P[cc * ld + (c - r0)] = prow[par][cc];
        if (p >= r0 && p < r0 + rcount)
          for (int cc = tid; cc < w; cc += blockDim.x)
            if (cc != c && cc != c + 1) P[cc * ld + (p - r0)] = crow[cc];
      }
      // (5) multipliers of column c, update of column c+1
      const bool use_rcp = absbits(piv) >= 0x0010000000000000ull;
      const double rcp = rcp_s;
      const double u1 = c + 1 < w ? prow[par][c + 1] : 0.0;
      for (int lr = tid; lr < rcount; lr += blockDim.x) {
        if (r0 + lr <= c) continue;
        const bool swapped = r0 + lr == p;             // (p > c here)
        const double a0 = swapped ? crow[c] : P[c * ld + lr];
        const double l = use_rcp ? a0 * rcp : a0 / piv;
        P[c * ld + lr] = l;
        if (c + 1 < w) P[(c + 1) * ld + lr] = fma(-l, u1, swapped ? crow[c + 1] : P[(c + 1) * ld + lr]);
      }
    }
    __syncthreads();
  }
  if (p_last != w - 1 && p_last >= 0) out.swap(d0 + w - 1, d0 + p_last);
  out.flush();
  for (int c = 0; c < w; ++c)
    for (int lr = tid; lr < rcount; lr += blockDim.x) A[(d0 + r0 + lr) + static_cast<long>(d0 + c) * lda] = P[c * ld + lr];
}

// The same leaf on one thread-block cluster, for panels of at most
// kClusterRows rows: the exchange of a column goes through distributed shared
// memory instead of L2.  Each CTA stores its candidate (|value|, row) and the
// candidate's row into every CTA of the cluster with st.async, which counts the
// bytes on the receiver's barrier, so one trip of a few hundred cycles replaces
// three through L2 (records out, records in, the winner's row), and the pivot
// row is at hand once the winner is known.  Row c is sent along by its owner.
// A column then costs one search, one exchange, one division and the rank-1
// update of R = ceil(rows / CTAs) rows, bound by FP64 (1.68 FMA per clock per
// SM; a warp's DFMA occupies its sub-partition for 64-76 cycles), so the rows
// are spread over up to 16 SMs.  The arithmetic is that of getf2_leaf_kernel,
// operation for operation.
//
// A leaf of 32 columns takes 58 us (26 with few rows, 69 with 2048), the same
// leaf through L2 93 to 102 at any height.  128 rows per CTA at most: with 256 the
// rank-1 update of a column (2400 cycles of FP64 on average) would no longer hide
// behind the exchange.
//
// Buffers are double-buffered by column parity: a CTA sends column c + 2 only
// after it has received column c + 1 from every CTA, which each sends after it
// has used column c.
constexpr int kClusterMax = 16;
constexpr int kClusterR = 128;                        // rows per CTA at most
constexpr int kClusterRows = kClusterMax * kClusterR;
constexpr int kPushWarps = 4;
__global__ void __launch_bounds__(kLeafThreads) getf2_cluster_kernel(double* A, long lda, int n, int d0, int w, int R,
                                                                    int pc0, int pc1, int32_t* ipiv, int32_t* info,
                                                                    int* status, long long limit) {
  extern __shared__ double P[];   // P[c*ld + lr], ld odd: rows are read and written across banks
  const int ld = R | 1;
  __shared__ double crow[2][kClusterMax][kLeaf], drow[2][kLeaf], prow[2][kLeaf];
  __shared__ uint64_t rec[2][kClusterMax][2];
  __shared__ double rcps[2][kClusterMax];
  __shared__ __align__(8) uint64_t full[2];
  __shared__ double rcp_s;
  __shared__ uint64_t red_v[kClusterR / 32];
  __shared__ int red_r[kClusterR / 32];
  __shared__ int win_s, ok_s;
  const int G = static_cast<int>(cluster_size()), b = static_cast<int>(cluster_rank());
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kWarps = kLeafThreads / 32;
  const int mp = n - d0;
  const int r0 = b * R;
  const int rcount = mp - r0 < R ? (mp - r0 > 0 ? mp - r0 : 0) : R;
  const int nleft = d0 - pc0;
  const int nout = nleft + (pc1 - d0 - w);
  const int q = (tid - 32) * G + b;      // outside column of this thread (as in getf2_leaf_kernel); none in warp 0
  double* ocol = tid >= 32 && q < nout ? A + static_cast<long>(q < nleft ? pc0 + q : d0 + w + (q - nleft)) * lda : nullptr;
  OutsideColumn out{ocol};
  int p_last = -1;                // pivot row of column c-1
  bool pend = false;
  // deferred updates: warps 1..7 share the row groups of 32, and the columns of each
  const int rgroups = (R + 31) / 32;
  const int cstep = (kWarps - 1) / rgroups;
  const int dgrp = warp >= 1 ? (warp - 1) % rgroups : 0, doff = warp >= 1 ? (warp - 1) / rgroups : cstep;
  const int dlr = dgrp * 32 + lane;
  if (tid < 2) mbar_init(&full[tid], 1);
  if (tid == 0) fence_mbar_init();
  grid_launch();
  grid_wait();
  for (int lr = tid & (kClusterR - 1), half = tid / kClusterR; lr < rcount; lr += kClusterR) {
    // 16 columns per half of the block, their loads in flight together
    const double* src = A + (d0 + r0 + lr) + static_cast<long>(d0) * lda;
    double v[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = half * 16 + j < w ? src[static_cast<long>(half * 16 + j) * lda] : 0.0;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (half * 16 + j < w) P[(half * 16 + j) * ld + lr] = v[j];
  }
  __syncthreads();
  cluster_sync();               // every CTA's barriers are initialised

  for (int c = 0; c < w; ++c) {
    const int par = c & 1;
    const double* pv = prow[par ^ 1];   // pivot row of column c-1
    if (tid == 0) mbar_arrive_expect_tx(&full[par], static_cast<uint32_t>(G * (24 + 8 * w) + 8 * w));
    // (1) candidate of the own rows: largest |value|, then the smallest row
    if (warp < kClusterR / 32) {
      const int pr = r0 + tid;
      const bool in = tid < rcount && pr >= c;
      uint64_t v = in ? absbits(P[c * ld + tid]) : 0ull;
      int r = in ? pr : 0x7FFFFFFF;
      warp_best(v, r);
      if (lane == 0) {
        red_v[warp] = v;
        red_r[warp] = r;
      }
    }
    __syncthreads();
    uint64_t bv = red_v[lane & (kClusterR / 32 - 1)];
    int br = red_r[lane & (kClusterR / 32 - 1)];
    warp_best(bv, br);
    // (2) candidate, its row and row c (current through pivot c-1) to every CTA
    // from warps 0-3, one per sub-partition; the candidate's reciprocal, whose
    // division takes as long as the exchange, follows from warp 4
    if (warp < kPushWarps) {
      const bool own_c = c >= r0 && c < r0 + rcount;
      double v = 0.0, dv = 0.0;
      if (lane < w) {
        if (br != 0x7FFFFFFF) {
          v = P[lane * ld + (br - r0)];
          if (pend && lane > c) v = fma(-P[(c - 1) * ld + (br - r0)], pv[lane], v);
        }
        if (own_c) {
          dv = P[lane * ld + (c - r0)];
          if (pend && lane > c) dv = fma(-P[(c - 1) * ld + (c - r0)], pv[lane], dv);
        }
      }
      for (int t = warp; t < G; t += kPushWarps) {
        const uint32_t bar = mapa_addr(smem_u32(&full[par]), t);
        const uint32_t to = bar - smem_u32(&full[par]);   // from an address here to the same one in CTA t
        if (lane < w) {
          st_async_b64(to + smem_u32(&crow[par][b][lane]), static_cast<uint64_t>(__double_as_longlong(v)), bar);
          if (own_c) st_async_b64(to + smem_u32(&drow[par][lane]), static_cast<uint64_t>(__double_as_longlong(dv)), bar);
        }
        if (lane < 2) st_async_b64(to + smem_u32(&rec[par][b][lane]), lane == 0 ? bv : static_cast<uint64_t>(br), bar);
      }
    } else if (warp == kPushWarps) {
      const double r = br != 0x7FFFFFFF ? 1.0 / P[c * ld + (br - r0)] : 0.0;
      if (lane < G) {
        const uint32_t bar = mapa_addr(smem_u32(&full[par]), lane);
        st_async_b64(bar - smem_u32(&full[par]) + smem_u32(&rcps[par][b]),
                     static_cast<uint64_t>(__double_as_longlong(r)), bar);
      }
    }
    __syncthreads();
    // (3) winner, its row and the reciprocal (warp 0); deferred update of pivot c-1
    if (warp == 0) {
      const bool ok = __all_sync(0xFFFFFFFFu, mbar_wait_cluster(&full[par], (c >> 1) & 1, limit));
      const uint64_t own_v = lane < G ? rec[par][lane][0] : 0ull;
      const int own_r = lane < G ? static_cast<int>(rec[par][lane][1]) : 0x7FFFFFFF;
      uint64_t gv = own_v;
      int gr = own_r;
      warp_best(gv, gr);
      const int src = __ffs(__ballot_sync(0xFFFFFFFFu, own_v == gv && own_r == gr)) - 1;
      if (lane < w) {
        const double x = crow[par][src][lane];
        prow[par][lane] = x;
      }
      if (lane == 0) {
        rcp_s = rcps[par][src];
        win_s = gr;
        ok_s = ok;
        if (!ok) atomicExch(status, kStatusTimeout);
        if (ok && b == 0) {
          ipiv[d0 + c] = d0 + gr + 1;
          if (gv == 0) atomicCAS(info, 0, d0 + c + 1);
        }
      }
    } else {
      if (c > 0 && p_last != c - 1) out.swap(d0 + c - 1, d0 + p_last);
      if (pend && doff < cstep && dlr < rcount && r0 + dlr > c - 1) {
        rank1_row(P + dlr, ld, P[(c - 1) * ld + dlr], pv, c + 1 + doff, w, cstep);
      }
    }
    __syncthreads();
    if (!ok_s) break;
    const int p = win_s;
    p_last = p;
    const double piv = prow[par][c];
    pend = absbits(piv) != 0;           // (an FP64 comparison takes 64 cycles)
    if (pend) {
      // (4) interchange rows c and p (both current through pivot c-1); columns
      // c and c+1 of row p are left to the thread that has row p in (5)
      if (p != c) {
        if (tid < w && c >= r0 && c < r0 + rcount) P[tid * ld + (c - r0)] = prow[par][tid];
        if (tid < w && tid != c && tid != c + 1 && p >= r0 && p < r0 + rcount) P[tid * ld + (p - r0)] = drow[par][tid];
      }
      // (5) multipliers of column c, update of column c+1
      if (tid < rcount && r0 + tid > c) {
        const bool swapped = r0 + tid == p;            // (p > c here)
        const double a0 = swapped ? drow[par][c] : P[c * ld + tid];
        const double l = absbits(piv) >= 0x0010000000000000ull ? a0 * rcp_s : a0 / piv;
        P[c * ld + tid] = l;
        if (c + 1 < w)
          P[(c + 1) * ld + tid] = fma(-l, prow[par][c + 1], swapped ? drow[par][c + 1] : P[(c + 1) * ld + tid]);
      }
    }
  }
  if (p_last != w - 1 && p_last >= 0) out.swap(d0 + w - 1, d0 + p_last);
  out.flush();
  __syncthreads();
  for (int e = tid; e < w * kClusterR; e += blockDim.x) {
    const int lr = e & (kClusterR - 1), c = e / kClusterR;
    if (lr < rcount) A[(d0 + r0 + lr) + static_cast<long>(d0 + c) * lda] = P[c * ld + lr];
  }
  cluster_sync();               // no CTA leaves while another may still store into it
}

// Row interchanges ipiv[k1..k2) (1-based global rows, ipiv[k]-1 >= k) resolved
// into a gather map: after the interchanges, row dst[i] holds the original row
// src[i], for the *count affected rows (at most 2 (k2-k1)).  The rows are
// numbered 0..nb-1 for the block's own and kPermMax + i for the row outside it
// that interchange i names first; the interchanges are taken in eight groups, each
// applied in order by one thread to an identity map of its own, and a row's source
// is found by following it through the groups' maps.  (One row after another
// through all 256 interchanges took 15 us, on the critical path of every panel.)
// The map's order is immaterial to its users.
constexpr int kPermMax = 256;          // interchanges per gather map (longer ranges: several maps)
constexpr int kPermGroups = 8;
struct PermShared {
  int piv[kPermMax];                               // global rows, 0-based
  unsigned short id[kPermMax];                     // number of the row interchange i names
  int key[4 * kPermMax], first[4 * kPermMax];      // rows outside the block: first interchange naming them
  unsigned short map[kPermGroups][2 * kPermMax];
  int dst[2 * kPermMax], src[2 * kPermMax], cnt;
};
// Called by all kPermMax threads of a block, S.piv[0..nb) set and visible.
__device__ void perm_map(PermShared& S, int k1, int nb) {
  const int i = threadIdx.x;
  if (i == 0) S.cnt = 0;
  for (int e = i; e < kPermGroups * 2 * kPermMax; e += kPermMax) S.map[0][e] = static_cast<unsigned short>(e & (2 * kPermMax - 1));
  for (int e = i; e < 4 * kPermMax; e += kPermMax) {
    S.key[e] = -1;
    S.first[e] = kPermMax;
  }
  __syncthreads();
  const int p = i < nb ? S.piv[i] : 0;
  const bool outside = i < nb && (p < k1 || p >= k1 + nb);
  int slot = 0;
  if (outside) {
    // open addressing, at most kPermMax of 4 kPermMax slots taken
    slot = p & (4 * kPermMax - 1);
    while (true) {
      const int was = atomicCAS(&S.key[slot], -1, p);
      if (was == -1 || was == p) break;
      slot = (slot + 1) & (4 * kPermMax - 1);
    }
    atomicMin(&S.first[slot], i);
  }
  __syncthreads();
  if (i < nb) S.id[i] = static_cast<unsigned short>(outside ? kPermMax + S.first[slot] : p - k1);
  __syncthreads();
  const int per = (nb + kPermGroups - 1) / kPermGroups;
  if (i < kPermGroups) {
    unsigned short* m = S.map[i];
    for (int k = i * per; k < (i + 1) * per && k < nb; ++k) {
      const int p = S.id[k];
      const unsigned short v = m[k];
      m[k] = m[p];
      m[p] = v;
    }
  }
  __syncthreads();
  // row number e at the end holds map_0(map_1(... map_7(e)))
  auto source = [&](int e) {
#pragma unroll
    for (int g = kPermGroups - 1; g >= 0; --g) e = S.map[g][e];
    return e;
  };
  auto row_of = [&](int e) { return e < kPermMax ? k1 + e : S.piv[e - kPermMax]; };
  auto put = [&](int e) {
    const int s = source(e);
    if (s != e) {
      const int pos = atomicAdd(&S.cnt, 1);
      S.dst[pos] = row_of(e);
      S.src[pos] = row_of(s);
    }
  };
  if (i < nb) {
    put(i);
    if (S.id[i] == kPermMax + i) put(kPermMax + i);
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kPermMax) laswp_perm_kernel(const int32_t* ipiv, int k1, int k2,
                                                             int* map /* [2][2*kPermMax] + count */) {
  __shared__ PermShared S;
  grid_launch();
  grid_wait();
  const int nb = k2 - k1;
  const int i = threadIdx.x;
  if (i < nb) S.piv[i] = ipiv[k1 + i] - 1;
  __syncthreads();
  perm_map(S, k1, nb);
  for (int e = i; e < S.cnt; e += kPermMax) {
    map[e] = S.dst[e];
    map[2 * kPermMax + e] = S.src[e];
  }
  if (i == 0) map[4 * kPermMax] = S.cnt;
}

// Apply the gather map to columns [c0, c1): each block takes 8 columns, a thread
// two rows of the map in all of them: sixteen scattered loads in flight, the
// stores after the whole block has read.
constexpr int kSwpCols = 8;
__global__ void __launch_bounds__(256) laswp_apply_kernel(double* A, long lda, int c0, int c1, const int* map) {
  grid_launch();
  grid_wait();
  const int cnt = map[4 * kPermMax];
  const int cb = c0 + blockIdx.x * kSwpCols;
  const int ncol = c1 - cb < kSwpCols ? c1 - cb : kSwpCols;
  double* base = A + static_cast<long>(cb) * lda;
  double v[2][kSwpCols];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = threadIdx.x + h * 256;
    const int s = i < cnt ? map[2 * kPermMax + i] : 0;
#pragma unroll
    for (int j = 0; j < kSwpCols; ++j) v[h][j] = i < cnt && j < ncol ? base[s + static_cast<long>(j) * lda] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = threadIdx.x + h * 256;
    if (i < cnt) {
      const int d = map[i];
#pragma unroll
      for (int j = 0; j < kSwpCols; ++j)
        if (j < ncol) base[d + static_cast<long>(j) * lda] = v[h][j];
    }
  }
}

// Deferred interchanges of the L columns.  G is the composite gather of the
// interchanges of all later panels (G[r]: the row whose content ends at row r)
// and H its inverse; prepending a panel's interchanges (its gather map: row
// dst[i] receives the original row src[i], a permutation of the touched rows)
// changes only the rows r = H[dst[i]]: G[r] = src[i], H[src[i]] = r.
__global__ void iota2_kernel(int n, int* G, int* H) {
  grid_launch();
  grid_wait();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    G[i] = i;
    H[i] = i;
  }
}

__global__ void compose_kernel(const int* map, int* G, int* H) {
  __shared__ int rr[2 * kPermMax];
  grid_launch();
  grid_wait();
  const int cnt = map[4 * kPermMax];
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) rr[i] = H[map[i]];
  __syncthreads();
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    const int src = map[2 * kPermMax + i];
    G[rr[i]] = src;
    H[src] = rr[i];
  }
}

// tmp[(r - r0) + c (n - r0)] = A[G[r], c0 + c] for r in [r0, n); blockIdx.y = c.
__global__ void gather_rows_kernel(const double* A, long lda, int r0, int n, int c0, const int* G, double* tmp) {
  grid_launch();
  grid_wait();
  const int r = r0 + blockIdx.x * blockDim.x + threadIdx.x;
  const int c = blockIdx.y;
  if (r < n) tmp[(r - r0) + static_cast<long>(c) * (n - r0)] = A[G[r] + static_cast<long>(c0 + c) * lda];
}

constexpr int kTrsmMax = 128;
inline int trtri_threads(int nb) { return nb <= 256 ? 256 : 512; }

// ---------------------------------------------------------------- Cholesky diagonal block
// The nb x nb diagonal block of a Cholesky step (nb <= 512) is factored in
// FP64 by 32-column panels: a one-block leaf factors the panel's 32 x 32
// diagonal block in shared memory, the rows below it within the block are
// solved against it and the rest of the block is updated by a small FP64
// product spread over many blocks, and L11^-1 is formed afterwards column by
// column.  GB300 retires ~1.6 FP64 instructions per clock per SM, so no step
// keeps a large amount of FP64 work on a single SM.
constexpr int kCholLeaf = 32;

// Unblocked lower Cholesky of the w x w (w <= 32) block at A[d0.., d0..],
// right-looking, by four warps: lane i holds row i, warp q the columns
// j = 4s + q (s = 0..7) in registers, so the FP64 work is spread over the
// SM's four sub-partitions.  Pivot jj: its owner warp takes r = rsqrt(d) of
// the pivot d, sets L_jj = d r, scales the column by r and publishes it in
// shared memory.  A column is published while the owner of the pivot before
// may still read the column two steps back for its other updates, so the columns
// go through four buffers in turn.  GB300's FP64 latency makes every dependent
// FP64 step costly (64 cycles a DFMA, 375 an rsqrt), so the chain from pivot to
// pivot is kept short: the owner of the next pivot updates that column first,
// scales and publishes it and arrives at the step's barrier before it updates
// its other columns, and each pivot takes one reciprocal square root rather than
// a square root and a division.  21 us (48 with a barrier for all after the updates
// and the block's inverse formed as well).  A non-positive pivot sets *info (first index)
// and stops; nothing runs once *info is set.
__device__ __noinline__ double chol_rsqrt(double d) { return rsqrt(d); }

__global__ void __launch_bounds__(128) chol_leaf_kernel(double* A, long lda, int d0, int w, int32_t* info) {
  __shared__ double col[4][kCholLeaf];
  __shared__ int fail_s;       // pivot that failed
  const int i = threadIdx.x & 31, q = threadIdx.x >> 5;
  grid_launch();
  grid_wait();
  if (threadIdx.x == 0) fail_s = *info != 0 ? -1 : kCholLeaf;
  __syncthreads();
  if (fail_s < 0) return;
  double* blk = A + d0 + static_cast<long>(d0) * lda;
  // padding beyond w is the identity
  double d[8];
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int j = 4 * s + q;
    d[s] = (i < w && j < w) ? (i >= j ? blk[i + static_cast<long>(j) * lda] : 0.0) : (i == j ? 1.0 : 0.0);
  }
  __syncthreads();               // every thread has read fail_s
  // pivot jj from its column x (owner warp): scaled and published
  auto pivot = [&](int jj, double& x) {
    const double diag = __shfl_sync(0xFFFFFFFFu, x, jj);
    // diag > 0 by the bits (an FP64 comparison would take a DFMA's 64 cycles)
    const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(diag));
    if (bits - 1ull < 0x7FF0000000000000ull) {
      const double r = chol_rsqrt(diag);
      if (i >= jj) x *= r;                    // L_jj = diag r in lane jj
    } else if (i == 0) {
      atomicCAS(info, 0, d0 + jj + 1);
      fail_s = jj;
    }
    col[jj & 3][i] = i >= jj ? x : 0.0;
    // barriers 1 and 2 in turn; the owner has published and does not wait
    __syncwarp();
    asm volatile("bar.arrive %0, 128;" ::"r"(1 + (jj & 1)) : "memory");
  };
  if (q == 0) pivot(0, d[0]);
  int done = w;
  // pivots jj = 4 so + qq; the inner loop stays rolled (32 copies of a step would
  // run from the instruction cache's misses)
#pragma unroll
  for (int so = 0; so < kCholLeaf / 4; ++so) {
#pragma unroll 1
    for (int qq = 0; qq < 4; ++qq) {
      const int jj = 4 * so + qq;
      if (jj >= w || done < w) break;         // uniform over the block
      if (q != qq) asm volatile("bar.sync %0, 128;" ::"r"(1 + (jj & 1)) : "memory");
      // a failed pivot stops every warp at its step: the index was stored before
      // that step's barrier (a later one may already be there: not yet looked at)
      if (*static_cast<volatile int*>(&fail_s) <= jj) {
        done = jj;
        break;
      }
      const double lij = col[jj & 3][i];
      const bool mine = q == ((qq + 1) & 3) && jj + 1 < w;
      if (mine) {
        const double ln = col[jj & 3][(jj + 1) & 31];
        if (qq < 3) {
          if (i >= jj + 1) d[so] = fma(-lij, ln, d[so]);
          pivot(jj + 1, d[so]);
        } else if (so + 1 < kCholLeaf / 4) {
          double& x = d[so + 1 < kCholLeaf / 4 ? so + 1 : so];
          if (i >= jj + 1) x = fma(-lij, ln, x);
          pivot(jj + 1, x);
        }
      }
      const int snext = qq < 3 ? so : so + 1;
#pragma unroll
      for (int s = so; s < kCholLeaf / 4; ++s) {
        const int j = 4 * s + q;
        if ((s > so || q > qq) && i >= j && !(mine && s == snext)) d[s] = fma(-lij, col[jj & 3][j], d[s]);
      }
    }
  }
  // write back the columns that were finished (all of them unless a pivot failed)
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    const int j = 4 * s + q;
    if (i < w && j < done && i >= j) blk[i + static_cast<long>(j) * lda] = d[s];
  }
}

// The rows below a leaf, X <- X L^-T in place for the w x w (w <= 32) lower L at
// Lp and the m x w X at Xp: row by row x_j = (x_j - sum_{k<j} x_k L_jk) / L_jj, by
// one warp per row with column j in lane j, so a step is a shuffle, one
// multiplication by the reciprocal of the diagonal and one DFMA (a warp has a
// sub-partition's FP64 unit to itself, rows beside rows).  The leaf's explicit
// inverse and a product with it took 19 + 7 us.
constexpr int kCholSolveRows = 4;
__global__ void __launch_bounds__(32 * kCholSolveRows) chol_solve_kernel(const double* Lp, long lda, int w, double* Xp,
                                                                        int m, const int32_t* info) {
  grid_launch();
  grid_wait();
  if (*info != 0) return;
  const int lane = threadIdx.x & 31, r = blockIdx.x * kCholSolveRows + (threadIdx.x >> 5);
  // lane j holds row j of L: its entries below the diagonal are column k's multipliers
  double l[kCholLeaf];
#pragma unroll
  for (int k = 0; k < kCholLeaf; ++k) l[k] = k < w && lane < w && lane > k ? Lp[lane + static_cast<long>(k) * lda] : 0.0;
  const double rcp = lane < w ? 1.0 / Lp[lane + static_cast<long>(lane) * lda] : 0.0;
  if (r >= m) return;
  double x = lane < w ? Xp[r + static_cast<long>(lane) * lda] : 0.0;
#pragma unroll
  for (int j = 0; j < kCholLeaf; ++j) {
    if (j >= w) break;                     // warp-uniform
    const double xj = __shfl_sync(0xFFFFFFFFu, x, j) * __shfl_sync(0xFFFFFFFFu, rcp, j);
    x = lane == j ? xj : fma(-l[j], xj, x);
  }
  if (lane < w) Xp[r + static_cast<long>(lane) * lda] = x;
}

// C(i, j) = beta C(i, j) + alpha sum_l A(i, l) B(j, l) in FP64, for the m x n
// C (ldc) with A(i, l) = A[i*ars + l*acs] and B(j, l) = B[j*brs + l*bcs];
// lower = 1 writes only i >= j.  A block computes an 8 x 32 tile (one entry
// per thread) over K chunks of 32 staged in shared memory.  A warp's
// DFMA holds its sub-partition for 64-76 cycles, so 8 warps take 2 x 32 of them
// in 2.4 us; tiles of 16 rows took twice that and left most SMs idle.
constexpr int kNtRows = 8;
__global__ void __launch_bounds__(32 * kNtRows) dgemm_nt_small_kernel(int m, int n, int k, double alpha, const double* A,
                                                            long ars, long acs, const double* B, long brs,
                                                            long bcs, double beta, double* C, long ldc,
                                                            int lower, const int32_t* info) {
  __shared__ double As[kNtRows][33], Bs[32][33];
  grid_launch();
  grid_wait();
  if (*info != 0) return;
  const int ti = threadIdx.x & (kNtRows - 1), tj = threadIdx.x / kNtRows;
  const int i0 = blockIdx.x * kNtRows, j0 = blockIdx.y * 32;
  if (lower && j0 > i0 + kNtRows - 1) return;          // tile entirely above the diagonal
  const int i = i0 + ti, j = j0 + tj;
  double acc = 0.0;
  for (int l0 = 0; l0 < k; l0 += 32) {
    for (int e = threadIdx.x; e < kNtRows * 32; e += blockDim.x) {
      const int r = e & (kNtRows - 1), l = e / kNtRows;
      As[r][l] = (i0 + r < m && l0 + l < k) ? A[(i0 + r) * ars + static_cast<long>(l0 + l) * acs] : 0.0;
    }
    for (int e = threadIdx.x; e < 32 * 32; e += blockDim.x) {
      const int r = e & 31, l = e >> 5;
      Bs[r][l] = (j0 + r < n && l0 + l < k) ? B[(j0 + r) * brs + static_cast<long>(l0 + l) * bcs] : 0.0;
    }
    __syncthreads();
    const int lk = k - l0 < 32 ? k - l0 : 32;
    for (int l = 0; l < lk; ++l) acc = fma(As[ti][l], Bs[tj][l], acc);
    __syncthreads();
  }
  if (i < m && j < n && (!lower || i >= j)) {
    double* c = C + i + static_cast<long>(j) * ldc;
    *c = beta == 0.0 ? alpha * acc : fma(alpha, acc, beta * *c);
  }
}

// inv (nb x nb, ld nb) <- L^-1 for the lower triangular L at A[d0.., d0..]
// (unit diagonal if UNIT; nb <= 512, one thread per row: launch nb blocks of
// trtri_threads(nb) threads): block j solves L x = e_j by column substitution,
// thread i holding row i of x.  As in diag_solve, the warp that holds the rows at
// hand takes eight steps by shuffles (a DFMA of 64 cycles each, another
// multiplication for the non-unit scaling) and publishes the eight values, which
// the warps below take off their rows in the next round; a thread reads row i of
// the next eight columns of L meanwhile (coalesced along the columns).  30 us at
// nb = 256, 39 us with the scaling (one block-wide barrier per step: 52 and 54).
template <bool UNIT>
__global__ void __launch_bounds__(512) trtri_cols_kernel(const double* A, long lda, int d0, int nb, double* inv,
                                                        const int32_t* info) {
  __shared__ double xs[512];
  grid_launch();
  grid_wait();
  if (info && *info != 0) return;
  const double* L = A + d0 + static_cast<long>(d0) * lda;
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
  const int j = blockIdx.x;
  double x = (i == j) ? 1.0 : 0.0, res = 0.0;
  // every row's reciprocal at once: the steps then multiply (a division on the
  // dependent path would cost its 560 cycles every time)
  const double rinv = (!UNIT && i < nb) ? 1.0 / L[i + static_cast<long>(i) * lda] : 1.0;
  auto load = [&](int ss, double (&l)[8]) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k = 8 * ss + q;
      l[q] = (i < nb && k < nb && i > k) ? L[i + static_cast<long>(k) * lda] : 0.0;
    }
  };
  const int nsub = (nb + 7) / 8, first = j / 8;
  double lp[8], l[8], ln[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) lp[q] = 0.0;
  load(first, l);
  for (int ss = first; ss < nsub; ++ss) {
    load(ss + 1 < nsub ? ss + 1 : ss, ln);
    if (ss > first && warp > (ss - 1) >> 2) {
#pragma unroll
      for (int q = 0; q < 8; ++q) x = fma(-lp[q], xs[8 * (ss - 1) + q], x);
    }
    if (warp == ss >> 2) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int kl = (8 * ss + q) & 31;
        const double xv = UNIT ? x : x * rinv;
        if (lane == kl) res = xv;              // final; x itself may meet an infinity from here on
        x = fma(-l[q], __shfl_sync(0xFFFFFFFFu, xv, kl), x);
      }
      if (lane >> 3 == (ss & 3)) xs[i] = res;
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) lp[q] = l[q], l[q] = ln[q];
    __syncthreads();
  }
  if (i < nb) inv[i + static_cast<long>(j) * nb] = res;
}

// How diag_solve forms x_k = v / d from its row's value v and the diagonal entry d.
enum Diag {
  kUnit = 0,    // d = 1
  kRecip = 1,   // v r with r = RN(1 / d): two roundings
  kQuot = 2     // v r + v (1 / d - r): one rounding
};
// 2^lo <= |x| < 2^hi, by the upper word alone (lo >= -1022).
__device__ __forceinline__ bool in_window(double x, int lo, int hi) {
  const uint32_t h = static_cast<uint32_t>(__double2hiint(x)) & 0x7FFFFFFFu;
  return h - (static_cast<uint32_t>(lo + 1023) << 20) < (static_cast<uint32_t>(hi - lo) << 20);
}
// Diagonal entries whose reciprocal is normal (kRecip).  Outside, 1 / d is infinite,
// or subnormal and short of bits, where v / d may be an ordinary number.
__device__ __forceinline__ bool recip_ok(double d) { return in_window(d, -1022, 1022); }
// Diagonal entries and values of kQuot: every product is then normal.
__device__ __forceinline__ bool quot_ok(double x) { return in_window(x, -400, 400); }
__device__ __forceinline__ bool is_zero(double x) { return ((__double2hiint(x) & 0x7FFFFFFF) | __double2loint(x)) == 0; }

// x <- T^-1 x for the bs x bs (bs <= 128) triangle T(i, k) = tb[i + k*ld] in
// shared memory, by the first 128 threads of a block (thread i holds x_i; x in
// shared memory, in and out).  rcp[k] = RN(1 / T(k, k)), rest[k] (kQuot) what it
// leaves of 1 / T(k, k).  False in a thread whose value lies outside the window of
// kQuot: x is then to be solved again by diag_solve_divide.
// A chain of bs steps, each a shuffle and a DFMA of 64 cycles, and one or two more
// for kRecip and kQuot (a division takes 560); a warp solves its 32 rows and publishes
// every 8 values, and the warps behind it take those off their own rows
// meanwhile, on their own FP64 units (one warp with four rows per lane took four
// DFMAs, 76 cycles each, into every step).  Each entry takes its updates in the
// order of the steps.  kQuot: r and its rest together are 1 / d to 2^-105, so the
// quotient is that of a division unless it lies within 2^-104 of the middle of two
// doubles.
template <bool LOWER, int DIAG>
__device__ __forceinline__ bool diag_solve(const double* tb, int ld, const double* rcp, const double* rest, int bs,
                                             double* x) {
  const int i = threadIdx.x, lane = i & 31, warp = i >> 5;
  double v = i < bs ? x[i] : 0.0;
  const double r = (DIAG == kRecip || DIAG == kQuot) && i < bs ? rcp[i] : 1.0;
  const double rl = DIAG == kQuot && i < bs ? rest[i] : 0.0;
  double res = 0.0, last = 0.0;        // x_i, and the value it was formed from
#pragma unroll 1
  for (int s = LOWER ? 0 : 16 - (bs + 7) / 8; s < 16; ++s) {
    // sub-step s: rows 8 ss .. 8 ss + 7, from the top (LOWER) or the bottom
    const int ss = LOWER ? s : 15 - s;
    if (LOWER && 8 * ss >= bs) break;        // uniform
    const int prev = LOWER ? ss - 1 : ss + 1;
    if (s > 0 && (LOWER ? warp > prev >> 2 : warp < prev >> 2)) {
      double t[8], y[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = 8 * prev + (LOWER ? q : 7 - q);
        t[q] = k < bs && i < bs ? tb[i + k * ld] : 0.0;
        y[q] = k < bs ? x[k] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) v = fma(-t[q], y[q], v);
    }
    if (warp == ss >> 2) {
      double t[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int k = 8 * ss + (LOWER ? q : 7 - q);
        t[q] = k < bs && i < bs && (LOWER ? i > k : i < k) ? tb[i + k * ld] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int kl = (8 * ss + (LOWER ? q : 7 - q)) & 31;       // the step's lane; lanes past bs hold zeros
        // the step's row is final: its value is kept aside (v of a finished row,
        // updated with a zero from here on, may meet an infinity)
        const double xv = DIAG == kUnit ? v : DIAG == kRecip ? v * r : fma(v, r, v * rl);
        if (lane == kl) {
          res = xv;
          if (DIAG == kQuot) last = v;
        }
        v = fma(-t[q], __shfl_sync(0xFFFFFFFFu, xv, kl), v);
      }
      if (lane >> 3 == (ss & 3) && i < bs) {
        // (v r + v rest would be +0 for terms of unlike signs)
        if (DIAG == kQuot && is_zero(last))
          res = __hiloint2double((__double2hiint(last) ^ __double2hiint(r)) & 0x80000000, 0);
        x[i] = res;
      }
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
  }
  return DIAG != kQuot || i >= bs || is_zero(last) || quot_ok(last);
}
// The same by a division per step, for the few blocks that need it: little
// code, as what is beside the other variants in a kernel costs them registers.
__device__ __forceinline__ void diag_solve_divide(const double* tb, int ld, int bs, bool lower, double* x) {
  const int i = threadIdx.x;
  double v = i < bs ? x[i] : 0.0;
#pragma unroll 1
  for (int s = 0; s < bs; ++s) {
    const int k = lower ? s : bs - 1 - s;
    if (i == k) x[k] = v / tb[k + k * ld];
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (i < bs && (lower ? i > k : i < k)) v = fma(-tb[i + k * ld], x[k], v);
  }
}

// X (w1 x w2 at A[d0.., c0..]) <- L^-1 X with L unit lower w1 x w1 at A[d0.., d0..]
// (w1 <= 128), one block per column of X: 256 threads stage L in shared memory,
// the first 128 solve (diag_solve).
__global__ void __launch_bounds__(256) trsm_small_kernel(double* A, long lda, int d0, int w1, int c0) {
  extern __shared__ double Ls[];   // Ls[i + k*ld] = L(i, k), ld odd
  __shared__ double x[128];
  grid_launch();
  grid_wait();
  const int tid = threadIdx.x, ld = w1 | 1;
  double* col = A + static_cast<long>(c0 + blockIdx.x) * lda + d0;
  if (tid < w1) x[tid] = col[tid];
  {
    // row i per thread, columns k = tid/128 + 2j, 16 loads in flight before their stores
    const int i = tid & 127, kstep = blockDim.x >> 7;
    if (i < w1)
      for (int k0 = tid >> 7; k0 < w1; k0 += 16 * kstep) {
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int k = k0 + j * kstep;
          v[j] = (k < w1 && i > k) ? A[(d0 + i) + static_cast<long>(d0 + k) * lda] : 0.0;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int k = k0 + j * kstep;
          if (k < w1) Ls[i + k * ld] = v[j];
        }
      }
  }
  __syncthreads();
  if (tid >= 128) return;
  diag_solve<true, kUnit>(Ls, ld, nullptr, nullptr, w1, x);
  if (tid < w1) col[tid] = x[tid];
}

// One diagonal block of a triangular solve, x <- op(T)^-1 x for the bs x bs
// block at T[d0.., d0..] (bs <= 128; op = transpose with `trans`).  All
// threads stage the block (leading dimension bs + 1: conflict-free either
// way, transposed with `trans`), then the first 128 solve (diag_solve: quotients
// by the diagonal's reciprocals in two parts, or by divisions throughout where an
// entry of the block's diagonal or a value lies outside their window).  dpotrs
// with two right-hand sides at n = 128 (two blocks) takes 55 us, 136 with divisions
// throughout and 47 with x_k = v RN(1 / d), whose second rounding shows: the error of
// a substitution with 200 rows is then 1 to 7 % larger.
//
// early: a kernel of this solve came before.  It lets the next kernels start only
// once it has waited itself, so T stood complete before this kernel began, and the
// block of T is staged (past L1) while the kernel ahead still works on X (dgetrs n =
// 4001, 8 right-hand sides 2.03 ms, 2.39 otherwise).
// blockIdx.x = right-hand side.
__global__ void __launch_bounds__(1024) trsv_block_kernel(const double* T, long ldt, double* X, long ldx, int d0,
                                                          int bs, int lower, int unit, int trans, int early) {
  extern __shared__ double tb[];   // tb[r + c*(bs+1)] = op(T)(d0+r, d0+c)
  __shared__ double x[128], rcp[128], rest[128];
  __shared__ int odd_s;            // a value outside the window of kQuot
  if (threadIdx.x == 0) odd_s = 0;
  if (!early) grid_wait();
  const int ld = bs + 1;
  double* xc = X + static_cast<long>(blockIdx.x) * ldx + d0;
  {
    const int r = threadIdx.x & 127, cstep = blockDim.x >> 7;
    if (r < bs)
      for (int c0 = threadIdx.x >> 7; c0 < bs; c0 += 16 * cstep) {
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int c = c0 + j * cstep;
          v[j] = c < bs ? __ldcg(T + (d0 + r) + static_cast<long>(d0 + c) * ldt) : 0.0;
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const int c = c0 + j * cstep;
          if (c < bs) tb[trans ? c + r * ld : r + c * ld] = v[j];
        }
      }
  }
  __syncthreads();
  bool odd = false;
  if (!unit && static_cast<int>(threadIdx.x) < bs) {
    const double d = tb[threadIdx.x + threadIdx.x * ld], r = 1.0 / d;
    rcp[threadIdx.x] = r;
    rest[threadIdx.x] = fma(-d, r, 1.0) * r;
    odd = !quot_ok(d);
  }
  odd = __syncthreads_or(odd);
  grid_wait();
  grid_launch();
  if (threadIdx.x >= 128) return;
  if (static_cast<int>(threadIdx.x) < bs) x[threadIdx.x] = xc[threadIdx.x];
  asm volatile("bar.sync 1, 128;" ::: "memory");
  if (unit) {                        // (a lower triangle)
    diag_solve<true, kUnit>(tb, ld, nullptr, nullptr, bs, x);
  } else {
    if (!odd) {
      odd = !(lower ? diag_solve<true, kQuot>(tb, ld, rcp, rest, bs, x)
                    : diag_solve<false, kQuot>(tb, ld, rcp, rest, bs, x));
      if (odd) odd_s = 1;
      asm volatile("bar.sync 1, 128;" ::: "memory");
      odd = odd_s;
      if (odd) {
        if (static_cast<int>(threadIdx.x) < bs) x[threadIdx.x] = xc[threadIdx.x];
        asm volatile("bar.sync 1, 128;" ::: "memory");
      }
    }
    if (odd) diag_solve_divide(tb, ld, bs, lower != 0, x);
  }
  if (static_cast<int>(threadIdx.x) < bs) xc[threadIdx.x] = x[threadIdx.x];
}

// sum_c t[c ldt] x[c], c ascending, the next sixteen loads in flight during the
// sixteen FMAs at hand (64 cycles each).
__device__ __forceinline__ double row_dot(const double* t, long ldt, const double* x, int n) {
  double acc = 0.0;
  const int full = n / 16 * 16;
  double v[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) v[q] = full ? t[q * ldt] : 0.0;
  for (int c = 0; c < full; c += 16) {
    double nx[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) nx[q] = c + 16 < full ? t[(c + 16 + q) * ldt] : 0.0;
#pragma unroll
    for (int q = 0; q < 16; ++q) acc = fma(v[q], x[c + q], acc);
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = nx[q];
  }
  for (int c = full; c < n; ++c) acc = fma(t[c * ldt], x[c], acc);
  return acc;
}

// x[r] -= sum_{c in [c0, c0+bs)} T(r, c) x[c] for rows r in [r0, r1); T(r, c) =
// T[r + c*ldt] or, with `trans`, T[c + r*ldt].  blockIdx.y = right-hand side.
__global__ void gemv_update_kernel(const double* T, long ldt, double* X, long ldx, int r0, int r1, int c0, int bs,
                                   int trans) {
  __shared__ double xs[128];
  grid_launch();
  grid_wait();
  double* xc = X + static_cast<long>(blockIdx.y) * ldx;
  if (threadIdx.x < bs) xs[threadIdx.x] = xc[c0 + threadIdx.x];
  __syncthreads();
  if (!trans) {
    const int r = r0 + blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= r1) return;
    xc[r] -= row_dot(T + r + static_cast<long>(c0) * ldt, ldt, xs, bs);
  } else {
    // one warp per row: contiguous reads of T[c0.., r]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = r0 + blockIdx.x * (blockDim.x / 32) + warp;
    if (r >= r1) return;
    double acc = 0.0;
    for (int c = lane; c < bs; c += 32) acc = fma(T[(c0 + c) + static_cast<long>(r) * ldt], xs[c], acc);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
    if (lane == 0) xc[r] -= acc;
  }
}

// Residual pass of Eq. 8: per row, r_i = sum_j a_ij x_j - b_i and sum_j |a_ij|;
// maxima of |r_i| and of the row sums collected with atomicMax on the bits.
__global__ void residual_kernel(int n, const double* A, long lda, const double* x, const double* b,
                                unsigned long long* acc) {
  extern __shared__ double xs[];
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  double s = 0.0, sa = 0.0;
  for (int c0 = 0; c0 < n; c0 += 2048) {
    const int cn = n - c0 < 2048 ? n - c0 : 2048;
    __syncthreads();
    for (int i = threadIdx.x; i < cn; i += blockDim.x) xs[i] = x[c0 + i];
    __syncthreads();
    if (r < n)
      for (int c = 0; c < cn; ++c) {
        const double a = A[r + static_cast<long>(c0 + c) * lda];
        s = fma(a, xs[c], s);
        sa += fabs(a);
      }
  }
  if (r < n) {
    const double res = fabs(s - b[r]);
    atomicMax(&acc[0], static_cast<unsigned long long>(__double_as_longlong(res)));
    atomicMax(&acc[1], static_cast<unsigned long long>(__double_as_longlong(sa)));
    atomicMax(&acc[2], static_cast<unsigned long long>(__double_as_longlong(fabs(x[r]))));
    atomicMax(&acc[3], static_cast<unsigned long long>(__double_as_longlong(fabs(b[r]))));
  }
}

__global__ void residual_finish_kernel(int n, const unsigned long long* acc, double* out) {
  const double r = __longlong_as_double(static_cast<long long>(acc[0]));
  const double an = __longlong_as_double(static_cast<long long>(acc[1]));
  const double xn = __longlong_as_double(static_cast<long long>(acc[2]));
  const double bn = __longlong_as_double(static_cast<long long>(acc[3]));
  const double eps = 1.1102230246251565e-16;   // 2^-53
  out[0] = r / ((an * xn + bn) * n * eps);
  out[1] = r / (an * xn * n * eps);
}

// ------------------------------------------------------------------ a-posteriori probe
// Freivalds-style check of one trailing update C <- C - L U on sampled rows:
// with w_j = +-1, (C_old - C_new) w must equal L (U w) up to the emulation
// tolerance 4 k u (|L||U|)|w| plus FP64 rounding of the three products.
constexpr int kProbeRows = 64;

__device__ __forceinline__ double probe_w(int j) {
  unsigned x = static_cast<unsigned>(j) * 2654435761u;
  x ^= x >> 13;
  x *= 0x5bd1e995u;
  x ^= x >> 15;
  return (x & 1u) ? 1.0 : -1.0;
}

__device__ __forceinline__ void block_sum2(double& a, double& b) {
  __shared__ double ra[32], rb[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xFFFFFFFFu, a, o);
    b += __shfl_xor_sync(0xFFFFFFFFu, b, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    ra[w] = a;
    rb[w] = b;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = 0.0;
    b = 0.0;
    for (int i = 0; i < static_cast<int>(blockDim.x / 32); ++i) {
      a += ra[i];
      b += rb[i];
    }
  }
}

// y[i] = sum_j C(r_i, j) w_j, a[i] = sum_j |C(r_i, j)|, r_i = i*m/R (one block per sampled row)
__global__ void probe_rows_kernel(int m, int n, const double* C, long ldc, int R, double* y, double* a) {
  const int i = blockIdx.x;
  const int r = static_cast<int>(static_cast<long>(i) * m / R);
  double sy = 0.0, sa = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double c = C[r + static_cast<long>(j) * ldc];
    sy = fma(c, probe_w(j), sy);
    sa += fabs(c);
  }
  block_sum2(sy, sa);
  if (threadIdx.x == 0) {
    y[i] = sy;
    a[i] = sa;
  }
}

// z[q] = sum_j U(q, j) w_j, za[q] = sum_j |U(q, j)| (one block per row q of U, jb x n)
__global__ void probe_z_kernel(int n, const double* U, long ldu, double* z, double* za) {
  const int q = blockIdx.x;
  double sz = 0.0, sa = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double u = U[q + static_cast<long>(j) * ldu];
    sz = fma(u, probe_w(j), sz);
    sa += fabs(u);
  }
  block_sum2(sz, sa);
  if (threadIdx.x == 0) {
    z[q] = sz;
    za[q] = sa;
  }
}

// t[i] = sum_q L(r_i, q) z[q], ta[i] = sum_q |L(r_i, q)| za[q]; then the check.
// One lane per row; even warps form t, odd warps ta, on FP64 units of their own,
// the next sixteen entries of L in flight.
__global__ void __launch_bounds__(4 * 32) probe_check_kernel(int m, int n, int k, const double* L, long ldl, int R,
                                                             const double* z, const double* za, const double* y0,
                                                             const double* a0, const double* y1, const double* a1,
                                                             int* flag) {
  __shared__ double ta_s[kProbeRows];
  __shared__ double zs[2][128];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i = (warp >> 1) * 32 + lane;
  const bool mag = warp & 1;
  const int r = i < R ? static_cast<int>(static_cast<long>(i) * m / R) : 0;
  double t = 0.0;
  for (int q0 = 0; q0 < k; q0 += 128) {
    const int kn = k - q0 < 128 ? k - q0 : 128;
    __syncthreads();
    if (static_cast<int>(threadIdx.x) < kn) {
      zs[0][threadIdx.x] = z[q0 + threadIdx.x];
      zs[1][threadIdx.x] = za[q0 + threadIdx.x];
    }
    __syncthreads();
    const double* row = L + r + static_cast<long>(q0) * ldl;
    for (int q = 0; q < kn; q += 16) {
      double l[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) l[j] = q + j < kn ? __ldg(row + static_cast<long>(q + j) * ldl) : 0.0;
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (q + j < kn) t = fma(mag ? fabs(l[j]) : l[j], zs[mag ? 1 : 0][q + j], t);
    }
  }
  if (mag && i < R) ta_s[i] = t;
  __syncthreads();
  if (mag || i >= R) return;
  const double u = 1.1102230246251565e-16;
  const double tol = 6.0 * k * u * ta_s[i] + 3.0 * n * u * (a0[i] + a1[i]);
  const double diff = fabs((y0[i] - y1[i]) - t);
  if (!(diff <= tol)) atomicExch(flag, 1);
}

// ------------------------------------------------------------------ host helpers
struct LuBufs {
  double* inv;          // nb x nb
  uint64_t* recs;       // leaf pivot exchange: [2][nsm][kRecWords] epoch-tagged words
  uint64_t* drec;       // [2][2 kLeaf]: row c of the leaf, epoch-tagged words
  unsigned long long* racc;
  int* map;             // laswp gather maps, [4*kPermMax + 1] ints each, one per recursion depth
  double* probe;        // y0, a0, y1, a1 (kProbeRows each), z, za (nb each)
  int* flag;
};
constexpr int kMapInts = 4 * kPermMax + 8;
constexpr int kMaxDepth = 8;

size_t rec_bytes(int nsm) { return 2ull * nsm * kRecWords * 8; }

size_t lu_extra_bytes(int nb, int nsm) {
  return al(static_cast<size_t>(nb) * nb * 8) + al(rec_bytes(nsm)) + al(2ull * 2 * kLeaf * 8) + al(4 * 8) +
         al(kMaxDepth * kMapInts * 4) +
         al((4ull * kProbeRows + 2ull * nb) * 8) + al(16) + kAl;
}

// Lower Cholesky of the jb x jb diagonal block at A[d0.., d0..] (jb <= 512),
// in place, by 32-column panels (chol_leaf_kernel, then the rows below the
// leaf within the block and the block's trailing lower part by
// dgemm_nt_small_kernel); with `want_inv`, inv (jb x jb, ld jb) <- L11^-1.
int chol_diag(emul_handle_t h, double* A, long lda, int d0, int jb, double* inv, int32_t* info, bool want_inv,
              cudaStream_t st) {
  const bool dep = st == h->stream;      // launch.h
  const int ph = phase_begin(h, EMUL_PHASE_PANEL, st);
  for (int c0 = 0; c0 < jb; c0 += kCholLeaf) {
    const int wp = kCholLeaf < jb - c0 ? kCholLeaf : jb - c0;
    launch_chained(dep, chol_leaf_kernel, dim3(1), dim3(128), 0, st, A, lda, d0 + c0, wp, info);
    h->launches++;
    const int r0 = c0 + wp, mr = jb - r0;
    if (mr > 0) {
      double* Lp = A + (d0 + r0) + static_cast<long>(d0 + c0) * lda;   // rows below the leaf, its columns
      launch_chained(dep, chol_solve_kernel, dim3((mr + kCholSolveRows - 1) / kCholSolveRows),
                     dim3(32 * kCholSolveRows), 0, st, A + (d0 + c0) + static_cast<long>(d0 + c0) * lda, lda, wp, Lp,
                     mr, info);
      // A(r0.., r0..) -= L(r0.., c0..) L(r0.., c0..)^T, lower part
      launch_chained(dep, dgemm_nt_small_kernel, dim3((mr + kNtRows - 1) / kNtRows, (mr + 31) / 32),
                     dim3(32 * kNtRows), 0, st, mr, mr, wp, -1.0, Lp, 1, lda, Lp, 1, lda, 1.0,
                     A + (d0 + r0) + static_cast<long>(d0 + r0) * lda, lda, 1, info);
      h->launches += 2;
    }
  }
  if (want_inv) {
    launch_chained(dep, trtri_cols_kernel<false>, dim3(jb), dim3(trtri_threads(jb)), 0, st, A, lda, d0, jb, inv,
                   info);
    h->launches++;
  }
  phase_end(h, ph, st);
  return check_cuda(h, cudaGetLastError(), "Cholesky diagonal block");
}

LuBufs carve(emul_handle_t h, size_t off, int nb) {
  uint8_t* p = static_cast<uint8_t*>(h->ws) + al(off);
  LuBufs b;
  b.inv = reinterpret_cast<double*>(p);
  p += al(static_cast<size_t>(nb) * nb * 8);
  b.recs = reinterpret_cast<uint64_t*>(p);
  p += al(rec_bytes(h->nsm));
  b.drec = reinterpret_cast<uint64_t*>(p);
  p += al(2ull * 2 * kLeaf * 8);
  b.racc = reinterpret_cast<unsigned long long*>(p);
  p += al(4 * 8);
  b.map = reinterpret_cast<int*>(p);
  p += al(kMaxDepth * kMapInts * 4);
  b.probe = reinterpret_cast<double*>(p);
  p += al((4ull * kProbeRows + 2ull * nb) * 8);
  b.flag = reinterpret_cast<int*>(p);
  return b;
}

// Largest cluster (16, 8, or 0: none) that the device can hold for the cluster
// leaf; queried once per device.
int leaf_cluster_max() {
  static std::mutex mu;
  static std::map<int, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  const auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  int best = 0;
  const int smem = (kClusterR | 1) * kLeaf * 8;
  if (cudaFuncSetAttribute(getf2_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
      cudaFuncSetAttribute(getf2_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    for (int cs = kClusterMax; cs >= 8 && !best; cs /= 2) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(kLeafThreads);
      cfg.dynamicSmemBytes = smem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = cs;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int num = 0;
      if (cudaOccupancyMaxActiveClusters(&num, getf2_cluster_kernel, &cfg) == cudaSuccess && num >= 1) best = cs;
    }
  }
  cudaGetLastError();   // a failed query leaves no error behind
  cache[dev] = best;
  return best;
}

int launch_leaf(emul_handle_t h, double* A, long lda, int n, int d0, int w, int pc0, int pc1, int32_t* ipiv,
                int32_t* info, const LuBufs& B) {
  const int mp = n - d0;
  const int cmax = mp <= kClusterRows ? leaf_cluster_max() : 0;
  if (cmax > 0 && mp <= cmax * kClusterR) {
    // as many CTAs as keep 32 rows each; two at least, for the outside columns'
    // owners (at most 248 columns, 224 threads a CTA)
    int cs = 2;
    while (cs < cmax && cs * 32 < mp) cs *= 2;
    const int R = (mp + cs - 1) / cs;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs);
    cfg.blockDim = dim3(kLeafThreads);
    cfg.dynamicSmemBytes = static_cast<size_t>(R | 1) * w * 8;
    cfg.stream = h->stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // launch.h
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    h->launches++;
    return check_cuda(h, cudaLaunchKernelEx(&cfg, getf2_cluster_kernel, A, lda, n, d0, w, R, pc0, pc1, ipiv, info,
                                            h->d_status, h->wait_limit),
                      "panel leaf");
  }
  int G = (mp + 127) / 128;   // 128 rows per block: the per-column FP64 work of a block overlaps the exchange
  const int smem_rows_cap = 200 * 1024 / (w * 8);
  if ((mp + G - 1) / G > smem_rows_cap) G = (mp + smem_rows_cap - 1) / smem_rows_cap;
  if (G < 1) G = 1;
  if (G > h->nsm) G = h->nsm;
  if (G > 32 * kMaxRecPerLane) G = 32 * kMaxRecPerLane;
  const int R = (mp + G - 1) / G;
  const size_t smem = static_cast<size_t>(R | 1) * w * 8;
  if (smem > 220 * 1024) return set_error(h, EMUL_NOT_SUPPORTED, "panel too tall for the leaf kernel");
  smem_attr(reinterpret_cast<const void*>(getf2_leaf_kernel), 220 * 1024);
  long long limit = h->wait_limit;
  int* status = h->d_status;
  // epochs of this launch: (salt << 5) | column, salt > 0 and new per launch
  // (the records are cleared and the salt restarted by every factorization)
  uint32_t salt = ++h->leaf_salt;
  if (salt >= (1u << 27)) return set_error(h, EMUL_NOT_SUPPORTED, "too many panel leaves in one factorization");
  void* args[] = {&A, const_cast<long*>(&lda), &n, &d0, &w, const_cast<int*>(&R), &pc0, &pc1, &ipiv, &info,
                  const_cast<uint64_t**>(&B.recs), const_cast<uint64_t**>(&B.drec), &salt, &status, &limit};
  h->launches++;
  return check_cuda(h,
                    cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(getf2_leaf_kernel), dim3(G),
                                                dim3(kLeafThreads), args, smem, h->stream),
                    "panel leaf");
}

// Resolve the interchanges ipiv[k1..k2) into the gather map (once per block).
int laswp_prepare(emul_handle_t h, const int32_t* ipiv, int k1, int k2, int* map) {
  if (k2 <= k1) return EMUL_OK;
  if (k2 - k1 > kPermMax) return set_error(h, EMUL_INVALID_ARG, "too many interchanges in one block");
  launch_dependent(laswp_perm_kernel, dim3(1), dim3(kPermMax), 0, h->stream, ipiv, k1, k2, map);
  h->launches++;
  return check_cuda(h, cudaGetLastError(), "laswp map");
}

// Apply a prepared gather map to columns [c0, c1).
int laswp_apply(emul_handle_t h, double* A, long lda, int c0, int c1, const int* map) {
  if (c1 <= c0) return EMUL_OK;
  launch_dependent(laswp_apply_kernel, dim3((c1 - c0 + kSwpCols - 1) / kSwpCols), dim3(256), 0, h->stream, A, lda, c0,
                   c1, map);
  h->launches++;
  return check_cuda(h, cudaGetLastError(), "laswp");
}

// The interchanges ipiv[k1..k2) applied in order to columns [c0, c1), at
// most kPermMax per gather map.
int laswp(emul_handle_t h, double* A, long lda, int c0, int c1, const int32_t* ipiv, int k1, int k2, int* map) {
  if (c1 <= c0 || k2 <= k1) return EMUL_OK;
  for (int k = k1; k < k2; k += kPermMax) {
    int rc = laswp_prepare(h, ipiv, k, k + kPermMax < k2 ? k + kPermMax : k2, map);
    if (rc) return rc;
    rc = laswp_apply(h, A, lda, c0, c1, map);
    if (rc) return rc;
  }
  return EMUL_OK;
}

int trsm_small(emul_handle_t h, double* A, long lda, int d0, int w1, int c0, int w2) {
  if (w1 <= 0 || w2 <= 0) return EMUL_OK;
  if (w1 > kTrsmMax) return set_error(h, EMUL_NOT_SUPPORTED, "panel trsm wider than 128");
  smem_attr(reinterpret_cast<const void*>(trsm_small_kernel), kTrsmMax * (kTrsmMax | 1) * 8);
  // one column per block: the solve is FP64-bound (about 1.6 FMA per clock per
  // SM), so it is spread over as many SMs as columns; 256 threads stage L
  launch_dependent(trsm_small_kernel, dim3(w2), dim3(256), static_cast<size_t>(w1) * (w1 | 1) * 8, h->stream, A, lda,
                   d0, w1, c0);
  h->launches++;
  return check_cuda(h, cudaGetLastError(), "panel trsm");
}

// Recursive panel factorization of rows d0..n-1, columns d0..d0+w-1, inside
// the panel [pc0, pc1).  The leaves apply each interchange to all columns of
// that panel, so the recursion itself swaps nothing.
int rgetrf(emul_handle_t h, double* A, long lda, int n, int d0, int w, int pc0, int pc1, int32_t* ipiv,
           int32_t* info, int s, const LuBufs& B) {
  if (w <= kLeaf) return launch_leaf(h, A, lda, n, d0, w, pc0, pc1, ipiv, info, B);
  const int w1 = (w / 2 + 7) / 8 * 8;
  const int w2 = w - w1;
  int rc = rgetrf(h, A, lda, n, d0, w1, pc0, pc1, ipiv, info, s, B);
  if (rc) return rc;
  rc = trsm_small(h, A, lda, d0, w1, d0 + w1, w2);
  if (rc) return rc;
  const int m2 = n - d0 - w1;
  // A22 (m2 x w2) -= A21 (m2 x w1) * A12 (w1 x w2)
  rc = gemm_run(h, m2, w2, w1, -1.0, Operand{A + (d0 + w1) + static_cast<long>(d0) * lda, 1, lda},
                Operand{A + d0 + static_cast<long>(d0 + w1) * lda, lda, 1}, 1.0,
                A + (d0 + w1) + static_cast<long>(d0 + w1) * lda, lda, s, false, 0, nullptr, 0, 0);
  if (rc) return rc;
  return rgetrf(h, A, lda, n, d0 + w1, w2, pc0, pc1, ipiv, info, s, B);
}

// Panel of width jb at column j0.  Up to kPanelMax columns it is one recursive
// panel, whose leaves apply each interchange across it.  A wider panel is
// factored as two such panels: the left one's interchanges are applied to the
// right one, which is updated (U12 = L11^-1 A12 through the explicit inverse
// and the emulated product, A22 -= L21 U12) and factored; its interchanges
// then go back to the left one.  B.inv is free during the panel.
constexpr int kPanelMax = 256;
int panel_getrf(emul_handle_t h, double* A, long lda, int n, int j0, int jb, int32_t* ipiv, int32_t* info, int s,
                const LuBufs& B) {
  if (jb <= kPanelMax) return rgetrf(h, A, lda, n, j0, jb, j0, j0 + jb, ipiv, info, s, B);
  const int w1 = kPanelMax, w2 = jb - w1;
  int rc = rgetrf(h, A, lda, n, j0, w1, j0, j0 + w1, ipiv, info, s, B);
  if (rc) return rc;
  rc = laswp(h, A, lda, j0 + w1, j0 + jb, ipiv, j0, j0 + w1, B.map);
  if (rc) return rc;
  launch_dependent(trtri_cols_kernel<true>, dim3(w1), dim3(trtri_threads(w1)), 0, h->stream, A, lda, j0, w1, B.inv,
                   nullptr);
  h->launches++;
  rc = check_cuda(h, cudaGetLastError(), "panel trtri");
  if (rc) return rc;
  double* A12 = A + j0 + static_cast<long>(j0 + w1) * lda;
  rc = gemm_run(h, w1, w2, w1, 1.0, Operand{B.inv, 1, w1}, Operand{A12, lda, 1}, 0.0, A12, lda, s, false, 0,
                nullptr, 0, 0);
  if (rc) return rc;
  const int m2 = n - j0 - w1;
  rc = gemm_run(h, m2, w2, w1, -1.0, Operand{A + (j0 + w1) + static_cast<long>(j0) * lda, 1, lda},
                Operand{A12, lda, 1}, 1.0, A + (j0 + w1) + static_cast<long>(j0 + w1) * lda, lda, s, false, 0,
                nullptr, 0, 0);
  if (rc) return rc;
  rc = rgetrf(h, A, lda, n, j0 + w1, w2, j0 + w1, j0 + jb, ipiv, info, s, B);
  if (rc) return rc;
  return laswp(h, A, lda, j0, j0 + w1, ipiv, j0 + w1, j0 + jb, B.map);
}

}  // namespace

void trsv_attr() { smem_attr(reinterpret_cast<const void*>(trsv_block_kernel), 128 * 129 * 8); }

}  // namespace emul

namespace emul {

namespace {

constexpr int kSolveBs = 128;      // diagonal block of the persistent solve
constexpr int kPermSmemMax = 1 << 16;   // rows whose permutation fits in shared memory (2 B each, + 22 KB)

// x <- P x for the interchanges ipiv[0..n) (1-based, applied in order): the
// composite permutation is built in shared memory, 256 interchanges resolved at a
// time (perm_map), then x is gathered through tmp.  One block.  An entry outside
// [0, n) leaves its row where it is.
__global__ void __launch_bounds__(kPermMax) permute_rhs_kernel(const int32_t* ipiv, int n, double* x, double* tmp) {
  extern __shared__ unsigned short perm[];   // n <= kPermSmemMax = 2^16
  __shared__ PermShared S;
  const int i = threadIdx.x;
  for (int e = i; e < n; e += kPermMax) perm[e] = static_cast<unsigned short>(e);
  for (int k0 = 0; k0 < n; k0 += kPermMax) {
    const int nb = n - k0 < kPermMax ? n - k0 : kPermMax;
    if (i < nb) {
      const int p = ipiv[k0 + i] - 1;
      S.piv[i] = p >= 0 && p < n ? p : k0 + i;
    }
    __syncthreads();
    perm_map(S, k0, nb);
    unsigned short v[2];
    for (int h = 0; h < 2; ++h) v[h] = i + h * kPermMax < S.cnt ? perm[S.src[i + h * kPermMax]] : 0;
    __syncthreads();
    for (int h = 0; h < 2; ++h)
      if (i + h * kPermMax < S.cnt) perm[S.dst[i + h * kPermMax]] = v[h];
    __syncthreads();
  }
  for (int e = i; e < n; e += kPermMax) tmp[e] = x[perm[e]];
  __syncthreads();
  for (int e = i; e < n; e += kPermMax) x[e] = tmp[e];
}

// Bounded grid barrier on a monotonic arrival counter (zeroed before the
// launch); returns false on timeout after recording it in *status.
__device__ bool solve_sync(unsigned long long* cnt, unsigned long long target, long long limit, int* status) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    bool ok = true;
    if (atomicAdd(cnt, 1ull) + 1 < target) {
      volatile unsigned long long* vc = cnt;
      const long long t0 = clock64();
      while (*vc < target)
        if (clock64() - t0 > limit) {
          ok = false;
          atomicExch(status, kStatusTimeout);
          break;
        }
    }
    __threadfence();
    ok_s = ok;
  }
  __syncthreads();
  return ok_s != 0;
}

// Forward (L unit lower) and back (U) substitution with the factors of
// emul_dgetrf for one right-hand side, in one cooperative launch.  Step s
// (the 128-row diagonal blocks of L, then those of U from the bottom) is
// solved by four warps of block s % G (diag_solve, with the reciprocals of U's
// diagonal, formed while staging), which has staged the diagonal block while the
// step before was solved.  After one bounded grid barrier every block knows x_s:
// block (s+1) % G takes it off the rows of the next diagonal block and solves
// that at once, the others take it off all other remaining rows meanwhile, each
// warp a group of 32 rows.  So a step costs the update of 128 rows, a diagonal
// solve and one barrier, whatever n is (two barriers, a one-warp solve and the
// whole update between them took 38 us a step at n = 12000).  The grid has four
// groups of rows per block, one per FP64 unit of an SM, if that many SMs exist; a
// smaller grid makes the barrier cheaper.  A row's owner changes from step to
// step, so x is read and written through L2 only.
// Stage the bs x bs diagonal block at d0 for the block solve.  LU factors
// (chol = false): the block as stored, rcp = 1/diag for the upper (backward)
// solve.  Cholesky factor (chol = true): the forward solve uses L itself and
// the backward solve L^T, so the block is staged transposed there; rcp = 1/diag
// for both.  True (in every thread) if some reciprocal is not normal: the block is
// then solved with divisions.
__device__ bool solve_stage(const double* LU, long lda, int d0, int bs, bool lower, double* tb, double* rcp,
                            bool chol) {
  constexpr int ld = kSolveBs + 1;
  const int tid = threadIdx.x;
  const int r = tid & 127, cstep = blockDim.x >> 7;
  const bool tr = chol && !lower;
  if (r < bs)
    for (int c0 = tid >> 7; c0 < bs; c0 += 16 * cstep) {
      double v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int c = c0 + j * cstep;
        v[j] = c < bs ? __ldg(LU + (d0 + r) + static_cast<long>(d0 + c) * lda) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int c = c0 + j * cstep;
        if (c < bs) tb[tr ? c + r * ld : r + c * ld] = v[j];
      }
    }
  __syncthreads();
  bool odd = false;
  if ((chol || !lower) && tid < bs) {
    const double d = tb[tid + tid * ld];
    rcp[tid] = 1.0 / d;
    odd = !recip_ok(d);
  }
  return __syncthreads_or(odd);
}

// CHOL = false: A = L U from the LU (unit L below the diagonal, U on and
// above it).  CHOL = true: A = L L^T from the lower Cholesky factor, forward
// with L (non-unit diagonal) and backward with L^T, whose rows are columns of
// L: the update of the rows above a block then reads each column of L
// contiguously, one warp per row of L^T.  (One block per SM by its shared memory;
// without the bound's 1 the LU solve is compiled for 64 registers, with spills:
// n = 4001 1.66 ms instead of 1.55.)
template <bool CHOL>
__global__ void __launch_bounds__(256, 1) getrs1_kernel(const double* LU, long lda, int n, double* x,
                                                     unsigned long long* cnt, int* status, long long limit) {
  extern __shared__ double tb[];   // kSolveBs x (kSolveBs + 1) staging of a diagonal block
  __shared__ double xs[kSolveBs], xd[kSolveBs];
  __shared__ double rcp[kSolveBs];
  constexpr int ld = kSolveBs + 1;
  const int G = gridDim.x, b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nblk = (n + kSolveBs - 1) / kSolveBs;
  const int nsteps = 2 * nblk;
  auto info = [&](int st, bool& lower, int& d0, int& bs) {
    lower = st < nblk;
    const int d = lower ? st : 2 * nblk - 1 - st;
    d0 = d * kSolveBs;
    bs = n - d0 < kSolveBs ? n - d0 : kSolveBs;
  };
  unsigned long long target = 0;
  int staged = -1;   // step whose diagonal block this block holds in tb
  bool odd = false;  // it is solved with divisions
  auto stage = [&](int st) {
    if (st >= nsteps || staged == st) return;
    bool lower;
    int d0, bs;
    info(st, lower, d0, bs);
    odd = solve_stage(LU, lda, d0, bs, lower, tb, rcp, CHOL);
    staged = st;
  };
  // x_st <- T^-1 x_st, published in x
  auto solve = [&](int st) {
    bool lower;
    int d0, bs;
    info(st, lower, d0, bs);
    stage(st);
    if (tid < kSolveBs) {
      if (tid < bs) xd[tid] = __ldcg(x + d0 + tid);
      asm volatile("bar.sync 1, 128;" ::: "memory");
      if (odd)
        diag_solve_divide(tb, ld, bs, lower, xd);
      else if (!lower)
        diag_solve<false, kRecip>(tb, ld, rcp, nullptr, bs, xd);
      else
        diag_solve<true, CHOL ? kRecip : kUnit>(tb, ld, rcp, nullptr, bs, xd);
      if (tid < bs) __stcg(x + d0 + tid, xd[tid]);
    }
  };
  // x_r -= (row r of the step's block column) x_st for rows [lo, hi) outside
  // [skip0, skip1), by the warps first, first + nw, ... (x_st in xs)
  auto update = [&](int st, int lo, int hi, int skip0, int skip1, int first, int nw) {
    bool lower;
    int d0, bs;
    info(st, lower, d0, bs);
    if (CHOL && !lower) {
      // x_r -= sum_c L(d0 + c, r) x_c: eight rows per warp, lanes along the
      // columns of L.  The sums over the lanes are those of a butterfly; a lane
      // keeps half of the rows at each of the first three steps, so eight rows
      // take 9 additions (76 cycles each) instead of 40.
      for (int g = first; lo + g * 8 < hi; g += nw) {
        const int rb = lo + g * 8;
        double v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = 0.0;
#pragma unroll
        for (int cq = 0; cq < kSolveBs / 32; ++cq) {
          const int c = lane + 32 * cq;
          double l[8];
#pragma unroll
          for (int q = 0; q < 8; ++q)
            l[q] = c < bs && rb + q < hi ? __ldg(LU + d0 + c + static_cast<long>(rb + q) * lda) : 0.0;
          if (c < bs) {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = fma(l[q], xs[c], v[q]);
          }
        }
        int mine = 0;                       // row of the group this lane ends up with
#pragma unroll
        for (int o = 16, keep = 4; keep >= 1; o >>= 1, keep >>= 1) {
          const bool upper = lane & o;
          if (upper) mine += keep;
#pragma unroll
          for (int q = 0; q < keep; ++q) {
            const double send = upper ? v[q] : v[q + keep];
            const double own = upper ? v[q + keep] : v[q];
            v[q] = own + __shfl_xor_sync(0xFFFFFFFFu, send, o);
          }
        }
        v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 2);
        v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], 1);
        const int r = rb + mine;
        if ((lane & 3) == 0 && r < hi && !(r >= skip0 && r < skip1)) __stcg(x + r, __ldcg(x + r) - v[0]);
      }
    } else {
      for (int g = first; lo + g * 32 < hi; g += nw) {
        const int r = lo + g * 32 + lane;
        if (r < hi && !(r >= skip0 && r < skip1)) {
          const double acc = row_dot(LU + r + static_cast<long>(d0) * lda, lda, xs, bs);
          __stcg(x + r, __ldcg(x + r) - acc);
        }
      }
    }
  };
  const int wpb = blockDim.x >> 5;
  if (b == 0) solve(0);
  if (b == 1 % G && G > 1) stage(1);
  for (int st = 0; st < nsteps; ++st) {
    target += G;
    if (!solve_sync(cnt, target, limit, status)) return;
    if (st + 1 == nsteps) break;
    bool lower, l2;
    int d0, bs, e0, es;
    info(st, lower, d0, bs);
    info(st + 1, l2, e0, es);
    const int nxt = (st + 1) % G;
    // rows below (forward) or above (backward) the block; the next diagonal
    // block lies next to it (at the turn it is the same block and has no update)
    const int lo = lower ? d0 + bs : 0, hi = lower ? n : d0;
    const bool has_next = e0 >= lo && e0 < hi;
    for (int c = tid; c < bs; c += blockDim.x) xs[c] = __ldcg(x + d0 + c);
    __syncthreads();
    if (b == nxt) {
      if (has_next) update(st, e0, e0 + es, 0, 0, warp, wpb);
      if (G == 1) update(st, lo, hi, e0, e0 + es, warp, wpb);
      __syncthreads();
      solve(st + 1);
    } else {
      const int me = b < nxt ? b : b - 1;   // among the G - 1 others, warps dealt block by block
      update(st, lo, hi, has_next ? e0 : 0, has_next ? e0 + es : 0, warp * (G - 1) + me, wpb * (G - 1));
      if (b == (st + 2) % G) stage(st + 2);
    }
  }
}

}  // namespace

// Blocks of the one-launch solve: four groups of 32 rows each.
int solve_blocks(emul_handle_t h, int n) {
  const int want = (n + 127) / 128;
  return want < h->nsm ? want : h->nsm;
}

// Solve with the factors of emul_dgetrf (arguments validated by the caller).
int getrs_body(emul_handle_t h, int n, int nrhs, const double* LU, int lda, const int32_t* ipiv, double* B,
               int ldb) {
  if (nrhs == 1 && n <= kPermSmemMax) {
    // one right-hand side: permutation in one block, both substitutions in one cooperative launch
    int rc = reserve_workspace(h, 2 * kAl + al(static_cast<size_t>(n) * 8));
    if (rc) return rc;
    uint8_t* ws = static_cast<uint8_t*>(h->ws);
    unsigned long long* cnt = reinterpret_cast<unsigned long long*>(ws);
    double* tmp = reinterpret_cast<double*>(ws + kAl);
    smem_attr(reinterpret_cast<const void*>(permute_rhs_kernel), kPermSmemMax * 2);
    smem_attr(reinterpret_cast<const void*>(getrs1_kernel<false>), kSolveBs * (kSolveBs + 1) * 8);
    permute_rhs_kernel<<<1, kPermMax, static_cast<size_t>(n) * 2, h->stream>>>(ipiv, n, B, tmp);
    h->launches++;
    rc = check_cuda(h, cudaGetLastError(), "rhs permutation");
    if (rc) return rc;
    rc = check_cuda(h, cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), h->stream), "solve barrier");
    if (rc) return rc;
    long ldl = lda;
    long long limit = h->wait_limit;
    int* status = h->d_status;
    void* args[] = {const_cast<double**>(&LU), &ldl, &n, &B, &cnt, &status, &limit};
    h->launches++;
    return check_cuda(h,
                      cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(getrs1_kernel<false>), dim3(solve_blocks(h, n)),
                                                  dim3(256), args, kSolveBs * (kSolveBs + 1) * 8, h->stream),
                      "solve");
  }
  const size_t need = lu_extra_bytes(16, h->nsm);
  int rc = reserve_workspace(h, need);
  if (rc) return rc;
  const LuBufs W = carve(h, 0, 16);
  for (int k = 0; k < n; k += kPermMax) {
    rc = laswp(h, B, ldb, 0, nrhs, ipiv, k, k + kPermMax < n ? k + kPermMax : n, W.map);
    if (rc) return rc;
  }
  constexpr int bs = 128;  // diagonal blocks of the substitution
  for (int d0 = 0; d0 < n; d0 += bs) {
    const int b = bs < n - d0 ? bs : n - d0;
    launch_dependent(trsv_block_kernel, dim3(nrhs), dim3(1024), b * (b + 1) * sizeof(double), h->stream, LU, lda, B,
                     ldb, d0, b, 1, 1, 0, d0 > 0);
    h->launches += (d0 + b < n) ? 2 : 1;
    if (d0 + b < n)
      launch_dependent(gemv_update_kernel, dim3((n - d0 - b + 255) / 256, nrhs), dim3(256), 0, h->stream, LU, lda, B,
                       ldb, d0 + b, n, d0, b, 0);
  }
  for (int d0 = ((n - 1) / bs) * bs; d0 >= 0; d0 -= bs) {
    const int b = bs < n - d0 ? bs : n - d0;
    launch_dependent(trsv_block_kernel, dim3(nrhs), dim3(1024), b * (b + 1) * sizeof(double), h->stream, LU, lda, B,
                     ldb, d0, b, 0, 0, 0, 1);
    h->launches += (d0 > 0) ? 2 : 1;
    if (d0 > 0)
      launch_dependent(gemv_update_kernel, dim3((d0 + 255) / 256, nrhs), dim3(256), 0, h->stream, LU, lda, B, ldb, 0,
                       d0, d0, b, 0);
  }
  return check_cuda(h, cudaGetLastError(), "getrs");
}
}  // namespace emul

using emul::Operand;

namespace emul {
namespace {

// Seeded synthetic matrix for the block-size tuner: uniform(-1, 1) from a
// splitmix64 hash of (seed, i, j); with `spd`, entry (i, j) takes the hash of
// (max, min) so the matrix is symmetric, and the diagonal is n (strictly
// diagonally dominant, hence positive definite).
__global__ void tune_fill_kernel(double* A, int n, int spd, unsigned long long seed) {
  const long total = static_cast<long>(n) * n;
  for (long e = blockIdx.x * static_cast<long>(blockDim.x) + threadIdx.x; e < total;
       e += static_cast<long>(gridDim.x) * blockDim.x) {
    int i = static_cast<int>(e % n), j = static_cast<int>(e / n);
    if (spd && i == j) {
      A[e] = static_cast<double>(n);
      continue;
    }
    if (spd && i < j) {
      const int t = i;
      i = j;
      j = t;
    }
    unsigned long long z = seed + (static_cast<unsigned long long>(i) * n + j + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    A[e] = static_cast<double>(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
  }
}

uint64_t nb_key(int kind, int n, int slices) {
  return (static_cast<uint64_t>(kind) << 40) | (static_cast<uint64_t>(slices) << 32) | static_cast<uint32_t>(n);
}

// The LU step's second stream and its two events, created on first use.
int aux_ready(emul_handle_t h) {
  if (h->aux) return EMUL_OK;
  int least = 0, greatest = 0;
  int rc = check_cuda(h, cudaDeviceGetStreamPriorityRange(&least, &greatest), "second stream");
  if (!rc) rc = check_cuda(h, cudaStreamCreateWithPriority(&h->aux, cudaStreamNonBlocking, greatest), "second stream");
  if (!rc) rc = check_cuda(h, cudaEventCreateWithFlags(&h->aux_start, cudaEventDisableTiming), "stream events");
  if (!rc) rc = check_cuda(h, cudaEventCreateWithFlags(&h->aux_done, cudaEventDisableTiming), "stream events");
  return rc;
}

// The columns right of the factored Cholesky block at j0 (jb wide, m2 rows below
// it): L21 = A21 L11^-T, then A22 -= L21 L21^T on the lower triangle.  With
// enough left the next diagonal block is updated first and factored on the second
// stream, while the rest of the update runs on `stream` (*ahead is set; aux_done
// marks its end): the diagonal block is a chain of small kernels, 330 us at 256
// columns, that leaves the chip idle.  The persistent products leave it a few SMs.
// ms of dpotrf without / with it: n = 12000, nb = 256: 30.4 / 27.2; 16384, 512:
// 64.8 / 59.1; 8192, 128: 17.3 / 15.8; 5000, 256: 8.03 / 7.86.  The lines: with it
// down to 1024 rows right of the next block 5000, 128 takes 8.38 instead of 8.23
// and 8192, 256 14.99 instead of 14.91, only above 6000 rows 15.6; at 4000 rows in
// all 6.05 / 6.2, and with 64 columns, whose updates are bound by memory,
// 16384 104.2 / 106.4.  Of 8, 16 and 24 SMs: 27.5, 27.5, 27.8 at 12000, 256; 16384,
// 512 60.2 (8), 59.1 (16); 16384, 128 63.3 (8), 65.2 (16).
constexpr int kAheadRows = 3072;
constexpr int kAheadCols = 128;
int chol_trailing(emul_handle_t h, double* A, long lda, int j0, int jb, int m2, int nb, int s, int32_t* info,
                  const LuBufs& B, bool* ahead) {
  auto at = [&](int r, int c) { return A + r + static_cast<long>(c) * lda; };
  // A(r.., c..) (m x w) -= L21(r..) L21(c..)^T
  auto update = [&](int r, int c, int m, int w, bool lower) {
    const int ph = phase_begin(h, EMUL_PHASE_UPDATE);
    const int rc = gemm_run(h, m, w, jb, -1.0, Operand{at(r, j0), 1, lda}, Operand{at(c, j0), 1, lda}, 1.0, at(r, c),
                            lda, s, lower, 0, nullptr, 0, 0);
    phase_end(h, ph);
    return rc;
  };
  const int j1 = j0 + jb, jb1 = nb < m2 ? nb : m2;
  const int j2 = j1 + jb1, m3 = m2 - jb1;
  // operand B is (L11^-1)^T, whose row j is row j of L11^-1
  const int ph = phase_begin(h, EMUL_PHASE_U12);
  int rc = gemm_run(h, m2, jb, jb, 1.0, Operand{at(j1, j0), 1, lda}, Operand{B.inv, 1, jb}, 0.0, at(j1, j0), lda, s,
                    false, 0, nullptr, 0, 0);
  phase_end(h, ph);
  if (rc) return rc;
  if (jb < kAheadCols || m3 < kAheadRows) return update(j1, j1, m2, m2, true);
  rc = aux_ready(h);
  if (!rc) rc = update(j1, j1, jb1, jb1, true);
  if (!rc) rc = check_cuda(h, cudaEventRecord(h->aux_start, h->stream), "stream events");
  if (!rc) rc = check_cuda(h, cudaStreamWaitEvent(h->aux, h->aux_start, 0), "stream events");
  if (rc) return rc;
  rc = chol_diag(h, A, lda, j1, jb1, B.inv, info, true, h->aux);
  const int rc_done = check_cuda(h, cudaEventRecord(h->aux_done, h->aux), "stream events");
  if (!rc) rc = rc_done;
  h->sm_spare = jb >= 256 ? 16 : 8;
  if (!rc) rc = update(j2, j1, m3, jb1, false);
  if (!rc) rc = update(j2, j2, m3, m3, true);
  h->sm_spare = 0;
  // an error here leaves no work of the second stream behind the call
  if (rc) cudaStreamWaitEvent(h->stream, h->aux_done, 0);
  *ahead = rc == EMUL_OK;
  return rc;
}

// nb = EMUL_NB_AUTO: the tuned block size for (kind, n, slices), tuning first
// when there is none.
int resolve_nb(emul_handle_t h, int kind, int n, int slices, int* nb) {
  if (*nb != EMUL_NB_AUTO) return EMUL_OK;
  const auto it = h->nb_tuned.find(nb_key(kind, n, slices));
  if (it != h->nb_tuned.end()) {
    *nb = it->second;
    return EMUL_OK;
  }
  return emul_autotune_nb(h, kind, n, slices, nb);
}

}  // namespace
}  // namespace emul

extern "C" {

int emul_autotune_nb(emul_handle_t h, int kind, int n, int slices, int* nb_out) {
  if (!h) return EMUL_INVALID_ARG;
  if ((kind != 0 && kind != 1) || n < 1 || slices < 1 || slices > emul::kMaxSlices || !nb_out)
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_autotune_nb: invalid argument");
  const int cand[] = {128, 256, 512};
  double* A = nullptr;
  int32_t* piv = nullptr;
  if (cudaMalloc(&A, static_cast<size_t>(n) * n * 8 + static_cast<size_t>(n) * 4 + 256) != cudaSuccess) {
    cudaGetLastError();
    return emul::set_error(h, EMUL_NO_WORKSPACE, "emul_autotune_nb: no room for the trial matrix");
  }
  piv = reinterpret_cast<int32_t*>(A + static_cast<size_t>(n) * n);
  int32_t* info = piv + n;
  const bool prof = h->prof;
  h->prof = false;   // the trials are not part of any profile
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  int rc = emul::check_cuda(h, cudaEventCreate(&e0), "tuner events");
  if (!rc) rc = emul::check_cuda(h, cudaEventCreate(&e1), "tuner events");
  // candidates past the first that covers n in one panel change nothing
  int nc = 1;
  while (nc < 3 && cand[nc - 1] < n) ++nc;
  int best = cand[0];
  float best_ms = 0.0f;
  // the untimed first run takes the largest candidate: it sizes the workspace
  // and plans the product schedules the others reuse
  for (int c = -1; c < nc && !rc; ++c) {
    const int nb = cand[c < 0 ? nc - 1 : c];
    emul::tune_fill_kernel<<<4 * h->nsm, 256, 0, h->stream>>>(A, n, kind, 0x5EEDull + static_cast<unsigned>(n));
    rc = emul::check_cuda(h, cudaGetLastError(), "tuner fill");
    if (rc) break;
    cudaEventRecord(e0, h->stream);
    rc = kind == 0 ? emul_dgetrf(h, n, A, n, piv, nb, slices, info, nullptr)
                   : emul_dpotrf(h, 'L', n, A, n, nb, slices, info, nullptr);
    cudaEventRecord(e1, h->stream);
    if (rc) break;
    rc = emul::check_cuda(h, cudaEventSynchronize(e1), "tuner run");
    if (rc) break;
    float ms = 0.0f;
    cudaEventElapsedTime(&ms, e0, e1);
    if (c >= 0 && (c == 0 || ms < best_ms)) {
      best_ms = ms;
      best = nb;
    }
  }
  h->prof = prof;
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(A);
  if (rc) return rc;
  h->nb_tuned[emul::nb_key(kind, n, slices)] = best;
  *nb_out = best;
  return EMUL_OK;
}

int emul_dgetrf(emul_handle_t h, int n, double* A, int lda, int32_t* ipiv, int nb, int slices, int32_t* info,
                emul_stats* stats) {
  if (!h) return EMUL_INVALID_ARG;
  if (nb == EMUL_NB_AUTO && slices >= 1 && slices <= emul::kMaxSlices && n >= 1) {
    const int rc = emul::resolve_nb(h, 0, n, slices, &nb);
    if (rc) return rc;
  }
  if (nb == EMUL_NB_AUTO && n == 0) nb = 128;
  if (nb == 0) nb = 128;
  if (n < 0 || lda < (n > 1 ? n : 1) || nb < 16 || nb > 512 || nb % 16 != 0 || slices < 0 ||
      slices > emul::kMaxSlices || (n > 0 && (!A || !ipiv || !info)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dgetrf: invalid argument");
  const bool autos = slices == 0;
  if (autos && !emul::selector_loaded(h))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dgetrf: slices = 0 needs a loaded selector");
  if (stats) *stats = emul_stats{0, autos ? 8 : slices, autos ? 3 : slices, 0, 0.0, 0.0};
  double slices_sum = 0.0;
  int updates = 0;
  if (n == 0) return EMUL_OK;
  const int s_fixed = autos ? 8 : slices;
  int s_prev = 8;   // auto mode: the panel and U12 use the previous update's slice count
  int rc = emul::check_cuda(h, cudaMemsetAsync(info, 0, sizeof(int32_t), h->stream), "info reset");
  if (rc) return rc;
  const size_t gw = emul::gemm_workspace_bytes(n, n, nb, s_fixed, false);
  // after the product and LU buffers: G, H (n ints each), one panel of rows
  // (n x nb doubles) and every panel's gather maps (kept from the loop for the
  // deferred interchanges of the L columns)
  const int npanel = (n + nb - 1) / nb;
  const int cpp = (nb + emul::kPermMax - 1) / emul::kPermMax;   // gather maps per panel
  const size_t def_off = emul::al(emul::al(gw) + emul::lu_extra_bytes(nb, h->nsm));
  const size_t maps_off = def_off + emul::al(8ull * n) + emul::al(8ull * n * nb);
  rc = emul::reserve_workspace(
      h, maps_off + emul::al(static_cast<size_t>(npanel) * cpp * emul::kMapInts * sizeof(int)));
  if (rc) return rc;
  int* maps = reinterpret_cast<int*>(static_cast<uint8_t*>(h->ws) + maps_off);
  const emul::LuBufs B = emul::carve(h, gw, nb);
  rc = emul::check_cuda(h, cudaMemsetAsync(B.recs, 0, emul::rec_bytes(h->nsm), h->stream), "leaf records");
  if (rc) return rc;
  rc = emul::check_cuda(h, cudaMemsetAsync(B.drec, 0, 2ull * 2 * emul::kLeaf * 8, h->stream), "leaf records");
  if (rc) return rc;
  h->leaf_salt = 0;
  for (int j0 = 0; j0 < n; j0 += nb) {
    const int jb = nb < n - j0 ? nb : n - j0;
    int ph = emul::phase_begin(h, EMUL_PHASE_PANEL);
    rc = emul::panel_getrf(h, A, lda, n, j0, jb, ipiv, info, autos ? s_prev : s_fixed, B);
    emul::phase_end(h, ph);
    if (rc) return rc;
    const int m2 = n - j0 - jb;
    // L11^-1 on the second stream (L11 is final: the leaves interchanged the
    // panel's own rows) while the interchanges reach the columns right of it
    bool joined = true;
    if (m2 > 0) {
      rc = emul::aux_ready(h);
      if (!rc) rc = emul::check_cuda(h, cudaEventRecord(h->aux_start, h->stream), "stream events");
      if (!rc) rc = emul::check_cuda(h, cudaStreamWaitEvent(h->aux, h->aux_start, 0), "stream events");
      if (rc) return rc;
      emul::launch_chained(false, emul::trtri_cols_kernel<true>, dim3(jb), dim3(emul::trtri_threads(jb)), 0, h->aux,
                           A, lda, j0, jb, B.inv, nullptr);
      h->launches++;
      rc = emul::check_cuda(h, cudaGetLastError(), "trtri");
      if (!rc) rc = emul::check_cuda(h, cudaEventRecord(h->aux_done, h->aux), "stream events");
      if (rc) return rc;
      joined = false;
    }
    ph = emul::phase_begin(h, EMUL_PHASE_SWAP);
    // the columns right of the panel; the columns left of it get all later
    // interchanges at once, after the loop, from the same maps
    for (int c = 0; c < cpp && !rc; ++c) {
      const int k1 = j0 + c * emul::kPermMax, k2 = k1 + emul::kPermMax < j0 + jb ? k1 + emul::kPermMax : j0 + jb;
      if (k1 >= k2) break;
      int* map = maps + static_cast<size_t>(j0 / nb * cpp + c) * emul::kMapInts;
      rc = emul::laswp_prepare(h, ipiv, k1, k2, map);
      if (!rc) rc = emul::laswp_apply(h, A, lda, j0 + jb, n, map);
    }
    emul::phase_end(h, ph);
    // the stream waits for L11^-1 on every path, so no work of this call is left behind on the second stream
    if (!joined) {
      const int rj = emul::check_cuda(h, cudaStreamWaitEvent(h->stream, h->aux_done, 0), "stream events");
      if (!rc) rc = rj;
    }
    if (rc) return rc;
    if (m2 > 0) {
      ph = emul::phase_begin(h, EMUL_PHASE_U12);
      double* A12 = A + j0 + static_cast<long>(j0 + jb) * lda;
      // U12 = L11^-1 A12 (jb x m2), written over A12
      rc = emul::gemm_run(h, jb, m2, jb, 1.0, Operand{B.inv, 1, jb}, Operand{A12, lda, 1}, 0.0, A12, lda,
                          autos ? s_prev : s_fixed, false, 0, nullptr, 0, 0);
      emul::phase_end(h, ph);
      if (rc) return rc;
      ph = emul::phase_begin(h, EMUL_PHASE_UPDATE);
      const double* L21 = A + (j0 + jb) + static_cast<long>(j0) * lda;
      double* A22 = A + (j0 + jb) + static_cast<long>(j0 + jb) * lda;
      int s_step = slices;
      if (autos) {
        // slice count of this update from the selector, then the probe's "before" sums
        rc = emul::selector_features(h, m2, m2, jb, Operand{L21, 1, lda}, Operand{A12, lda, 1},
                                     emul::selector_feature_buffer(h));
        if (rc) return rc;
        rc = emul::selector_predict(h, 1, emul::selector_feature_buffer(h), emul::selector_pred_buffer(h));
        if (rc) return rc;
        int32_t sp = 8;
        rc = emul::check_cuda(h, cudaMemcpyAsync(&sp, emul::selector_pred_buffer(h), 4, cudaMemcpyDeviceToHost,
                                                 h->stream), "selector read");
        if (rc) return rc;
        rc = emul::check_cuda(h, cudaStreamSynchronize(h->stream), "selector read");
        if (rc) return rc;
        s_step = sp < 3 ? 3 : (sp > 8 ? 8 : sp);
        const int R = m2 < emul::kProbeRows ? m2 : emul::kProbeRows;
        double* y0 = B.probe;
        double* a0 = y0 + emul::kProbeRows;
        double* z = y0 + 4 * emul::kProbeRows;
        double* za = z + nb;
        emul::probe_rows_kernel<<<R, 256, 0, h->stream>>>(m2, m2, A22, lda, R, y0, a0);
        emul::probe_z_kernel<<<jb, 256, 0, h->stream>>>(m2, A12, lda, z, za);
        h->launches += 2;
        cudaMemsetAsync(B.flag, 0, sizeof(int), h->stream);
      }
      // A22 -= L21 U12
      rc = emul::gemm_run(h, m2, m2, jb, -1.0, Operand{L21, 1, lda}, Operand{A12, lda, 1}, 1.0, A22, lda, s_step,
                          false, 0, nullptr, 0, 0);
      if (rc) return rc;
      if (autos) {
        const int R = m2 < emul::kProbeRows ? m2 : emul::kProbeRows;
        double* y0 = B.probe;
        double* a0 = y0 + emul::kProbeRows;
        double* y1 = a0 + emul::kProbeRows;
        double* a1 = y1 + emul::kProbeRows;
        double* z = y0 + 4 * emul::kProbeRows;
        double* za = z + nb;
        emul::probe_rows_kernel<<<R, 256, 0, h->stream>>>(m2, m2, A22, lda, R, y1, a1);
        emul::probe_check_kernel<<<1, 4 * 32, 0, h->stream>>>(m2, m2, jb, L21, lda, R, z, za, y0, a0, y1,
                                                                       a1, B.flag);
        h->launches += 2;
        int fl = 0;
        rc = emul::check_cuda(h, cudaMemcpyAsync(&fl, B.flag, 4, cudaMemcpyDeviceToHost, h->stream), "probe read");
        if (rc) return rc;
        rc = emul::check_cuda(h, cudaStreamSynchronize(h->stream), "probe read");
        if (rc) return rc;
        if (fl && s_step < 8) {
          // undo with the same slice count, redo with 8
          rc = emul::gemm_run(h, m2, m2, jb, 1.0, Operand{L21, 1, lda}, Operand{A12, lda, 1}, 1.0, A22, lda, s_step,
                              false, 0, nullptr, 0, 0);
          if (rc) return rc;
          rc = emul::gemm_run(h, m2, m2, jb, -1.0, Operand{L21, 1, lda}, Operand{A12, lda, 1}, 1.0, A22, lda, 8,
                              false, 0, nullptr, 0, 0);
          if (rc) return rc;
          if (stats) stats->checks_failed++;
          s_step = 8;
        }
        if (stats) {
          stats->slices_min = s_step < stats->slices_min ? s_step : stats->slices_min;
          stats->slices_max = s_step > stats->slices_max ? s_step : stats->slices_max;
        }
      }
      emul::phase_end(h, ph);
      slices_sum += s_step;
      updates++;
      s_prev = s_step;
    }
    if (stats) stats->steps++;
  }
  if (stats) stats->slices_mean = updates ? slices_sum / updates : static_cast<double>(s_fixed);
  // the L columns of every panel but the last: all interchanges of the later
  // panels, composed from the last panel back and gathered once per panel
  const int K = (n + nb - 1) / nb;
  if (K > 1) {
    const int ph = emul::phase_begin(h, EMUL_PHASE_SWAP);
    int* G = reinterpret_cast<int*>(static_cast<uint8_t*>(h->ws) + def_off);
    int* H = G + n;
    double* tmp = reinterpret_cast<double*>(static_cast<uint8_t*>(h->ws) + def_off + emul::al(8ull * n));
    emul::launch_dependent(emul::iota2_kernel, dim3((n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024), dim3(256), 0,
                           h->stream, n, G, H);
    h->launches++;
    for (int k = K - 2; k >= 0; --k) {
      const int r0 = (k + 1) * nb, r1 = r0 + nb < n ? r0 + nb : n;
      // panel k+1's interchanges, composed from its last gather map back
      for (int c = (r1 - r0 - 1) / emul::kPermMax; c >= 0; --c) {
        emul::launch_dependent(emul::compose_kernel, dim3(1), dim3(512), 0, h->stream,
                               maps + static_cast<size_t>((k + 1) * cpp + c) * emul::kMapInts, G, H);
        h->launches++;
      }
      emul::launch_dependent(emul::gather_rows_kernel, dim3((n - r0 + 255) / 256, nb), dim3(256), 0, h->stream, A,
                             lda, r0, n, k * nb, G, tmp);
      h->launches++;
      rc = emul::check_cuda(h,
                            cudaMemcpy2DAsync(A + r0 + static_cast<long>(k) * nb * lda, static_cast<size_t>(lda) * 8,
                                              tmp, static_cast<size_t>(n - r0) * 8, static_cast<size_t>(n - r0) * 8,
                                              nb, cudaMemcpyDeviceToDevice, h->stream),
                            "deferred interchanges");
      if (rc) return rc;
    }
    emul::phase_end(h, ph);
  }
  return EMUL_OK;
}

int emul_dgetrs(emul_handle_t h, int n, int nrhs, const double* LU, int lda, const int32_t* ipiv, double* B,
                int ldb) {
  emul::trsv_attr();
  if (!h) return EMUL_INVALID_ARG;
  if (n < 0 || nrhs < 0 || lda < (n > 1 ? n : 1) || ldb < (n > 1 ? n : 1) || (n > 0 && nrhs > 0 && (!LU || !ipiv || !B)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dgetrs: invalid argument");
  if (n == 0 || nrhs == 0) return EMUL_OK;
  const int ph = emul::phase_begin(h, EMUL_PHASE_SOLVE);
  const int rc = emul::getrs_body(h, n, nrhs, LU, lda, ipiv, B, ldb);
  emul::phase_end(h, ph);
  return rc;
}

int emul_dpotrf(emul_handle_t h, char uplo, int n, double* A, int lda, int nb, int slices, int32_t* info,
                emul_stats* stats) {
  if (!h) return EMUL_INVALID_ARG;
  if (nb == EMUL_NB_AUTO && slices >= 1 && slices <= emul::kMaxSlices && n >= 1) {
    const int rc = emul::resolve_nb(h, 1, n, slices, &nb);
    if (rc) return rc;
  }
  if (nb == EMUL_NB_AUTO && n == 0) nb = 128;
  if (nb == 0) nb = 128;
  if ((uplo != 'L' && uplo != 'l') || n < 0 || lda < (n > 1 ? n : 1) || nb < 16 || nb > 512 || nb % 16 != 0 ||
      slices < 1 || slices > emul::kMaxSlices || (n > 0 && (!A || !info)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dpotrf: invalid argument");
  if (stats) *stats = emul_stats{0, slices, slices, 0, 0.0, static_cast<double>(slices)};
  if (n == 0) return EMUL_OK;
  int rc = emul::check_cuda(h, cudaMemsetAsync(info, 0, sizeof(int32_t), h->stream), "info reset");
  if (rc) return rc;
  const size_t gw = emul::gemm_workspace_bytes(n, n, nb, slices, false);
  rc = emul::reserve_workspace(h, gw + emul::lu_extra_bytes(nb, h->nsm));
  if (rc) return rc;
  const emul::LuBufs B = emul::carve(h, gw, nb);
  bool ahead = false;       // block j0 was factored on the second stream
  for (int j0 = 0; j0 < n && !rc; j0 += nb) {
    const int jb = nb < n - j0 ? nb : n - j0;
    const int m2 = n - j0 - jb;
    if (ahead)
      rc = emul::check_cuda(h, cudaStreamWaitEvent(h->stream, h->aux_done, 0), "stream events");
    else
      rc = emul::chol_diag(h, A, lda, j0, jb, B.inv, info, m2 > 0, h->stream);
    ahead = false;
    if (!rc && m2 > 0) rc = emul::chol_trailing(h, A, lda, j0, jb, m2, nb, slices, info, B, &ahead);
    if (stats) stats->steps++;
  }
  return rc;
}

int emul_dpotrs(emul_handle_t h, char uplo, int n, int nrhs, const double* L, int lda, double* B, int ldb) {
  emul::trsv_attr();
  if (!h) return EMUL_INVALID_ARG;
  if ((uplo != 'L' && uplo != 'l') || n < 0 || nrhs < 0 || lda < (n > 1 ? n : 1) || ldb < (n > 1 ? n : 1) ||
      (n > 0 && nrhs > 0 && (!L || !B)))
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_dpotrs: invalid argument");
  if (n == 0 || nrhs == 0) return EMUL_OK;
  const int ph = emul::phase_begin(h, EMUL_PHASE_SOLVE);
  if (nrhs == 1) {
    // one right-hand side: both substitutions in one cooperative launch
    int rc = emul::reserve_workspace(h, emul::kAl);
    if (rc) return rc;
    unsigned long long* cnt = static_cast<unsigned long long*>(h->ws);
    rc = emul::check_cuda(h, cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), h->stream), "solve barrier");
    if (rc) return rc;
    emul::smem_attr(reinterpret_cast<const void*>(emul::getrs1_kernel<true>),
                    emul::kSolveBs * (emul::kSolveBs + 1) * 8);
    long ldl = lda;
    long long limit = h->wait_limit;
    int* status = h->d_status;
    void* args[] = {const_cast<double**>(&L), &ldl, &n, &B, &cnt, &status, &limit};
    h->launches++;
    rc = emul::check_cuda(h,
                          cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(emul::getrs1_kernel<true>),
                                                      dim3(emul::solve_blocks(h, n)), dim3(256), args,
                                                      emul::kSolveBs * (emul::kSolveBs + 1) * 8, h->stream),
                          "Cholesky solve");
    emul::phase_end(h, ph);
    return rc;
  }
  constexpr int bs = 128;
  for (int d0 = 0; d0 < n; d0 += bs) {
    const int b = bs < n - d0 ? bs : n - d0;
    emul::launch_dependent(emul::trsv_block_kernel, dim3(nrhs), dim3(1024), b * (b + 1) * sizeof(double), h->stream,
                           L, lda, B, ldb, d0, b, 1, 0, 0, d0 > 0);
    h->launches += (d0 + b < n) ? 2 : 1;
    if (d0 + b < n)
      emul::launch_dependent(emul::gemv_update_kernel, dim3((n - d0 - b + 255) / 256, nrhs), dim3(256), 0, h->stream,
                             L, lda, B, ldb, d0 + b, n, d0, b, 0);
  }
  for (int d0 = ((n - 1) / bs) * bs; d0 >= 0; d0 -= bs) {
    const int b = bs < n - d0 ? bs : n - d0;
    emul::launch_dependent(emul::trsv_block_kernel, dim3(nrhs), dim3(1024), b * (b + 1) * sizeof(double), h->stream,
                           L, lda, B, ldb, d0, b, 0, 0, 1, 1);
    h->launches += (d0 > 0) ? 2 : 1;
    if (d0 > 0)
      emul::launch_dependent(emul::gemv_update_kernel, dim3((d0 + 7) / 8, nrhs), dim3(256), 0, h->stream, L, lda, B,
                             ldb, 0, d0, d0, b, 1);
  }
  emul::phase_end(h, ph);
  return emul::check_cuda(h, cudaGetLastError(), "potrs");
}

int emul_backward_error(emul_handle_t h, int n, const double* A, int lda, const double* x, const double* b,
                        double* out) {
  if (!h) return EMUL_INVALID_ARG;
  if (n <= 0 || lda < n || !A || !x || !b || !out)
    return emul::set_error(h, EMUL_INVALID_ARG, "emul_backward_error: invalid argument");
  const size_t need = emul::lu_extra_bytes(16, h->nsm);
  int rc = emul::reserve_workspace(h, need);
  if (rc) return rc;
  const emul::LuBufs B = emul::carve(h, 0, 16);
  rc = emul::check_cuda(h, cudaMemsetAsync(B.racc, 0, 4 * sizeof(unsigned long long), h->stream), "residual reset");
  if (rc) return rc;
  emul::residual_kernel<<<(n + 255) / 256, 256, 2048 * sizeof(double), h->stream>>>(n, A, lda, x, b, B.racc);
  h->launches += 2;
  emul::residual_finish_kernel<<<1, 1, 0, h->stream>>>(n, B.racc, out);
  return emul::check_cuda(h, cudaGetLastError(), "residual");
}

}  // extern "C"
