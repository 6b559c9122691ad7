// Slice-pair products on tcgen05 tensor cores with the fused exact
// recombination and C update (arXiv 2509.23565, Section 2, Eq. 2 with the
// truncation threshold t; Section 4, Eq. 7 when alpha = -1, beta = 1).
//
// For an output tile (128 rows x BN columns) the level sums
//   I_L = sum_{p+q=L} SA_p SB_q^T,  L = 2..t,
// are accumulated in TMEM as FP32.  The slices are integers |S| <= 127 held as
// BF16, so every product and every partial sum is an integer; an accumulator
// never receives more than 1040 * 127^2 < 2^24 in magnitude (the schedule
// splits K where needed), so the FP32 sums are exact.  The epilogue converts
// each drained level sum exactly to an integer and adds it with its weight,
// R += I_L 2^(7(t-L)) (int64, or 128-bit for the wide variant), so the levels
// may be drained in any order; the schedule issues the longest jobs (the
// highest levels) first and level 2 last.  The exact value
// T = sum_L I_L 2^(7(t-L)) is rounded once to FP64,
//   D = RN(T * 2^(e_i + f_j - 7t)),
// in integer arithmetic, and C = RN(RN(alpha D) + RN(beta C))
// is written straight back.  For the Schur update (alpha = -1, beta = 1) the
// epilogue does not read C: it issues red.global.add.f64 of -D, an FP64 add
// rounded to nearest that L2 performs, so the C update costs no load latency
// and no FP64 instruction on the SM (GB300 retires ~1.6 per clock per SM).
//
// Warp roles (640 threads): warp 0 issues TMA loads of the slice tiles of each
// K chunk into a ring of shared-memory stages; warp 1 owns TMEM (4 accumulator
// slots); warps 1 and 2 issue the MMAs, every other job of a sweep each; these
// loops run
// on the whole warp (warp-uniform operands, one elected lane issues: a lone
// thread recomputing descriptors issues an MMA only every ~84 cycles, short of
// the 64 a 128 x 128 x 16 MMA takes); warps 4-19 drain the slots and write C.  The
// first warpgroup gives registers to the epilogue warpgroups (setmaxnreg).  A sweep
// of one to four jobs shares the staged tiles of a chunk; the jobs take the
// four TMEM slots in turn (they are drained in order, so the next slot is always
// the one drained first), and the issuers fill slots while the epilogue drains
// others.  All waits are bounded.
//
// With more than 128 rows the blocks run as CTA pairs (clusters of two,
// cta_group::2, the PAIR instantiation): a pair owns a 256 x BN tile, each CTA
// stages its 128 rows of A and half of B's rows, rank 0 issues M = 256 MMAs
// that read both CTAs' tiles, and its commits reach the barriers of both; each
// CTA drains its own TMEM.  Each SM then stages a quarter fewer bytes.
#pragma once
#include <atomic>
#include <cstdint>
#include <type_traits>

#include "emul_internal.h"
#include "launch.h"
#include "ptx.cuh"
#include "round.cuh"

namespace emul {

namespace {

constexpr int kThreads = 640;          // 5 warpgroups: producer/MMA, 4 x epilogue
constexpr int kMmaWarps = 2;           // warps 1 .. kMmaWarps issue MMAs
constexpr int kLaunchRegs = 96;         // 640 x 96 = 61440 registers at launch
constexpr int kLowRegs = 32;            // producer warpgroup after setmaxnreg.dec
constexpr int kHighRegs = 112;          // epilogue warpgroups: 128*32 + 512*112 = 61440
constexpr int kSlots = kTmemSlots;
constexpr int kEpiWarps = 16;
constexpr int kStashBits = 16;         // low bits of the exact sum put aside (STASH)
constexpr int kSchedSmem = 64;
constexpr int kMaxStages = kMaxStagesCfg;
constexpr uint32_t kRowBytes = kBK * 2;     // one K-major row of a staged tile
static_assert(kBK == 32, "mma_bf16_k32_elect issues one staged chunk");
constexpr uint32_t kSwizzleCode = kRowBytes == 64 ? 4u : 6u;   // descriptor code of SWIZZLE_64B / _32B
constexpr int kStatusTimeout = -4;

template <bool WIDE, int BN_>
struct Cfg {
  static constexpr int BM = 128;
  static constexpr int BN = BN_;
  static constexpr int CPT = BN / 4;                  // columns per epilogue thread
  static constexpr uint32_t A_TILE = BM * kBK * 2;    // bytes
  static constexpr uint32_t B_TILE = BN * kBK * 2;
  static constexpr uint32_t TMEM_COLS = kSlots * BN;
  using State = typename std::conditional<WIDE, __int128, long long>::type;
};

// I 2^w in the state's width (the shift is done unsigned: I may be negative).
template <typename State>
__device__ __forceinline__ State shl_state(int I, int w);
template <>
__device__ __forceinline__ long long shl_state<long long>(int I, int w) {
  return (long long)((unsigned long long)(long long)I << w);
}
template <>
__device__ __forceinline__ __int128 shl_state<__int128>(int I, int w) {
  return (__int128)((unsigned __int128)(__int128)I << w);
}

// Integers from FP32 level sums without the conversion unit.  A sum v is an
// integer below 2^24 in magnitude; below 2^22, v + 1.5 2^23 is exact and its
// bits are 0x4B400000 + v.  F2I runs at 13 lanes per clock per SM, an FP32 add
// at 118 and a 32-bit integer operation at 64 (measured), and a 128 x 128 tile
// converts 16384 values per job, so the drains set the kernel's pace: with F2I and
// one 64-bit shift and add per job the 4096^3 product at s = 7 took 3.56 ms,
// against 2.65 with empty drains.  The constants are not subtracted: the state
// starts from minus their weighted sum (GemmArgs::r_init).  A thread whose
// values reach 2^22 (coherent signs) converts them with F2I and adds the
// constant, so both ways leave the same state.
constexpr float kMagic = 12582912.0f;            // 1.5 2^23
constexpr float kMagicMax = 4194304.0f;          // 2^22
__device__ __forceinline__ int magic_bits(uint32_t r) { return __float_as_int(__uint_as_float(r) + kMagic); }
__device__ __forceinline__ float max_abs8(const uint32_t (&r)[8]) {
  float m = 0.0f;
#pragma unroll
  for (int i = 0; i < 8; ++i) m = fmaxf(m, fabsf(__uint_as_float(r[i])));
  return m;
}
// c 2^w as 64 bits, for a signed c and 0 <= w < 64, in 32-bit halves.
__device__ __forceinline__ unsigned long long shl_bits(int c, int w) {
  const uint32_t lo = w < 32 ? (uint32_t)c << w : 0u;
  const uint32_t hi = w < 32 ? (uint32_t)(c >> (w ? 32 - w : 31)) : (uint32_t)c << (w - 32);
  return ((unsigned long long)hi << 32) | lo;
}
// R += c 2^w for eight signed 32-bit c; from 2^32 on only the upper half changes.
__device__ __forceinline__ void add_shifted(long long* R, const int (&c)[8], int w) {
  if (w < 32) {
    const int up = w ? 32 - w : 31;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      R[i] = (long long)((unsigned long long)R[i] +
                         (((unsigned long long)(uint32_t)(c[i] >> up) << 32) | ((uint32_t)c[i] << w)));
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i)
      R[i] = (long long)((unsigned long long)R[i] + ((unsigned long long)((uint32_t)c[i] << (w - 32)) << 32));
  }
}
__device__ __forceinline__ void add_magic(long long* R, const uint32_t (&r)[8], int w) {
  int c[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) c[i] = magic_bits(r[i]);
  add_shifted(R, c, w);
}
// One job's sums: R += (I + kMagicBits) 2^w.
__device__ __forceinline__ void add_single(long long* R, const uint32_t (&r)[8], int w) {
  if (max_abs8(r) < kMagicMax) {
    add_magic(R, r, w);
  } else {
    int c[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = __float2int_rn(__uint_as_float(r[i])) + kMagicBits;
    add_shifted(R, c, w);
  }
}
// Two jobs' sums, I of weight 2^w and J of weight 2^(w+7): R += (I + 2^7 J +
// kMagicPair) 2^w.  Below 2^22 the 32-bit combination of the two bit patterns
// stays inside int32 with the constant taken modulo 2^32 (-348127232).
__device__ __forceinline__ void add_pair(long long* R, const uint32_t (&r)[8], const uint32_t (&q)[8], int w) {
  if (fmaxf(max_abs8(r), max_abs8(q)) < kMagicMax) {
    int c[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) c[i] = (int)((uint32_t)magic_bits(r[i]) + (uint32_t)magic_bits(q[i]) * 128u);
    add_shifted(R, c, w);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const long long v = (long long)__float2int_rn(__uint_as_float(r[i])) +
                          (long long)__float2int_rn(__uint_as_float(q[i])) * 128 + kMagicPair;
      R[i] = (long long)((unsigned long long)R[i] + ((unsigned long long)v << w));
    }
  }
}

// |I 2^w| <= 2^62 for lim = min(62 - w, 31): I >> lim is 0 or -1 exactly then.
__device__ __forceinline__ bool term_fits(int I, int lim) { return lim >= 31 || (I >> lim) == (I >> 31); }

// D of a 64-bit exact sum x: the branchless path when sh keeps every result
// normal, else the general one.
__device__ __forceinline__ double rn_sum64(long long x, int sh) {
  if (sh >= -1022 && sh <= 960) return rn_x64(x, sh);
  return rn_scaled((__int128)x, sh);
}

__device__ __forceinline__ int f2i(uint32_t r) { return __float2int_rn(__uint_as_float(r)); }

// D = RN(T * 2^(e + f - 7t)) (NaN for a non-finite scale), then
// out = RN(RN(alpha D) + RN(beta C)); alpha = +-1 and beta in {0, 1} skip the
// exact multiplications.
// Update modes of C: kSub: C - D (alpha = -1, beta = 1); kSet: D (alpha = 1,
// beta = 0); kGeneral: RN(RN(alpha D) + RN(beta C)) (beta = 0: RN(alpha D)).
enum UpdMode { kGeneral = 0, kSub = 1, kSet = 2 };

template <int UPD>
__device__ __forceinline__ double apply_update(const GemmArgs& a, double D, double c_old) {
  if (UPD == kSub) return __dadd_rn(c_old, neg_d(D));
  if (UPD == kSet) return D;
  const double ad = __dmul_rn(a.alpha, D);
  if (a.beta == 0.0) return ad;
  return __dadd_rn(ad, __dmul_rn(a.beta, c_old));
}

__device__ __forceinline__ void tile_coords(const GemmArgs& a, int tile, int& tm, int& tn) {
  if (a.tri) {
    // lower-triangular enumeration of square tiles: tile = tm(tm+1)/2 + tn, tn <= tm
    int r = (int)((sqrtf(8.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
    while ((long)r * (r + 1) / 2 > tile) --r;
    while ((long)(r + 1) * (r + 2) / 2 <= tile) ++r;
    tm = r;
    tn = tile - r * (r + 1) / 2;
  } else {
    tm = tile % a.tiles_m;
    tn = tile / a.tiles_m;
  }
}

// Tiles of a CTA pair: 256 rows (128 per CTA) x BN columns; tiles_m counts
// 256-row tiles.  The lower-triangular enumeration keeps the tiles that reach
// the diagonal: row pair r holds min(2r + 2, tiles_n) of them.
__device__ __forceinline__ void tile_coords_pair(const GemmArgs& a, int tile, int& tm, int& tn) {
  if (a.tri) {
    const int full = (a.tiles_m - 1) * a.tiles_m;   // row pairs before the last: r (r + 1) tiles before row pair r
    if (tile >= full) {
      tm = a.tiles_m - 1;
      tn = tile - full;
      return;
    }
    int r = (int)((sqrtf(4.0f * (float)tile + 1.0f) - 1.0f) * 0.5f);
    while ((long)r * (r + 1) > tile) --r;
    while ((long)(r + 1) * (r + 2) <= tile) ++r;
    tm = r;
    tn = tile - r * (r + 1);
  } else {
    tm = tile % a.tiles_m;
    tn = tile / a.tiles_m;
  }
}

__device__ __forceinline__ bool aborted(volatile int* flag) { return *flag != 0; }

// A sweep's 16 bytes as four words: the fields are then taken by shifts (a
// struct indexed by a run-time job number would live in local memory), and a
// whole warp's copy is made uniform by one shuffle per word, so that what is
// derived from it stays in the uniform datapath.
struct SweepWords {
  uint32_t w[4];
  __device__ __forceinline__ SweepWords(const Sweep* p) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
  }
  __device__ __forceinline__ void make_uniform() {
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = __shfl_sync(0xFFFFFFFFu, w[i], 0);
  }
  __device__ __forceinline__ int k0c() const { return (int)(w[0] & 0xFFFFu); }
  __device__ __forceinline__ int k1c() const { return (int)(w[0] >> 16); }
  __device__ __forceinline__ int L(int j) const { return (int)((w[1] >> ((8 * j) & 31)) & 255u); }
  __device__ __forceinline__ int pb(int j) const { return (int)((w[2] >> (8 * j)) & 15u); }
  __device__ __forceinline__ int pe(int j) const { return (int)((w[2] >> (8 * j + 4)) & 15u); }
  __device__ __forceinline__ int nplanes() const { return (int)(w[3] & 255u); }
  __device__ __forceinline__ int kcs() const { return (int)((w[3] >> 8) & 255u); }
  __device__ __forceinline__ int njobs() const { return (int)((w[3] >> 16) & 255u); }
  __device__ __forceinline__ bool fin(int j) const { return (w[3] >> (24 + j)) & 1u; }
};

// Jobs j and j + 1 of a sweep are drained in one step (the host's r_init counts
// on the same rule, drained_constants in api.cu).
__device__ __forceinline__ bool drained_together(const SweepWords& S, int j, int nj) {
  const int d = S.L(j + 1) - S.L(j);
  return j + 1 < nj && (d == 1 || d == -1) && !S.fin(j + 1);
}

// The MMAs of the N slice pairs (p, L-p), p ascending, of one level and one K
// chunk: A tiles step up, B tiles step down.  Unrolled: a loop's counter and
// branches cost the issuing warp as much as the MMA takes when the epilogue
// warps compete for its scheduler.
template <bool PAIR, int N>
__device__ __forceinline__ void issue_pairs(uint32_t dcol, uint32_t da, uint32_t db, uint32_t a_step, uint32_t b_step,
                                            uint32_t hi, uint32_t idesc, uint32_t acc) {
#pragma unroll
  for (int i = 0; i < N; ++i)
    mma_bf16_k32_elect<PAIR>(dcol, da + (uint32_t)i * a_step, db - (uint32_t)i * b_step, hi, idesc, i ? 1u : acc);
}

__device__ __forceinline__ void raise_timeout(const GemmArgs& a, volatile int* flag) {
  atomicExch(a.status, kStatusTimeout);
  *flag = 1;
}

}  // namespace

// PAIR: a cluster of two CTAs per tile of 256 x BN (cta_group::2).  Each
// CTA stages its 128 rows of A and BN/2 rows of B; both CTAs' copies complete
// on rank 0's stage barrier; rank 0's MMA warps issue M = 256 MMAs whose
// commits reach both CTAs; each CTA drains its own TMEM and both release a
// slot on rank 0's barrier.  Rank 1's MMA warps stay idle.
//
// STASH: the 16 lowest bits of the exact sum, final once every level of weight
// below 2^16 has been added (job a.stash_job of the tile), go to shared memory
// and the state continues 16 bits up, so that 64 + 16 bits hold the sums of 8
// slices and of long K in the 128-column tile.
template <bool WIDE, int BN, int UPD, bool PAIR, bool STASH>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const GemmArgs a,
                int stages) {
  static_assert(!(WIDE && (PAIR || STASH)), "the 128-bit state runs one CTA per tile");
  using Cf = Cfg<WIDE, BN>;
  using State = typename Cf::State;
  constexpr uint32_t B_T = PAIR ? Cf::B_TILE / 2 : Cf::B_TILE;   // bytes of one staged B plane
  constexpr int G = PAIR ? 2 : 1;                                  // CTAs per tile
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t stage_full[kMaxStages], stage_empty[kMaxStages];
  __shared__ __align__(8) uint64_t slot_full[kSlots], slot_empty[kSlots], mma_done[kMmaWarps];
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  __shared__ __align__(16) Sweep sched_s[kSchedSmem];   // the schedule, when it is short enough

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int s = a.s;
  const uint32_t stage_bytes = (uint32_t)s * (Cf::A_TILE + B_T);
  volatile int* abortp = &abort_flag;
  const uint32_t rank = PAIR ? cluster_rank() : 0u;
  const int cta0 = (int)blockIdx.x / G, ncta = (int)gridDim.x / G;   // tile loop over CTAs or CTA pairs

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) {
      mbar_init(&stage_full[i], 1);
      mbar_init(&stage_empty[i], kMmaWarps);   // one commit per issuing warp
    }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&slot_full[i], 1);
      mbar_init(&slot_empty[i], G * kEpiWarps);
    }
    for (int i = 0; i < kMmaWarps; ++i) mbar_init(&mma_done[i], 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    if (PAIR)
      tmem_alloc_pair(&tmem_base, Cf::TMEM_COLS);
    else
      tmem_alloc(&tmem_base, Cf::TMEM_COLS);
  }
  grid_wait();
  const bool sched_in_smem = a.nsweeps <= kSchedSmem;
  if (sched_in_smem)
    for (int i = threadIdx.x; i < a.nsweeps; i += blockDim.x) sched_s[i] = a.sched[i];
  const Sweep* sched = sched_in_smem ? sched_s : a.sched;
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();   // barriers of both CTAs initialised before any copy or arrival
  grid_launch();              // with the TMEM in hand (ptx.cuh)
  tc_fence_after();
  const uint32_t tmem = tmem_base;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kLowRegs));
  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    // the whole warp runs the loop (warp-uniform values); one elected lane issues
    if (lane == 0) {
      prefetch_tmap(&tmA);
      prefetch_tmap(&tmB);
    }
    __syncwarp();
    int st = 0, filled = 0;   // ring stage, stages filled so far (up to `stages`)
    uint32_t par = 1;         // parity of stage_empty's phase to wait for
    bool ok = true;
    for (int tile = cta0; tile < a.ntiles && ok; tile += ncta) {
      int tm, tn;
      if (PAIR)
        tile_coords_pair(a, tile, tm, tn);
      else
        tile_coords(a, tile, tm, tn);
      const int m0 = (tm * G + (int)rank) * Cf::BM, n0 = tn * Cf::BN + (int)rank * (Cf::BN / G);
      for (int sw = 0; sw < a.nsweeps && ok; ++sw) {
        SweepWords S(sched + sw);
        S.make_uniform();
        const int np = S.nplanes(), k1c = S.k1c(), kcs = S.kcs();
        for (int kc = S.k0c(); kc < k1c; kc += kcs) {
          const int nu = k1c - kc < kcs ? k1c - kc : kcs;
          if (aborted(abortp) || !mbar_wait_warp(&stage_empty[st], par, a.wait_limit)) {
            if (!aborted(abortp) && lane == 0) raise_timeout(a, abortp);
            ok = false;
            break;
          }
          uint8_t* base = smem + (size_t)st * stage_bytes;
          if (!PAIR) {
            mbar_arrive_expect_tx_elect(&stage_full[st], (uint32_t)(nu * np) * (Cf::A_TILE + B_T));
            for (int u = 0; u < nu; ++u)
              for (int p = 0; p < np; ++p) {
                const int t = u * np + p;
                tma_load_3d_elect(base + t * Cf::A_TILE, &tmA, &stage_full[st], (kc + u) * kBK, m0, p);
                tma_load_3d_elect(base + s * Cf::A_TILE + t * B_T, &tmB, &stage_full[st], (kc + u) * kBK, n0, p);
              }
          } else {
            // rank 0's barrier counts the bytes of both CTAs (a copy of rank 1
            // may land before rank 0 announces them: the phase still waits for
            // rank 0's arrival)
            if (rank == 0)
              mbar_arrive_expect_tx_elect(&stage_full[st], (uint32_t)(G * nu * np) * (Cf::A_TILE + B_T));
            const uint32_t bar0 = mapa_rank(&stage_full[st], 0);
            for (int u = 0; u < nu; ++u)
              for (int p = 0; p < np; ++p) {
                const int t = u * np + p;
                tma_load_3d_pair_elect(base + t * Cf::A_TILE, &tmA, bar0, (kc + u) * kBK, m0, p);
                tma_load_3d_pair_elect(base + s * Cf::A_TILE + t * B_T, &tmB, bar0, (kc + u) * kBK, n0, p);
              }
          }
          if (filled < stages) ++filled;
          if (++st == stages) {
            st = 0;
            par ^= 1u;
          }
        }
      }
    }
    if (!ok && rank == 0) {
      // wait (bounded) for the copies still in flight before the block exits
      // (a pair's copies all complete on rank 0's barriers)
      for (int j = 0; j < filled; ++j) {
        // stages before st were filled in the current turn of the ring, the others in the last one
        const uint32_t fpar = j < st ? par ^ 1u : par;
        mbar_wait(&stage_full[j], fpar, a.wait_limit / 8);
      }
    }
  } else if (warp <= kMmaWarps && rank == 0) {
    // ------------------------------------------------------------ MMA issuers
    // the whole warp runs the loop (warp-uniform values); one elected lane
    // issues.  Within a stage the jobs of the sweep are issued one after
    // another in the order the epilogue drains them: a job's slot is waited
    // for only before its own first MMA and committed right after its last,
    // so with all four slots in one sweep the drain of a job overlaps the MMAs
    // of the others (28.7K cycles of MMAs per 256 x 128 tile at k = 256, s = 7).
    constexpr uint32_t idesc = idesc_bf16_f32(128 * G, Cf::BN);
    const int w0 = warp - 1;
    const uint32_t tmem_u = __shfl_sync(0xFFFFFFFFu, tmem, 0);
    const uint32_t smem_base = smem_u32(smem);
    uint32_t job0 = 0;      // job number of the sweep's first job, counted over all tiles
    int st = 0;             // ring stage and the parity of stage_full's phase
    uint32_t par = 0;
    bool ok = true;
    for (int tile = cta0; tile < a.ntiles && ok; tile += ncta) {
      for (int sw = 0; sw < a.nsweeps && ok; ++sw) {
        SweepWords S(sched + sw);
        S.make_uniform();
        const int nj = S.njobs(), np = S.nplanes(), k0c = S.k0c(), k1c = S.k1c(), kcs = S.kcs();
        for (int kc = k0c; kc < k1c && ok; kc += kcs) {
          const int nu = k1c - kc < kcs ? k1c - kc : kcs;
          const bool first = kc == k0c, last = kc + kcs >= k1c;
          if (aborted(abortp) || !mbar_wait_warp(&stage_full[st], par, a.wait_limit)) {
            if (!aborted(abortp) && lane == 0) raise_timeout(a, abortp);
            ok = false;
            break;
          }
          tc_fence_after();
          // descriptors of the stage's first A and B tiles; a tile further is a
          // plain add on the start-address field (addr >> 4, 14 bits, no carry:
          // shared memory addresses stay below 256 KB)
          const uint32_t base = smem_base + (uint32_t)st * stage_bytes;
          const uint64_t dA0 = umma_desc(base, kRowBytes, kSwizzleCode);
          const uint64_t dB0 = umma_desc(base + (uint32_t)s * Cf::A_TILE, kRowBytes, kSwizzleCode);
          const uint32_t hi = (uint32_t)(dA0 >> 32);   // the same for every tile
          for (int j = w0; j < nj; j += kMmaWarps) {
            const uint32_t job = job0 + (uint32_t)j;
            const int slot = (int)(job % kSlots);
            const uint32_t dcol = tmem_u + (uint32_t)(slot * Cf::BN);
            if (first) {
              const uint32_t spar = ((job / kSlots) & 1u) ^ 1u;
              if (aborted(abortp) || !(PAIR ? mbar_wait_cluster_warp(&slot_empty[slot], spar, a.wait_limit)
                                            : mbar_wait_warp(&slot_empty[slot], spar, a.wait_limit))) {
                if (!aborted(abortp) && lane == 0) raise_timeout(a, abortp);
                ok = false;
                break;
              }
              tc_fence_after();
            }
            const int pb = S.pb(j), n = S.pe(j) - pb + 1, q0 = S.L(j) - pb;
            uint32_t acc = first ? 0u : 1u;
            for (int u = 0; u < nu; ++u) {
              const uint32_t da = (uint32_t)dA0 + (uint32_t)((u * np + pb - 1) * (int)(Cf::A_TILE >> 4));
              const uint32_t db = (uint32_t)dB0 + (uint32_t)((u * np + q0 - 1) * (int)(B_T >> 4));
              switch (n) {
#define EMUL_PAIRS(N)                                                                                             \
  case N:                                                                                                         \
    issue_pairs<PAIR, N>(dcol, da, db, Cf::A_TILE >> 4, B_T >> 4, hi, idesc, acc);                                \
    break;
                EMUL_PAIRS(1) EMUL_PAIRS(2) EMUL_PAIRS(3) EMUL_PAIRS(4)
                EMUL_PAIRS(5) EMUL_PAIRS(6) EMUL_PAIRS(7) EMUL_PAIRS(8)
#undef EMUL_PAIRS
              }
              acc = 1u;
            }
            if (last) {
              if (PAIR)
                mma_commit_pair_both_elect(&slot_full[slot]);
              else
                mma_commit_elect(&slot_full[slot]);
            }
          }
          if (!ok) break;
          if (PAIR)
            mma_commit_pair_both_elect(&stage_empty[st]);
          else
            mma_commit_elect(&stage_empty[st]);
          if (++st == stages) {
            st = 0;
            par ^= 1u;
          }
        }
        job0 += (uint32_t)nj;
      }
    }
    // every MMA issued must be complete before TMEM is released
    if (PAIR)
      mma_commit_pair_both_elect(&mma_done[w0]);
    else
      mma_commit_elect(&mma_done[w0]);
    mbar_wait(&mma_done[w0], 0, a.wait_limit);
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kHighRegs));
    // ------------------------------------------------------------ epilogue
    const int ew = warp - 4;
    const int quarter = warp & 3;      // TMEM lane quarter this warp may access
    const int half = ew >> 2;          // column group of CPT columns
    const int row_t = quarter * 32 + lane;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    constexpr int CPT = Cf::CPT;
    const bool needs_c = (UPD == kSub) || (UPD == kGeneral && a.beta != 0.0);
    const int sh0 = -7 * a.t;
    State R[CPT];
    // this thread's low bits, two columns per word
    uint32_t* stash = reinterpret_cast<uint32_t*>(smem + (size_t)stages * stage_bytes) + (threadIdx.x - 128);
    auto low_bits = [&](int c) -> uint32_t {
      const uint32_t w = stash[(c >> 1) * (kEpiWarps * 32)];
      return c & 1 ? w >> 16 : w & 0xFFFFu;
    };
    // D of the exact sum; `normal`: -1022 <= sh <= 944 is known
    auto round_sum = [&](int c, int sh, bool normal) -> double {
      if constexpr (STASH) {
        const uint32_t low = low_bits(c);
        if (!normal && (sh < -1022 || sh > 944)) return rn_scaled(((__int128)R[c] << kStashBits) + (__int128)low, sh);
        return rn_x80((long long)R[c], low, sh);
      } else {
        return normal ? rn_x64((long long)R[c], sh) : rn_sum64((long long)R[c], sh);
      }
    };
    uint32_t job = 0;      // counted over all tiles: slot job % 4, parity of its use
    bool ok = true;
    // rank 0's slot barriers, where both CTAs of a pair release a slot
    uint32_t slot_empty0 = 0;
    if (PAIR) slot_empty0 = mapa_rank(&slot_empty[0], 0);
    auto release = [&](uint32_t slot) {
      if (PAIR)
        mbar_arrive_cluster(slot_empty0 + slot * 8u);
      else
        mbar_arrive_relaxed(&slot_empty[slot]);
    };
    // wait until job n is complete in its slot; its TMEM address for this thread
    auto wait_job = [&](uint32_t n) -> uint32_t {
      const uint32_t slot = n % kSlots;
      if (aborted(abortp) || !mbar_wait(&slot_full[slot], (n / kSlots) & 1u, a.wait_limit)) {
        if (!aborted(abortp)) raise_timeout(a, abortp);
        ok = false;
      }
      return tmem + lane_addr + slot * (uint32_t)Cf::BN + (uint32_t)(half * CPT);
    };
    for (int tile = cta0; tile < a.ntiles && ok; tile += ncta) {
      int tm, tn;
      if (PAIR)
        tile_coords_pair(a, tile, tm, tn);
      else
        tile_coords(a, tile, tm, tn);
      const int row = (tm * G + (int)rank) * Cf::BM + row_t;
      const int col0 = tn * Cf::BN + half * CPT;
      const int e_row = row < a.M ? a.ea[row] : 0;
      // column scales of this thread's CPT columns, one per lane (broadcast by shuffle)
      int fcol[1];
      {
        const int col = col0 + lane;
        fcol[0] = (lane < CPT && col < a.N) ? a.fb[col] : 0;
      }
#pragma unroll
      for (int c = 0; c < CPT; ++c) R[c] = WIDE ? (State)0 : (State)a.r_init;
      int jj = 0;            // job of the tile
      bool final_done = false;
      for (int sw = 0; sw < a.nsweeps && ok; ++sw) {
        const SweepWords S(sched + sw);
        const int nj = S.njobs();
        for (int j = 0; j < nj && ok;) {
          const bool fin = S.fin(j);
          const uint32_t ta = wait_job(job);
          if (!ok) break;
          bool released = false;   // slot already released (final step, 64-bit path)
          int taken = 1;           // jobs drained by this step
          // weight of the level, 2^(7(t-L)), in units of the state
          const int wsh = 7 * (a.t - S.L(j)) - (STASH && jj > a.stash_job ? kStashBits : 0);
          if (a.mode == 1) {
            tc_fence_after();
            // level sums out (exact int32), added so that K segments / pair groups accumulate
            const int L = S.L(j);
#pragma unroll
            for (int c16 = 0; c16 < CPT / 16; ++c16) {
              uint32_t r[16];
              tmem_ld16(ta + c16 * 16, r);
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 16; ++q) {
                const int col = col0 + c16 * 16 + q;
                if (row < a.M && col < a.N) {
                  int32_t* lp = a.levels + (long)(L - 2) * a.ldl_plane + row + (long)col * a.ldl;
                  *lp += f2i(r[q]);
                }
              }
            }
          } else if (WIDE) {
            tc_fence_after();
#pragma unroll
            for (int c16 = 0; c16 < CPT / 16; ++c16) {
              uint32_t r[16];
              tmem_ld16(ta + c16 * 16, r);
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 16; ++q) R[c16 * 16 + q] += shl_state<State>(f2i(r[q]), wsh);
            }
          } else if (!fin) {
            // a job and the next one of the sweep, when their levels are adjacent,
            // are drained together: I_L + 2^7 I_(L-1) fits in 32 bits, so
            // the two share one 64-bit addition
            if constexpr (!WIDE) {
              if (drained_together(S, j, nj)) {
                const uint32_t tb = wait_job(job + 1);
                if (!ok) break;
                tc_fence_after();
                taken = 2;
                const bool up = S.L(j + 1) > S.L(j);   // the second job has the smaller weight
                const uint32_t t0 = up ? tb : ta, t1 = up ? ta : tb;
                const int w0 = up ? wsh - 7 : wsh;
#pragma unroll
                for (int c8 = 0; c8 < CPT / 8; ++c8) {
                  uint32_t r[8], q[8];
                  tmem_ld8(t0 + c8 * 8, r);
                  tmem_ld8(t1 + c8 * 8, q);
                  tmem_ld_wait();
                  add_pair(R + c8 * 8, r, q, w0);
                }
              } else {
                tc_fence_after();
#pragma unroll
                for (int c8 = 0; c8 < CPT / 8; ++c8) {
                  uint32_t r[8];
                  tmem_ld8(ta + c8 * 8, r);
                  tmem_ld_wait();
                  add_single(R + c8 * 8, r, wsh);
                }
              }
            }
          } else {
            // final step (64-bit variants): T = R + I 2^wsh, rounded once, C
            // updated in place.  R, the other levels, stays below 2^61, so T
            // fits in 64 bits when |I| 2^wsh <= 2^62.  When that holds for the
            // whole warp (it fails only for rows and columns whose leading
            // digits are near 127 of one sign along the whole K) the term is
            // added at once, the slot is released and the rounding runs while
            // the MMAs of the next tile fill it; otherwise the slot is held,
            // and the elements over the limit re-read I and round T from 128 bits.
            if constexpr (!WIDE) {
              tc_fence_after();
              final_done = true;
              const bool rowok = row < a.M;
              const int lim = 62 - wsh < 31 ? 62 - wsh : 31;
              float mx = 0.0f;
#pragma unroll
              for (int c8 = 0; c8 < CPT / 8; ++c8) {
                uint32_t r[8];
                tmem_ld8(ta + c8 * 8, r);
                tmem_ld_wait();
                mx = fmaxf(mx, max_abs8(r));
                add_magic(R + c8 * 8, r, wsh);
              }
              // exact below 2^22 in magnitude; the term fits below 2^lim
              bool fits = __all_sync(0xFFFFFFFFu, mx < kMagicMax && mx < __int_as_float((127 + lim) << 23));
              if (fits) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) release(job % kSlots);
                released = true;
              } else {
                // take the additions back and repeat them on exact integers
                fits = true;
#pragma unroll
                for (int c8 = 0; c8 < CPT / 8; ++c8) {
                  uint32_t r[8];
                  tmem_ld8(ta + c8 * 8, r);
                  tmem_ld_wait();
#pragma unroll
                  for (int q = 0; q < 8; ++q) {
                    State& x = R[c8 * 8 + q];
                    const int I = f2i(r[q]);
                    x = (State)((unsigned long long)x - shl_bits(magic_bits(r[q]), wsh) + shl_bits(kMagicBits, wsh));
                    if (term_fits(I, lim))
                      x += shl_state<State>(I, wsh);
                    else
                      fits = false;
                  }
                }
                fits = __all_sync(0xFFFFFFFFu, fits);
                if (fits) {
                  tc_fence_before();
                  __syncwarp();
                  if (lane == 0) release(job % kSlots);
                  released = true;
                }
              }
              double* cp = a.C + row + (long)col0 * a.ldc;
              // a warp whose rows and columns are all inside C (no triangle), with
              // finite scales that keep every result normal, rounds without
              // per-element checks; scales outside +-2000 fail the test of the
              // sums below without overflowing them
              const int f_first = __shfl_sync(0xFFFFFFFFu, fcol[0], 0);
              const int f_any = lane < CPT ? fcol[0] : f_first;
              const int fmin = max(__reduce_min_sync(0xFFFFFFFFu, f_any), -4000);
              const int fmax_ = min(__reduce_max_sync(0xFFFFFFFFu, f_any), 4000);
              const int er = max(min(e_row, 4000), -4000);
              const bool interior =
                  fits && col0 + CPT <= a.N && !a.lower &&
                  __all_sync(0xFFFFFFFFu, rowok && er + fmin + sh0 >= -1022 && er + fmax_ + sh0 <= 944);
              if (interior) {
#pragma unroll
                for (int c = 0; c < CPT; ++c, cp += a.ldc) {
                  const int f = __shfl_sync(0xFFFFFFFFu, fcol[0], c);
                  const double D = round_sum(c, e_row + f + sh0, true);
                  if (UPD == kSub)
                    red_add_f64(cp, neg_d(D));
                  else if (UPD == kSet)
                    *cp = D;
                  else
                    *cp = apply_update<UPD>(a, D, needs_c ? *cp : 0.0);
                }
              } else
#pragma unroll
              for (int c4 = 0; c4 < CPT / 4; ++c4) {
                uint32_t r[4] = {0u, 0u, 0u, 0u};
                if (!fits) {            // warp-uniform
                  tmem_ld4(ta + c4 * 4, r);
                  tmem_ld_wait();
                }
#pragma unroll
                for (int q = 0; q < 4; ++q, cp += a.ldc) {
                  const int c = c4 * 4 + q;
                  const int col = col0 + c;
                  const int f = __shfl_sync(0xFFFFFFFFu, fcol[0], c);
                  if (!rowok || col >= a.N || (a.lower && row < col)) continue;
                  const int I = f2i(r[q]);
                  const int sh = e_row + f + sh0;
                  double D;
                  if (e_row == kNonFinite || f == kNonFinite)
                    D = __longlong_as_double(0x7FF8000000000000ll);
                  else if (fits || term_fits(I, lim))
                    D = round_sum(c, sh, false);
                  else if (STASH)
                    D = rn_scaled((((__int128)R[c] + shl_state<__int128>(I, wsh)) << kStashBits) + low_bits(c), sh);
                  else
                    D = rn_scaled((__int128)R[c] + shl_state<__int128>(I, wsh), sh);
                  if (UPD == kSub)
                    red_add_f64(cp, neg_d(D));
                  else if (UPD == kSet)
                    *cp = D;
                  else
                    *cp = apply_update<UPD>(a, D, needs_c ? *cp : 0.0);
                }
              }
            }
          }
          if (!released) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              release(job % kSlots);
              if (taken == 2) release((job + 1) % kSlots);
            }
          }
          job += (uint32_t)taken;
          jj += taken;
          j += taken;
          if constexpr (STASH) {
            if (jj == a.stash_job + 1) {
#pragma unroll
              for (int c2 = 0; c2 < CPT / 2; ++c2) {
                State& r0 = R[2 * c2];
                State& r1 = R[2 * c2 + 1];
                stash[c2 * (kEpiWarps * 32)] = ((uint32_t)r0 & 0xFFFFu) | ((uint32_t)r1 << 16);
                r0 = (r0 >> kStashBits) + a.r_init2;
                r1 = (r1 >> kStashBits) + a.r_init2;
              }
            }
          }
        }
      }
      if (ok && a.mode == 0 && !final_done) {
        // every level was folded into R (wide variant): T = R
        const bool rowok = row < a.M;
#pragma unroll
        for (int c = 0; c < CPT; ++c) {
          const int col = col0 + c;
          const int f = __shfl_sync(0xFFFFFFFFu, fcol[0], c);
          if (!rowok || col >= a.N || (a.lower && row < col)) continue;
          double D;
          if (e_row == kNonFinite || f == kNonFinite)
            D = __longlong_as_double(0x7FF8000000000000ll);
          else
            D = rn_scaled((__int128)R[c], e_row + f + sh0);
          double* cp = a.C + row + (long)col * a.ldc;
          if (UPD == kSub)
            red_add_f64(cp, neg_d(D));
          else if (UPD == kSet)
            *cp = D;
          else
            *cp = apply_update<UPD>(a, D, needs_c ? *cp : 0.0);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();   // neither CTA leaves while the other may still use its barriers or TMEM
  if (warp == 1) {
    tc_fence_after();
    if (PAIR)
      tmem_dealloc_pair(tmem, Cf::TMEM_COLS);
    else
      tmem_dealloc(tmem, Cf::TMEM_COLS);
  }
}

// Launch of one instantiation.  The kernel's attributes are set once per
// device: the register hand-over between warpgroups is only valid if the block
// is launched with exactly kLaunchRegs registers per thread, and the dynamic
// shared memory limit is raised to the largest any launch takes.
constexpr int kMaxDynSmem = 232448 - 2048;
constexpr int kMaxDevices = 64;
template <bool WIDE, int BN, int UPD, bool PAIR, bool STASH>
cudaError_t launch_one(cudaStream_t st, const CUtensorMap& tmA, const CUtensorMap& tmB, const GemmArgs& args, int grid,
                       int stages, size_t smem_bytes) {
  static std::atomic<bool> ready[kMaxDevices];
  auto kern = gemm_kernel<WIDE, BN, UPD, PAIR, STASH>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= kMaxDevices || !ready[dev].load(std::memory_order_acquire)) {
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, (const void*)kern);
    if (e != cudaSuccess) return e;
    if (fa.numRegs != kLaunchRegs) return cudaErrorInvalidConfiguration;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynSmem);
    if (e != cudaSuccess) return e;
    if (dev < kMaxDevices) ready[dev].store(true, std::memory_order_release);
  }
  if (!PAIR) return launch_dependent(kern, dim3(grid), dim3(kThreads), smem_bytes, st, tmA, tmB, args, stages);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem_bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;   // launch.h
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.numAttrs = 2;
  // the persistent grid holds no more pairs than can be resident at once (an
  // SM left without a partner would otherwise run its pair after the others)
  const int pairs = gemm_pair_capacity(smem_bytes);
  if (pairs < 1) return cudaErrorInvalidConfiguration;
  if (grid > 2 * pairs) cfg.gridDim = dim3(2 * pairs);
  return cudaLaunchKernelEx(&cfg, kern, tmA, tmB, args, stages);
}

template <int UPD>
cudaError_t launch_upd(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                       const GemmArgs& args, int grid, int stages, size_t smem_bytes) {
  if (cfg.var == Variant::kWide) return launch_one<true, 64, UPD, false, false>(st, tmA, tmB, args, grid, stages, smem_bytes);
  if (cfg.var == Variant::kNarrow)
    return launch_one<false, 128, UPD, false, false>(st, tmA, tmB, args, grid, stages, smem_bytes);
  if (cfg.bn == 64)
    return cfg.stash ? launch_one<false, 64, UPD, true, true>(st, tmA, tmB, args, grid, stages, smem_bytes)
                     : launch_one<false, 64, UPD, true, false>(st, tmA, tmB, args, grid, stages, smem_bytes);
  return cfg.stash ? launch_one<false, 128, UPD, true, true>(st, tmA, tmB, args, grid, stages, smem_bytes)
                   : launch_one<false, 128, UPD, true, false>(st, tmA, tmB, args, grid, stages, smem_bytes);
}

}  // namespace emul
