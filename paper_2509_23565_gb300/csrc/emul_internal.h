// Internal declarations shared by the CUDA sources of the library.
#pragma once
#include <cstdint>
#include <cuda.h>
#include <cuda_runtime.h>

namespace emul {

constexpr int kNonFinite = 2147483647;   // scale of a row / column holding Inf or NaN
constexpr int kMaxSlices = 8;
constexpr int kBK = 32;                  // K elements per staged chunk (64 B of BF16: SWIZZLE_64B)
constexpr int kMaxStagesCfg = 8;         // deepest ring of staged chunks
constexpr int kExactBudget = 1040;       // k * pairs per accumulator: 1040 * 127^2 < 2^24

// One sweep of the product schedule: up to four accumulator jobs over the K
// chunks [k0c, k1c), sharing the staged slice tiles of each chunk.  A job
// sums the slice pairs (p, L-p), p = pb..pe, of one level L into one TMEM slot.
// The epilogue takes the jobs in schedule order and adds each job's sum with
// its weight into the state, R += I 2^(7(t-L)); the job in final_mask (the last
// job of the 64-bit variants) completes T = R + I 2^(7(t-L)), rounds it and
// updates C.
constexpr int kSweepJobs = 4;
// TMEM accumulator slots.  Job j, counted over all tiles of a CTA or CTA pair, takes
// slot j % 4; its barriers' phase is the parity of j / 4.
constexpr int kTmemSlots = 4;
struct Sweep {
  int16_t k0c, k1c;       // chunk range
  int8_t L[kSweepJobs];   // job levels (0: no job)
  uint8_t pp[kSweepJobs]; // pair ranges, pb | pe << 4
  int8_t nplanes;         // slice planes 1..nplanes of A and of B are staged
  int8_t kcs;             // K chunks per stage (kcs * nplanes <= s tiles of A and of B)
  int8_t njobs;
  int8_t final_mask;      // bit j: job j completes and rounds the sum
};
static_assert(sizeof(Sweep) == 16, "a sweep is one 16-byte record");

// Constants that the drains of the 64-bit state leave in it (gemm_kernel.cuh):
// kMagicBits per unit of weight for a job drained alone, kMagicPair for two
// adjacent levels drained together (129 kMagicBits modulo 2^32, signed).
constexpr int kMagicBits = 0x4B400000;
constexpr long long kMagicPair = -348127232;

// Where the low bits are put aside and what the state starts from (GemmArgs).
struct DrainConstants {
  int stash_job;            // job of the tile after which the low bits are put aside (-1: never)
  long long r_init, r_init2;
};

struct GemmArgs {
  int M, N, K;
  int s, t;                 // slices, threshold (t = s + 1)
  double alpha, beta;
  double* C;
  long ldc;
  const int32_t* ea;        // row scales of A   [M]
  const int32_t* fb;        // column scales of B [N]
  const Sweep* sched;       // device array
  int nsweeps;
  int stash_job;            // job of the tile after which the low bits are put aside (STASH variants)
  long long r_init;         // the state's start: minus the drains' constants (64-bit variants, mode 0)
  long long r_init2;        // the same for the jobs after stash_job, in the units of the state then
  int tiles_m, tiles_n, ntiles;
  int lower;                // 1: only entries with row >= col are written
  int tri;                  // 1: tiles enumerated over the lower triangle (square tiles)
  int mode;                 // 0: update C; 1: add level sums into `levels`
  int32_t* levels;
  long ldl, ldl_plane;
  int* status;              // device status word (EMUL_TIMEOUT on a bounded-wait expiry)
  long long wait_limit;     // cycles
};

cudaError_t launch_split(cudaStream_t st, int rows, int k, const double* X, long rs, long cs, int s, int32_t* exps,
                         uint16_t* out, long ldk);

// Both operands of a product in one launch (same k, s and ldk).
cudaError_t launch_split2(cudaStream_t st, int k, int s, long ldk, int rows_a, const double* A, long ars, long acs,
                          int32_t* ea, uint16_t* sa, int rows_b, const double* B, long brs, long bcs, int32_t* fb,
                          uint16_t* sb);

// One-launch product for short K and few tiles (gemm_small.cu).
bool small_product_fits(int m, int n, int k, int s, int nsm);
cudaError_t launch_small_product(cudaStream_t st, int m, int n, int k, double alpha, const double* A, long ars,
                                 long acs, const double* B, long brs, long bcs, double beta, double* C, long ldc,
                                 int s, int* status, long long wait_limit);

// The product kernel's variants.  kWide: 64-column tiles, 128-bit state, one CTA
// per tile.  kNarrow: 128-column tiles, 64-bit state, one CTA per tile.  kPair:
// clusters of two CTAs, tiles of 256 rows (args.tiles_m counts them) x bn
// columns (tmB stages bn / 2 rows per CTA, grid even), 64-bit state, with the
// 16 low bits of the sum put aside in shared memory if `stash`.
enum class Variant { kWide, kNarrow, kPair };
struct GemmConfig {
  Variant var;
  int bn;                   // tile columns: 64 (kWide), 128 (kNarrow), 128 or 64 (kPair)
  bool stash;               // kPair only
};

cudaError_t launch_gemm(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                        const GemmArgs& args, int grid, int stages, size_t smem_bytes);
// The update modes of C, each compiled in a source file of its own.
cudaError_t launch_gemm_sub(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                            const GemmArgs& args, int grid, int stages, size_t smem_bytes);
cudaError_t launch_gemm_set(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA, const CUtensorMap& tmB,
                            const GemmArgs& args, int grid, int stages, size_t smem_bytes);
cudaError_t launch_gemm_general(cudaStream_t st, const GemmConfig& cfg, const CUtensorMap& tmA,
                                const CUtensorMap& tmB, const GemmArgs& args, int grid, int stages,
                                size_t smem_bytes);
// Ring stages of a launch and its shared-memory bytes.
int gemm_stages(const GemmConfig& cfg, int s, size_t* smem_bytes);
// CTA pairs that can be resident at once with this much shared memory.
int gemm_pair_capacity(size_t smem_bytes);

}  // namespace emul
