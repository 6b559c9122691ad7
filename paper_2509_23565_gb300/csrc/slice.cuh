// Scale and slice arithmetic of an operand (arXiv 2509.23565, Section 2, Eq.
// 1-4) on the IEEE-754 bit fields, shared by the slicing kernels and the small
// product: per row, e = smallest exponent with max |x| < 2^e, N = trunc(|x|
// 2^(7s - e)) and its s digits of 7 bits, carried with x's sign as BF16.
#pragma once
#include <cstdint>

#include "emul_internal.h"

namespace emul {

__device__ __forceinline__ int exponent_of_maxbits(uint64_t u) {
  if (u >= 0x7FF0000000000000ull) return kNonFinite;
  if (u == 0) return 0;
  const int E = static_cast<int>(u >> 52);
  if (E > 0) return E - 1022;                      // |x| in [2^(E-1023), 2^(E-1022))
  return -1010 - __clzll(static_cast<long long>(u));  // subnormal: |x| = u * 2^-1074
}

// |N| = trunc(|x| 2^(7S - e)) for |x| < 2^e; u = x's bit pattern.  With 53
// significant bits the shift is to the right for S <= 7 (by 53 - 7S or more) and
// to the left by at most 3 for S = 8; a shift past the word gives 0.  Only a row
// of subnormals shifts further left.
template <int S>
__device__ __forceinline__ uint64_t scaled_magnitude(uint64_t u, int e) {
  const uint32_t hi = static_cast<uint32_t>(u >> 32);
  const int E = static_cast<int>((hi >> 20) & 0x7FFu);
  const uint32_t mhi = (hi & 0xFFFFFu) | (E ? 0x100000u : 0u);
  uint64_t M = (static_cast<uint64_t>(mhi) << 32) | static_cast<uint32_t>(u);
  constexpr int kUp = S == 8 ? 3 : 0;
  M <<= kUp;
  const int r = e + (1075 - 7 * S + kUp) - (E > 1 ? E : 1);   // x = M 2^(max(E,1) - 1075 - kUp)
  if (r < 0) return M << -r;
  return M >> (r < 63 ? r : 63);
}

// The digits of eight elements of one row (u: their bit patterns, e: the row's
// exponent), lowest plane first: put(p, words) receives plane p's eight BF16
// values as four words.  Integer operations run at 64 lanes per clock per SM
// and set the pace, so two neighbouring elements share them: 14-bit pieces (two
// digits) of both magnitudes are put side by side, a digit pair is masked into
// the low bits of two BF16 128.0, where one unit is the last place, and a packed
// FMA takes 128 off and gives it the sign (a zero digit is +0).  About 25
// integer operations per element at s = 7, against about 70 with a table or a
// conversion per digit.
template <int S, typename Put>
__device__ __forceinline__ void slice8(const uint64_t (&u)[8], int e, Put put) {
  const int er = e == kNonFinite ? 4096 : e;     // every digit of such a row is 0
  uint32_t out[S][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint64_t a = scaled_magnitude<S>(u[2 * i], er), b = scaled_magnitude<S>(u[2 * i + 1], er);
    const uint32_t sgn = __byte_perm(static_cast<uint32_t>(u[2 * i] >> 32), static_cast<uint32_t>(u[2 * i + 1] >> 32), 0x7632) &
                         0x80008000u;
    const uint32_t one = sgn ^ 0x3F803F80u, off = sgn ^ 0xC300C300u;   // +-1, -+128
#pragma unroll
    for (int q = 0; q < (S + 1) / 2; ++q) {
      const uint32_t w = __byte_perm(static_cast<uint32_t>(a >> (14 * q)), static_cast<uint32_t>(b >> (14 * q)), 0x5410);
#pragma unroll
      for (int d = 2 * q; d < 2 * q + 2 && d < S; ++d) {
        const uint32_t x = (((d & 1) ? w >> 7 : w) & 0x007F007Fu) | 0x43004300u;
        asm("fma.rn.bf16x2 %0, %1, %2, %3;" : "=r"(out[d][i]) : "r"(x), "r"(one), "r"(off));
      }
    }
  }
#pragma unroll
  for (int d = 0; d < S; ++d) put(S - 1 - d, make_uint4(out[d][0], out[d][1], out[d][2], out[d][3]));
}

// Largest magnitude of eight elements by their upper words (sign taken off).
// A row whose largest one has a zero exponent field is all zeros or subnormals
// and needs the full patterns (max_bits8).
__device__ __forceinline__ uint32_t max_upper8(const uint64_t (&u)[8]) {
  uint32_t m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) m = max(m, static_cast<uint32_t>(u[j] >> 32) & 0x7FFFFFFFu);
  return m;
}
__device__ __forceinline__ uint64_t max_bits8(const uint64_t (&u)[8]) {
  uint64_t m = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const uint64_t v = u[j] & 0x7FFFFFFFFFFFFFFFull;
    m = v > m ? v : m;
  }
  return m;
}
// Exponent from the largest upper word; only valid when needs_full_max is false.
// The word alone tells Inf / NaN (0x7FF in the exponent field) from finite.
__device__ __forceinline__ bool needs_full_max(uint32_t upper) { return upper < 0x00100000u; }
__device__ __forceinline__ int exponent_of_upper(uint32_t upper) {
  return upper >= 0x7FF00000u ? kNonFinite : static_cast<int>(upper >> 20) - 1022;
}

}  // namespace emul
