// Correct rounding of exact integer sums to FP64 with integer operations
// (shared by the product kernels and the selector's label kernel).
#pragma once
#include <cstdint>

namespace emul {

// Correctly rounded double of T * 2^sh (round to nearest even), computed with
// integer operations on the IEEE-754 fields (overflow gives +-inf, results
// below the normal range are rounded as subnormals).
__device__ __noinline__ static double rn_scaled(__int128 T, int sh) {
  if (T == 0) return 0.0;
  const bool neg = T < 0;
  const unsigned __int128 mag = neg ? (unsigned __int128)(-(T + 1)) + 1u : (unsigned __int128)T;
  const uint64_t hi = (uint64_t)(mag >> 64), lo = (uint64_t)mag;
  const int msb = hi ? 127 - __clzll((long long)hi) : 63 - __clzll((long long)lo);
  const int E = msb + sh;
  const uint64_t sign = neg ? 0x8000000000000000ull : 0ull;
  if (E > 1023) return __longlong_as_double((long long)(sign | 0x7FF0000000000000ull));
  const int keep = (E >= -1022) ? msb - 52 : -1074 - sh;   // bit of mag kept as the last mantissa bit
  uint64_t q;
  if (keep <= 0) {
    q = (uint64_t)(mag << (-keep));
  } else {
    if (keep > msb + 1) return __longlong_as_double((long long)sign);   // below half the smallest subnormal
    q = (uint64_t)(mag >> keep);
    const unsigned __int128 rem = mag - ((unsigned __int128)q << keep);
    const unsigned __int128 half = (unsigned __int128)1 << (keep - 1);
    if (rem > half || (rem == half && (q & 1ull))) q += 1;
  }
  const uint64_t bits = (E >= -1022) ? ((uint64_t)(E + 1022) << 52) + q : q;
  return __longlong_as_double((long long)(sign | bits));
}

// RN(x * 2^sh) for a 64-bit integer x, in integer arithmetic only and without
// branches (the lanes of a warp hold unrelated values), valid for
// -1022 <= sh <= 960: every |x| < 2^64 then gives a normal result (or, after a
// carry, the top binade).  |x| is normalised so that its leading one sits at
// bit 63 and its top 53 bits are kept: 0x3FF plus the last kept bit is added,
// which rounds to nearest, ties to even, and a carry out of the word moves into
// the exponent field.
__device__ __forceinline__ double rn_x64(long long x, int sh) {
  const unsigned long long sgn = (unsigned long long)(x >> 63);      // 0 or all ones
  const unsigned long long a = ((unsigned long long)x ^ sgn) - sgn;   // |x|
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);
  const unsigned long long r = m + (0x3FFull + ((m >> 11) & 1ull));
  const unsigned long long q = (r >> 11) + ((unsigned long long)(r < m) << 53);
  const int E = (uint32_t)(m >> 32) ? 63 - lz + sh + 1022 : 0;        // zero stays zero
  return __longlong_as_double((long long)((((unsigned long long)(uint32_t)E << 52) + q) | (sgn << 63)));
}

// RN(T * 2^sh) for T = x 2^16 + low, low the 16 bits put aside before the upper
// levels were added (low >= 0 also for a negative T): the same rounding on the
// magnitude of T, whose low bits enter the normalised word from below and the
// sticky bits; valid for -1022 <= sh <= 944.
__device__ __forceinline__ double rn_x80(long long x, uint32_t low, int sh) {
  const unsigned long long sgn = (unsigned long long)(x >> 63);      // 0 or all ones
  const uint32_t lo = (sgn ? 0u - low : low) & 0xFFFFu;
  unsigned long long a = (unsigned long long)x ^ sgn;                  // |T| >> 16
  if (sgn && low == 0) a += 1ull;
  if (a == 0) return rn_scaled(((__int128)x << 16) + (__int128)low, sh);
  const int lz = __clzll((long long)a);
  const unsigned long long l64 = (unsigned long long)lo << 48;
  const unsigned long long m = (a << lz) | ((l64 >> 1) >> (63 - lz));
  const unsigned long long rest = l64 << lz;
  // a sticky bit in place of the dropped ones: bit 0 lies far below the rounding bit
  const unsigned long long ms = m | (rest ? 1ull : 0ull);
  const unsigned long long r = ms + (0x3FFull + ((ms >> 11) & 1ull));
  const unsigned long long q = (r >> 11) + ((unsigned long long)(r < ms) << 53);
  const int E = 63 - lz + 16 + sh + 1022;
  return __longlong_as_double((long long)((((unsigned long long)(uint32_t)E << 52) + q) | (sgn << 63)));
}

// C <- RN(C + v) as a reduction in L2 (fire and forget: no load of C, no FP64
// instruction on the SM).  The FP64 add of red.global rounds to nearest even;
// each element of C is updated by exactly one thread of one launch.
__device__ __forceinline__ void red_add_f64(double* p, double v) {
  asm volatile("red.global.add.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}

__device__ __forceinline__ double neg_d(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ull);
}

}  // namespace emul
