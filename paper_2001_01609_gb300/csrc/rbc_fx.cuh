// 64-bit fixed-point arithmetic for the FP64 mode's transforms.
//
// sm_103a issues 2 FP64 operations per clock and SM, but 32 32x32->64-bit
// multiply-adds (mad.wide) and about 60 64-bit additions (measured: 152 SMs,
// 512-thread blocks).  The transforms of the FP64 mode (z transforms, x FFTs,
// products) therefore run in block fixed point: the values of one row or
// column share an exponent and are held as integers of 56 to 62 bits, more
// than the 53 bits of a double relative to the largest values of that row or
// column; additions are exact, products drop terms below 2^-60 of their
// bound.  The stage solves, whose systems are ill conditioned, stay in FP64.
// Integer sums do not depend on their order, so the split of a sum over
// threads and warps never changes a bit.
#pragma once
#include <cuda_runtime.h>
#include <cstdint>

namespace rbc {
namespace fx {

using i64 = long long;

// High word of a double: sign, 11 exponent bits, 20 mantissa bits.
__device__ __forceinline__ int hi_abs(double v) { return __double2hiint(v) & 0x7fffffff; }
__device__ __forceinline__ int biased_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v 2^(BITS - E) truncated to an integer, for |v| < 2^E and finite v; ebias = E + 1022.
// A double below 2^-1022 counts as zero.
template <int BITS>
__device__ __forceinline__ i64 from_double(double v, int ebias) {
  const int hi = __double2hiint(v);
  const unsigned lo = (unsigned)__double2loint(v);
  const int e = (hi >> 20) & 0x7ff;
  const unsigned mh = (unsigned)(hi & 0xfffff) | (e ? 0x100000u : 0u);
  unsigned long long m = ((unsigned long long)mh << 32) | (e ? lo : 0u);   // 53-bit mantissa
  const int s = min(max(ebias - e, 0), 63);
  m = (m << (BITS - 53)) >> s;
  const i64 sg = (i64)(hi >> 31);
  return ((i64)m ^ sg) - sg;
}

// 2^e as a double, e clamped to the normal range's ends (0 below, infinity above).
__device__ __forceinline__ double pow2(int e) {
  return e > 1023 ? __hiloint2double(0x7ff00000, 0) : e < -1022 ? 0.0 : __hiloint2double((e + 1023) << 20, 0);
}

// v 2^e rounded to nearest even, for a result in the normal range or zero
// (others: the FP64 instructions).  About 20 integer instructions; a conversion
// and a multiplication hold the sub-partition's FP64 pipe for 64 clocks each.
__device__ __forceinline__ double to_double(i64 v, int e) {
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);
  const int be = 1023 + 63 - lz + e;          // of a value in [2^(63 - lz + e), 2^(64 - lz + e))
  const unsigned long long q = m >> 11;
  const unsigned up = (((unsigned)m & 0x7ffu) + 0x3ffu + ((unsigned)q & 1u)) >> 11;
  unsigned long long r = ((unsigned long long)(unsigned)(be - 1) << 52) + q + up;   // q holds the leading 1
  if (a == 0) r = 0;
  else if ((unsigned)(be - 1) >= 2045u) return (double)v * pow2(e);
  return __longlong_as_double((long long)(r | (v < 0 ? 0x8000000000000000ull : 0ull)));
}

// a = h 2^32 + l, -2^31 <= l < 2^31.
__device__ __forceinline__ void split32(i64 a, int& h, int& l) {
  l = (int)a;
  h = (int)(a >> 32) + (int)((unsigned)l >> 31);
}

__device__ __forceinline__ i64 madw(int a, int b, i64 c) { return (i64)a * b + c; }

}  // namespace fx
}  // namespace rbc
