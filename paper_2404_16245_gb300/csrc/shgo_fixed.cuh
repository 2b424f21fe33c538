// 58-bit fixed-point arithmetic on the integer pipe, for the FP64 path's bulk sums.
//
// GB300 issues 64 integer multiply-adds (32 x 32 + 64 bits) per clock and SM and 1.7 FP64 ones (measured;
// shgo_measure_fma_rate for the latter), so a product of two 58-bit numbers formed from three such multiply-adds
// costs a twelfth of an FP64 one.  Values are scaled by a power of two, common to the entries that are summed together,
// to |v| <= 1, so the largest carry five bits more than an FP64 mantissa and one smaller by 2^-k carries 58 - k bits: sums
// are accurate relative to their scale, not relative to each entry.  A value is held as q = round(v 2^58) = h 2^29 + l with l in [-2^28, 2^28).  A sum of at most 35
// products keeps the partial sums of h h and of h l + l h in one 64-bit accumulator each (32 nuclei, or the 2 Lambda + 1
// terms of a degree, 35 at Lambda = 17); the products l l (at most 2^-60 of a full-scale one) are left out.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace shgo {
namespace {

constexpr int kFxLimb = 29;
constexpr int kFxBits = 2 * kFxLimb;

struct fx {
  int h, l;
};

__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

__device__ __forceinline__ fx fx_split(long long q) {
  const int l = ((int)q << (32 - kFxLimb)) >> (32 - kFxLimb);
  return {(int)((q - l) >> kFxLimb), l};
}

__device__ __forceinline__ fx fx_neg(fx a) { return {-a.h, -a.l}; }

// Rounded value of the accumulators of sum h h and sum h l + l h, in units of 2^-58 (times the operands' scales).
__device__ __forceinline__ long long fx_sum(long long hh, long long mid) {
  return hh + ((mid + (1ll << (kFxLimb - 1))) >> kFxLimb);
}

// v 2^(1023 - be2) as fixed point, |v| 2^(1023 - be2) <= 1; zero and subnormal v give 0.
__device__ __forceinline__ fx fx_of(double v, int be2) {
  const int hi = __double2hiint(v);
  const int e = (hi >> 20) & 0x7ff;
  if (e == 0) return {0, 0};
  const int sh = min(max(be2 - e, 0), 63);
  const unsigned long long m =
      ((unsigned long long)((unsigned)(hi & 0xfffff) | 0x100000u) << 32) | (unsigned)__double2loint(v);
  // m = |v| 2^(1075 - e): shift to units of 2^-58 with one bit more, round it off
  long long q = (long long)(((m << (kFxBits - 52 + 1)) >> sh) + 1) >> 1;
  if (hi < 0) q = -q;
  return fx_split(q);
}

// t 2^e as a double (round to nearest; 0 below the normal range, infinity above it).
__device__ __forceinline__ double fx_double(long long t, int e) {
  if (t == 0) return 0.0;
  unsigned long long a = t < 0 ? 0ull - (unsigned long long)t : (unsigned long long)t;
  const int lz = __clzll((long long)a);
  a <<= lz;
  const int b = e + 63 - lz + 1023;  // biased exponent
  const unsigned long long r = (a >> 11) + ((a >> 10) & 1ull);  // 53 bits, or 2^53 after rounding up
  long long bits = (long long)(((unsigned long long)(unsigned)(b - 1) << 52) + r);
  if (b <= 0) bits = 0;
  if (b >= 0x7ff) bits = 0x7ffll << 52;
  return __longlong_as_double(bits | (t < 0 ? (long long)0x8000000000000000ull : 0ll));
}

}  // namespace
}  // namespace shgo
