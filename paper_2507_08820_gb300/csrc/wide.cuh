// FP64-accurate arithmetic on the float32 and integer pipes.
//
// A GB300 SM retires about 1.9 FP64 operations per clock, conversions from and to FP64
// included, against 128 float32 and 64 integer ones (measured: chains of dadd, dfma and the
// cvt forms 1.6-2.7 lanes per clock and SM, ffma 107, lop3 62), while HBM delivers a site's 27
// float32 populations every 5 clocks. A kernel that forms its FP64 results with a handful of
// FP64 operations per site is bound by them, not by memory; the routines here replace
// them by exact float32 splits, unevaluated sums of float32 values, and integer packing.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace rflbm_dev {

// s + e = a + b exactly (Knuth).
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return s;
}

// A value as an unevaluated sum hi + lo (about 46 bits; not renormalised, so lo may reach
// a few units in the last place of hi).
struct Pair32 {
  float hi, lo;
};
__device__ __forceinline__ Pair32 padd(Pair32 a, Pair32 b) {
  float e;
  const float s = two_sum(a.hi, b.hi, e);
  return {s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ Pair32 pmul(Pair32 a, Pair32 b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return {p, e};
}

// True when x is zero or 2^-74 <= |x| < 2^top (top <= 128): pair_of splits such x (the low
// part stays normal).
__device__ __forceinline__ bool pair_range(double x, int top) {
  const uint32_t h = (uint32_t)__double2hiint(x) & 0x7fffffffu;
  return (h >= (1023u - 74u) << 20 && h < (uint32_t)(1023 + top) << 20) || (h | (uint32_t)__double2loint(x)) == 0u;
}
// x = hi + lo + rest, |rest| <= 2^-48 |x|: hi takes the top 24 bits, lo the other 29 rounded to
// 24, both by moving bits (pair_range(x)).
__device__ __forceinline__ Pair32 pair_of(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t sign = h & 0x80000000u;
  const uint32_t e = ((h >> 20) & 0x7ffu) - (1023u - 127u);  // float exponent field
  if (((h << 1) | l) == 0u) return {0.0f, 0.0f};
  const float hi = __uint_as_float(sign | (e << 23) | (__funnelshift_l(l, h, 3) & 0x7fffffu));
  const float lo = __fmul_rn(__uint2float_rn(l & 0x1fffffffu), __uint_as_float(sign | ((e - 52u) << 23)));
  return {hi, lo};
}

// The double nearest to t 2^k, ties to even (the result must be normal or zero).
__device__ __forceinline__ double scaled_double(long long t, int k) {
  const uint32_t sign = (uint32_t)(t >> 32) & 0x80000000u;
  const unsigned long long a = (unsigned long long)(t < 0 ? -t : t);
  const int lz = __clzll((long long)a);
  const unsigned long long n = a << (lz & 63);  // leading bit at 63
  const unsigned long long m = n >> 11;
  const uint32_t rest = (uint32_t)n & 0x7ffu;
  const uint32_t up = (rest > 0x400u || (rest == 0x400u && ((uint32_t)m & 1u))) ? 1u : 0u;
  // the leading bit of m adds 1 to the exponent field, and so does a carry out of the rounding
  unsigned long long bits = m + up + ((unsigned long long)(uint32_t)(1023 + 62 - lz + k) << 52);
  if (a == 0ull) bits = 0ull;
  return __hiloint2double((int)((uint32_t)(bits >> 32) | sign), (int)(uint32_t)bits);
}

}  // namespace rflbm_dev
