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

// 1 / x for a normal x far from overflow: the approximation instruction and two Newton-Raphson steps (4 FP64
// operations), and a / x from it, corrected once by its remainder (3; P. Markstein, "Computation of elementary functions on the
// IBM RISC System/6000 processor", IBM J. Res. Dev. 34, 1990). Within 2 units in the last place of the correctly rounded
// quotient, as tested.
__device__ __forceinline__ double reciprocal64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = __fma_rn(y, __fma_rn(-x, y, 1.0), y);
  return __fma_rn(y, __fma_rn(-x, y, 1.0), y);
}
__device__ __forceinline__ double divide64(double a, double x, double inv_x) {
  const double q = __dmul_rn(a, inv_x);
  return __fma_rn(__fma_rn(-x, q, a), inv_x, q);
}

// A running sum of float32 values as three of them: the rounding errors of each addition are
// carried exactly into the next (the last one rounds), so that it holds more than the 53 bits
// of an FP64 sum without an FP64 operation per term.
struct RunningSum {
  float s0 = 0.0f, s1 = 0.0f, s2 = 0.0f;
  __device__ __forceinline__ void add(float v) {
    float e0, e1;
    s0 = two_sum(s0, v, e0);
    s1 = two_sum(s1, e0, e1);
    s2 = __fadd_rn(s2, e1);
  }
  __device__ __forceinline__ double value() const { return ((double)s2 + (double)s1) + (double)s0; }
};

// Sums over one axis of a 3x3x3 tile after another: drho = sum g, j = sum g c, the raw second
// moments s = sum g c_a c_b (xx, yy, zz, xy, xz, yz).
__device__ __forceinline__ void raw_sums(const float (&G)[3][3][3], float (&m)[10]) {
  float X0[3][3], X1[3][3], X2[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      X2[b][c] = __fadd_rn(G[2][b][c], G[0][b][c]);
      X1[b][c] = __fsub_rn(G[2][b][c], G[0][b][c]);
      X0[b][c] = __fadd_rn(X2[b][c], G[1][b][c]);
    }
  const auto sum3 = [](float a, float b, float c) { return __fadd_rn(__fadd_rn(a, b), c); };
  float T00[3], T01[3], T02[3], T10[3], T11[3], T20[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    T02[c] = __fadd_rn(X0[2][c], X0[0][c]);
    T01[c] = __fsub_rn(X0[2][c], X0[0][c]);
    T00[c] = __fadd_rn(T02[c], X0[1][c]);
    T11[c] = __fsub_rn(X1[2][c], X1[0][c]);
    T10[c] = sum3(X1[2][c], X1[0][c], X1[1][c]);
    T20[c] = sum3(X2[2][c], X2[0][c], X2[1][c]);
  }
  m[6] = __fadd_rn(T00[2], T00[0]);
  m[0] = __fadd_rn(m[6], T00[1]);
  m[1] = sum3(T10[0], T10[1], T10[2]);
  m[2] = sum3(T01[0], T01[1], T01[2]);
  m[3] = __fsub_rn(T00[2], T00[0]);
  m[4] = sum3(T20[0], T20[1], T20[2]);
  m[5] = sum3(T02[0], T02[1], T02[2]);
  m[7] = sum3(T11[0], T11[1], T11[2]);
  m[8] = __fsub_rn(T10[2], T10[0]);
  m[9] = __fsub_rn(T01[2], T01[0]);
}

// The same sums as integers in units of 2^(e - 53), where e is the least exponent with every
// |g| < 2^e: each g is split on the grids 2^(e - 17) and 2^(e - 35), so that in every part a g is at most
// 2^17 of its units and a sum of 27 at most 27 2^17 < 2^22. The sums of the first two parts are exact in
// float32, and so is the remainder's to 2^(e - 53); adding 1.5 2^23 leaves such an integer in the low bits, which holds
// up to 2^22 only. An FP64 accumulation of the 27 terms keeps 2^(e - 50) or so. E = e + 126 (the
// exponent field of the largest |g|), 60 <= E <= 240. G is used up.
__device__ __forceinline__ void fixed_sums(float (&G)[3][3][3], uint32_t E, long long (&t)[10]) {
  const float half23 = 12582912.0f;  // 1.5 2^23
  float m[10];
#pragma unroll
  for (int part = 0; part < 3; ++part) {
    const uint32_t down = part == 0 ? 270u : (part == 1 ? 288u : 306u);  // 1 / unit
    if (part < 2) {
      const float grid = __uint_as_float(((part == 0 ? E + 7u : E - 11u) << 23) | 0x400000u);  // 1.5 2^23 units
      float H[3][3][3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            H[a][b][c] = __fsub_rn(__fadd_rn(G[a][b][c], grid), grid);
            G[a][b][c] = __fsub_rn(G[a][b][c], H[a][b][c]);
          }
      raw_sums(H, m);
    } else {
      raw_sums(G, m);
    }
    const float scale = __uint_as_float((down - E) << 23);
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const int n = __float_as_int(__fmaf_rn(m[k], scale, half23)) - __float_as_int(half23);
      if (part == 0) t[k] = n;
      else t[k] = t[k] * 262144 + n;
    }
  }
}

}  // namespace rflbm_dev
