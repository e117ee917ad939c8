// The two-site collision of 16-bit storage, straight from the stored values.
//
// A stored value is g 2^e with one exponent per velocity class, and a step's first use of it is a
// sum along x. The sm_100 family adds a 16-bit value to a float32 one in one instruction, and powers
// of two commute with rounding, so the sums run on the stored values: along each axis the centre
// value, of the class one below its neighbours', enters by a multiply-add with the ratio of the two
// scales, and only the ten moments are unscaled. Against converting and scaling 27 values
// first, float16 with noise, microseconds per step: 256^3 503.5 -> 500.2, AA 256^3 539.4 -> 530.9, without
// noise 300x128x64 45.0 -> 43.9; the ensembles' row tiles and the flat tiles with noise measured
// slower (64 replicas 446 -> 479) and convert first. Same bits.
#pragma once

#include "collide.cuh"
#include "storage.cuh"

namespace rflbm_dev {

// raw(a, b, c, v): the stored values of tile entry (a, b, c) of both sites.
template <int kStore, bool kNoise, class Raw, class Noise, class OutWeight>
__device__ __forceinline__ void collide_stored(const Raw& raw, const StoreScale& ss, float2 (&G)[3][3][3],
                                               const CollideParams& cp, const Noise& noise, const OutWeight& outw) {
  using S = Storage<kStore>;
  using T = typename S::T;
  float ratio[3];  // of the scales of classes k and k + 1
  T ratio16[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ratio[k] = ss.inv_scale[k] * ss.scale[k + 1];
    ratio16[k] = S::pack(ratio[k]);
  }
  // along x: in units of class (b != 1) + (c != 1) + 1
  float2 X0[3][3], X1[3][3], X2[3][3];
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      T m[2], z[2], p[2];
      raw(0, b, c, m);
      raw(1, b, c, z);
      raw(2, b, c, p);
      const int k = (b != 1) + (c != 1);
      const float m0 = S::to_float(m[0]), m1 = S::to_float(m[1]);
      X2[b][c] = make_float2(S::add(p[0], m0), S::add(p[1], m1));
      X1[b][c] = make_float2(S::sub(p[0], m0), S::sub(p[1], m1));
      X0[b][c] = make_float2(S::fma(z[0], ratio16[k], X2[b][c].x), S::fma(z[1], ratio16[k], X2[b][c].y));
    }
  // along y: in units of class (c != 1) + 2
  float2 T00[3], T01[3], T02[3], T10[3], T11[3], T20[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float r = ratio[(c != 1) + 1];
    T02[c] = vadd(X0[2][c], X0[0][c]);
    T01[c] = vsub(X0[2][c], X0[0][c]);
    T00[c] = kfma(r, X0[1][c], T02[c]);
    T11[c] = vsub(X1[2][c], X1[0][c]);
    T10[c] = kfma(r, X1[1][c], vadd(X1[2][c], X1[0][c]));
    T20[c] = kfma(r, X2[1][c], vadd(X2[2][c], X2[0][c]));
  }
  // along z: in units of class 3, then unscaled
  const float r = ratio[2], u = ss.inv_scale[3];
  const float2 s002 = vadd(T00[2], T00[0]);
  const float2 drho = kmul(u, kfma(r, T00[1], s002));
  const float2 jz = kmul(u, vsub(T00[2], T00[0]));
  const float2 jy = kmul(u, vadd(kfma(r, T01[1], T01[0]), T01[2]));
  const float2 syz = kmul(u, vsub(T01[2], T01[0]));
  const float2 syy = kmul(u, vadd(kfma(r, T02[1], T02[0]), T02[2]));
  const float2 jx = kmul(u, vadd(kfma(r, T10[1], T10[0]), T10[2]));
  const float2 sxz = kmul(u, vsub(T10[2], T10[0]));
  const float2 sxy = kmul(u, vadd(kfma(r, T11[1], T11[0]), T11[2]));
  const float2 sxx = kmul(u, vadd(kfma(r, T20[1], T20[0]), T20[2]));
  const float2 szz = kmul(u, s002);
  collide_moments<kNoise, false, false>(drho, jx, jy, jz, sxy, sxz, syz, kfma(-1.0f / 3.0f, drho, sxx),
                                        kfma(-1.0f / 3.0f, drho, syy), kfma(-1.0f / 3.0f, drho, szz), G, cp, noise, outw);
}

// The two values at p, p + 1 (16-bit storage; aligned: p is an even element).
template <class T>
__device__ __forceinline__ void stored_pair(const T* p, bool aligned, T (&v)[2]) {
  if (aligned) {
    const uint32_t w = *reinterpret_cast<const uint32_t*>(p);
    v[0] = reinterpret_cast<const T*>(&w)[0];
    v[1] = reinterpret_cast<const T*>(&w)[1];
  } else {
    v[0] = p[0];
    v[1] = p[1];
  }
}

}  // namespace rflbm_dev
