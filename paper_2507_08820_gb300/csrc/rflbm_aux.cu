// Kernels around the step: initial states, population import/export in the pull layout,
// FP64 moments and global diagnostics, and the noise-source test kernels. Every kernel
// that touches the populations is instantiated for the three storage formats.
#include "rflbm_aux.h"
#include "wide.cuh"

namespace rflbm_dev {

constexpr int kAuxBlock = 256;

__device__ __forceinline__ uint32_t site_of(int64_t t) { return (uint32_t)t; }

// One 1-D factor of the product-form equilibrium (Eq. 26 factorised over the axes):
// Psi(0, u) = 2/3 - u^2, Psi(+-1, u) = (1/3 +- u + u^2)/2. Every rounding is spelled out, so that a stored state does
// not depend on which products a compiler joins with a sum.
__device__ __forceinline__ double psi(int c, double u) {
  const double q = __dmul_rn(u, u);
  return c == 0 ? __dsub_rn(2.0 / 3.0, q) : __dmul_rn(0.5, __dadd_rn(__dadd_rn(1.0 / 3.0, c * u), q));
}

// Population with the velocity of tile entry (a, b, c) = (c_x + 1, c_y + 1, c_z + 1).
__host__ __device__ constexpr int pop_at(int a, int b, int c) {
  for (int k = 0; k < kQ; ++k)
    if (cx_of(k) == a - 1 && cy_of(k) == b - 1 && cz_of(k) == c - 1) return k;
  return 0;
}

// ---------------------------------------------------------------- initial states
// The rest populations w_i rho0 in the element type of an import or export, rounded once on
// the host.
template <class Tio>
struct RestPops {
  Tio f[kQ];
};
template <class Tio>
static RestPops<Tio> rest_pops(float rho0) {
  RestPops<Tio> r;
  for (int i = 0; i < kQ; ++i) r.f[i] = (Tio)(weight_of(i) * (double)rho0);
  return r;
}

// delta = psi(c, u) / w_c - 1 for c = -1, 0, +1: 3 u^2 -+ 3 u, -3 u^2 / 2. size: the sum of the terms'
// magnitudes, which the errors of d are relative to (near |u| = 1 the terms of c = -+1 cancel).
__device__ __forceinline__ void psi_excess(Pair32 u, Pair32 (&d)[3], float (&size)[3]) {
  const Pair32 q = pmul(u, u);
  const Pair32 q3 = pmul(Pair32{3.0f, 0.0f}, q), u3 = pmul(Pair32{3.0f, 0.0f}, u);
  d[0] = padd(q3, Pair32{-u3.hi, -u3.lo});
  d[1] = pmul(Pair32{-1.5f, 0.0f}, q);
  d[2] = padd(q3, u3);
  size[0] = size[2] = __fadd_rn(q3.hi, fabsf(u3.hi));
  size[1] = fabsf(d[1].hi);
}

// g_i = r psi(c_x, u_x) psi(c_y, u_y) psi(c_z, u_z) - w_i rho0 of one site in FP64.
template <int kStore>
__device__ __noinline__ void init_site_fp64(const Geometry& g, uint32_t s, float rho0, const StoreScale& ss, double r,
                                            double ux, double uy, double uz, typename Storage<kStore>::T* dst) {
  using S = Storage<kStore>;
  const PopSlots slots(s, g);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const double f = __dmul_rn(__dmul_rn(r, psi(cx_of(i), ux)), psi(cy_of(i), uy));
    const double g_i = __fma_rn(f, psi(cz_of(i), uz), -__dmul_rn(weight_of(i), (double)rho0));
    dst[slots(i)] = S::store((float)g_i, class_of(i), ss);
  }
}

// The same for every site, scattered to the view's slots. With psi(c, u) = w_c (1 + delta_c),
// g_i / w_i = Q_ab + (rho0 + Q_ab) delta_c where Q_ab = r D_ab + (r - rho0) and 1 + D_ab =
// (1 + delta_a)(1 + delta_b): the rest value is no difference any more, so sums of two float32 values
// carry it to some 2^-43 of the magnitudes of its terms, and FP64 differs from it by no more than its own dozen
// roundings of f_i. Where every value within these errors rounds to one float32 value, that is
// the FP64 result; a site with any population that they leave open is redone in FP64 (one site in
// thousands for flows with velocities of a percent; most below 1e-6, where g_i is lost in the roundings of
// f_i, and a warp with one such site takes as long as one of them). Bound by the 32 bytes read and
// 108 written per site (146 us at 192^3): 192^3 takes 367 us with velocities of 2 %, 1270 us at rest or with
// velocities up to 1e-4, and took 1255 us with 100 FP64 operations for every site.
template <int kStore>
__global__ void __launch_bounds__(kAuxBlock) k_init_field(Geometry g, float rho0, StoreScale ss, const double* __restrict__ rho,
                             const double* __restrict__ u, typename Storage<kStore>::T* __restrict__ dst) {
  using S = Storage<kStore>;
  const int64_t s = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (s >= g.n) return;
  const double r = rho ? rho[s] : (double)rho0;
  const double ux = u ? u[s] : 0.0, uy = u ? u[g.n + s] : 0.0, uz = u ? u[2 * (int64_t)g.n + s] : 0.0;
  const double dr = r - (double)rho0;
  // (below 2^16 no product of r with the three delta_c overflows)
  bool open = !(pair_range(r, 16) && pair_range(dr, 16) && pair_range(ux, 16) && pair_range(uy, 16) && pair_range(uz, 16));
  if (!open) {
    const PopSlots slots(site_of(s), g);
    const Pair32 R = pair_of(r), dR = pair_of(dr);
    Pair32 dx[3], dy[3], dz[3];
    float tx[3], ty[3], tz[3];
    psi_excess(pair_of(ux), dx, tx);
    psi_excess(pair_of(uy), dy, ty);
    psi_excess(pair_of(uz), dz, tz);
    const float own = fmaf(0x1p-43f, fabsf(dR.hi), 0x1p-48f * (fabsf(R.hi) + rho0));
    // The pairs' errors over R A, A the terms of f_i / w_i r - 1: at most 0.42, 0.67, 1.1, 1.9 and 4.3 times 2^-43 for
    // velocities of 0.03, 0.1, 0.3, 1 and 10 to 2^16 (the largest of 2 M random sites each); FP64's: below 2^-47.
    const float corner = fmaf(1.0f + tx[0], fmaf(ty[0], 1.0f + tz[0], tz[0]), tx[0]);  // the largest A of the site
    const float slope = fmaf(fminf(corner, 8.0f), 0x1p-43f, 0x1.1p-43f);
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const float Aab = fmaf(tx[a], ty[b], tx[a] + ty[b]);
        const Pair32 D = padd(padd(dx[a], dy[b]), pmul(dx[a], dy[b]));
        const Pair32 Q = padd(pmul(R, D), dR);
        const Pair32 P = padd(Pair32{rho0, 0.0f}, Q);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          constexpr double w[4] = {w1d(1) * w1d(1) * w1d(1), w1d(1) * w1d(1) * w1d(0), w1d(1) * w1d(0) * w1d(0),
                                   w1d(0) * w1d(0) * w1d(0)};
          const int cls = class_at(a, b, c);
          const Pair32 W{(float)w[cls], (float)(w[cls] - (double)(float)w[cls])};
          const Pair32 v = pmul(W, padd(Q, pmul(P, dz[c])));
          const float A = fmaf(tz[c], 1.0f + Aab, Aab);  // over the terms of f_i / w_i r - 1
          const float err = W.hi * fmaf(fabsf(R.hi) * A, slope, own);
          const float lo = __fadd_rn(v.hi, __fsub_rn(v.lo, err));
          open = open || !(lo == __fadd_rn(v.hi, __fadd_rn(v.lo, err)));
          dst[slots(pop_at(a, b, c))] = S::store(lo, cls, ss);
        }
      }
  }
  if (open) init_site_fp64<kStore>(g, site_of(s), rho0, ss, r, ux, uy, uz, dst);
}

// Thermal initial state: every mode of every site an independent normal of variance
// rho0 kT b_k / cs2 (the variance the amplitude of Eq. 10 maintains) around the rest
// state, drawn with Philox calls j = 6..12 of counter (site, 0, j, replica) (the step
// draws use j = 0..5). The scaled moments M = m_k / b_k = sqrt(3 rho0 kT / b_k) n_k go
// through the back transform of Eq. 11 (three sweeps of 1-D lines, then the weights).
template <int kStore>
__global__ void k_init_thermal(Geometry g, float rho0, float kT, StoreScale ss, uint32_t key0, uint32_t key1,
                               uint32_t replica, typename Storage<kStore>::T* __restrict__ dst) {
  using S = Storage<kStore>;
  const int64_t s = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (s >= g.n) return;
  float nrm[28];
#pragma unroll
  for (int j = 0; j < 7; ++j) {
    const uint4 w = philox4x32_10(make_uint4(site_of(s) + g.site0, 0u, 6u + (uint32_t)j, replica), key0, key1);
    float r, c, sn;
    box_muller(w.x, w.y, r, c, sn);
    nrm[4 * j] = r * c;
    nrm[4 * j + 1] = r * sn;
    box_muller(w.z, w.w, r, c, sn);
    nrm[4 * j + 2] = r * c;
    nrm[4 * j + 3] = r * sn;
  }
  float M[3][3][3];
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int r = 0; r < 3; ++r)
        M[p][q][r] = sqrtf((float)(3.0 * (1.0 / bnorm(p, q, r))) * rho0 * kT) * nrm[mode_of(p, q, r)];
  float Z[3][3][3], Y[3][3][3];
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q)
      line_inverse(M[p][q][0], M[p][q][1], M[p][q][2], Z[p][q][0], Z[p][q][1], Z[p][q][2]);
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int c = 0; c < 3; ++c)
      line_inverse(Z[p][0][c], Z[p][1][c], Z[p][2][c], Y[p][0][c], Y[p][1][c], Y[p][2][c]);
  const PopSlots slots(site_of(s), g);
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      float o[3];
      line_inverse(Y[0][b][c], Y[1][b][c], Y[2][b][c], o[0], o[1], o[2]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        dst[slots(pop_at(a, b, c))] =
            S::store((float)(w1d(a) * w1d(b) * w1d(c)) * o[a], class_at(a, b, c), ss);
      }
    }
}

// Import and export move 216 bytes per site (f32): 128^3 float32 takes 65 us each way, and took
// 96 us in and 116 us out with the rest populations formed by four FP64 products in every thread.
// Import of public-layout populations (double: exact shift in FP64; float: in FP32).
template <class Tin, int kStore>
__global__ void k_set_populations(Geometry g, RestPops<Tin> rest, StoreScale ss, const Tin* __restrict__ f,
                                  typename Storage<kStore>::T* __restrict__ dst) {
  using S = Storage<kStore>;
  const int64_t s = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (s >= g.n) return;
  const PopSlots slots(site_of(s), g);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const Tin v = f[i * (int64_t)g.n + s] - rest.f[i];
    dst[slots(i)] = S::store((float)v, class_of(i), ss);
  }
}

template <class Tout, int kStore>
__global__ void k_get_populations(Geometry g, RestPops<Tout> rest, StoreScale ss,
                                  const typename Storage<kStore>::T* __restrict__ src, Tout* __restrict__ f) {
  using S = Storage<kStore>;
  const int64_t s = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (s >= g.n) return;
  const PopSlots slots(site_of(s), g);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const float v = S::load(src[slots(i)], class_of(i), ss);
    f[i * (int64_t)g.n + s] = (Tout)v + rest.f[i];
  }
}

template <int kStore>
__global__ void k_get_sites(Geometry g, float rho0, StoreScale ss,
                            const typename Storage<kStore>::T* __restrict__ src,
                            const int64_t* __restrict__ sites, int64_t n, double* __restrict__ f) {
  using S = Storage<kStore>;
  const int64_t j = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (j >= n) return;
  const uint32_t s = site_of(sites[j]);
  const PopSlots slots(s, g);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    f[i * n + j] = (double)S::load(src[slots(i)], class_of(i), ss) +
                   weight_of(i) * (double)rho0;
  }
}

// Raw moments of order <= 2 of the shifted populations of one site in FP64.
struct SiteMoments {
  double drho, j[3], s[6];  // s: sum g c_a c_b for xx, yy, zz, xy, xz, yz
};

template <int kStore>
__device__ __forceinline__ SiteMoments site_moments(const Geometry& g, uint32_t s,
                                                    const typename Storage<kStore>::T* src,
                                                    const StoreScale& ss) {
  const PopSlots slots(s, g);
  using S = Storage<kStore>;
  double drho = 0, j0 = 0, j1 = 0, j2 = 0, s0 = 0, s1 = 0, s2 = 0, s3 = 0, s4 = 0, s5 = 0;
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const double v = (double)S::load(src[slots(i)], class_of(i), ss);
    const int cx = cx_of(i), cy = cy_of(i), cz = cz_of(i);
    drho += v;
    if (cx) j0 += cx * v;
    if (cy) j1 += cy * v;
    if (cz) j2 += cz * v;
    if (cx) s0 += v;
    if (cy) s1 += v;
    if (cz) s2 += v;
    if (cx * cy) s3 += cx * cy * v;
    if (cx * cz) s4 += cx * cz * v;
    if (cy * cz) s5 += cy * cz * v;
  }
  SiteMoments m;
  m.drho = drho;
  m.j[0] = j0; m.j[1] = j1; m.j[2] = j2;
  m.s[0] = s0; m.s[1] = s1; m.s[2] = s2; m.s[3] = s3; m.s[4] = s4; m.s[5] = s5;
  return m;
}

// The moments of one site in plain FP64.
template <int kStore>
__device__ __noinline__ void moments_fp64(const Geometry& g, uint32_t s, const StoreScale& ss,
                                          const typename Storage<kStore>::T* src, double rho0, double* rho, double* u,
                                          double* pi) {
  const SiteMoments m = site_moments<kStore>(g, s, src, ss);
  const double r = rho0 + m.drho;
  if (rho) rho[s] = r;
  if (u) {
#pragma unroll
    for (int a = 0; a < 3; ++a) u[a * (int64_t)g.n + s] = m.j[a] / r;
  }
  if (pi) {
    // Pi_ab = sum_i f_i (c_a c_b - delta_ab/3) = sum_i g_i c_a c_b - delta_ab drho/3
#pragma unroll
    for (int a = 0; a < 6; ++a)
      pi[a * (int64_t)g.n + s] = m.s[a] - (a < 3 ? m.drho / 3.0 : 0.0);
  }
}

// FP64 moments of every site: sums of 27 float32 values carried in 64-bit integers (fixed_sums),
// packed into FP64 by integer operations, so that 15 FP64 operations per site are left (the
// density and the three quotients) where plain FP64 takes 250. Bound by the 108 bytes read and
// 80 written per site (196 us at 192^3; it takes 337 us, plain FP64 took 3224 us). Values outside the
// split's range (a population of 2^114 or more, or all below 2^-66 and not zero; non-finite ones)
// go through FP64.
template <int kStore>
__global__ void __launch_bounds__(kAuxBlock) k_moments(Geometry g, double rho0, StoreScale ss,
                          const typename Storage<kStore>::T* __restrict__ src,
                          double* __restrict__ rho, double* __restrict__ u, double* __restrict__ pi) {
  using S = Storage<kStore>;
  const int64_t s = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (s >= g.n) return;
  float G[3][3][3];
  uint32_t top = 0;
  {
    const PopSlots slots(site_of(s), g);
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const float v = S::load(src[slots(i)], class_of(i), ss);
      G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = v;
      top = max(top, __float_as_uint(v) & 0x7fffffffu);
    }
  }
  const uint32_t E = top == 0u ? 127u : top >> 23;
  if (E < 60u || E > 240u) {
    moments_fp64<kStore>(g, site_of(s), ss, src, rho0, rho, u, pi);
    return;
  }
  long long t[10];
  fixed_sums(G, E, t);
  const int k = (int)E - 179;  // units of 2^(e - 53)
  if (rho || u) {
    const double r = rho0 + scaled_double(t[0], k);
    if (rho) rho[s] = r;
    if (u) {
      // (the reciprocal's Newton steps need a normal r far from overflow)
      const uint32_t er = ((uint32_t)__double2hiint(r) >> 20) & 0x7ffu;
      const bool plain = er < 1023u - 130u || er > 1023u + 130u;
      const double inv = reciprocal64(r);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double j = scaled_double(t[1 + a], k);
        u[a * (int64_t)g.n + s] = plain ? j / r : divide64(j, r, inv);
      }
    }
  }
  if (pi) {
    // Pi_ab = sum_i f_i (c_a c_b - delta_ab/3) = sum_i g_i c_a c_b - delta_ab drho/3
    const long long third = (t[0] + (t[0] < 0 ? -1 : 1)) / 3;  // to the nearest unit
#pragma unroll
    for (int a = 0; a < 6; ++a) pi[a * (int64_t)g.n + s] = scaled_double(a < 3 ? t[4 + a] - third : t[4 + a], k);
  }
}

// Partial sums: drho, j (3), max |u|, count of unstable sites (non-finite, or density not
// positive).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// x^2 + y^2 + z^2 rounded once from a sum with its rounding errors kept.
__device__ __forceinline__ float sum_squares(float x, float y, float z) {
  const float p = __fmul_rn(x, x), q = __fmul_rn(y, y), r = __fmul_rn(z, z);
  float e1, e2;
  const float s1 = two_sum(p, q, e1);
  const float s2 = two_sum(s1, r, e2);
  const float ep = __fmaf_rn(x, x, -p), eq = __fmaf_rn(y, y, -q), er = __fmaf_rn(z, z, -r);
  return __fadd_rn(s2, __fadd_rn(__fadd_rn(e1, e2), __fadd_rn(ep, __fadd_rn(eq, er))));
}

__device__ __noinline__ float speed64(float x, float y, float z, float r) {
  return (float)(sqrt((double)x * x + (double)y * y + (double)z * z) / (double)r);
}

// Global sums: every block sums the sites of its stride into one row of partials, and the last
// block to finish adds the rows in a fixed order into out. Bound by the 108 bytes read per
// site. A site's sums are taken into FP64 once per thread (RunningSum), not once per site: with
// 20 FP64 operations per site, and the final sum in a launch of its own, 128^3 float32 took
// 375 + 7 us, and takes 52 us.
constexpr int kStatSums = 4;  // drho, j
template <int kStore>
__global__ void __launch_bounds__(kAuxBlock, 3) k_stats(Geometry g, float rho0, StoreScale ss,
                                const typename Storage<kStore>::T* __restrict__ src,
                                double* __restrict__ partials, double* __restrict__ out, unsigned* __restrict__ done) {
  using S = Storage<kStore>;
  RunningSum acc[kStatSums];
  double big[kStatSums] = {0, 0, 0, 0};  // values of 2^100 and more
  float vmax = 0.0f;
  int bad = 0;
  // the next site's loads are issued as soon as this one's values are summed, and its sums follow in their
  // shadow (128^3 float32 61 -> 52 us, with 3 blocks of 80 registers per SM instead of
  // 4 of 64, where the waiting values spill)
  typename S::T raw[kQ];
  const auto fetch = [&](int64_t s) {
    const PopSlots slots(site_of(s), g);
#pragma unroll
    for (int i = 0; i < kQ; ++i) raw[i] = src[slots(i)];
  };
  int64_t s = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (s < g.n) fetch(s);
#pragma unroll 1
  while (s < g.n) {
    float m[kStatSums] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const float v = S::load(raw[i], class_of(i), ss);
      m[0] += v;
      if (cx_of(i)) m[1] += cx_of(i) * v;
      if (cy_of(i)) m[2] += cy_of(i) * v;
      if (cz_of(i)) m[3] += cz_of(i) * v;
    }
    s += (int64_t)gridDim.x * kAuxBlock;
    if (s < g.n) fetch(s);
    const float r = __fadd_rn(rho0, m[0]);
    const float mj = fmaxf(fabsf(m[1]), fmaxf(fabsf(m[2]), fabsf(m[3])));
    // a non-finite site, or one whose density is not positive, counts as unstable
    if (!(isfinite(m[0]) && isfinite(m[1]) && isfinite(m[2]) && isfinite(m[3]) && r > 0.0f)) {
      ++bad;
    } else if (fmaxf(fabsf(m[0]), mj) < 0x1p100f) {
#pragma unroll
      for (int f = 0; f < kStatSums; ++f) acc[f].add(m[f]);
      // outside 2^-40 .. 2^60 the squares leave the range where their errors are exact
      vmax = fmaxf(vmax, mj == 0.0f || (mj < 0x1p60f && mj > 0x1p-40f) ? sqrtf(sum_squares(m[1], m[2], m[3])) / r
                                                                      : speed64(m[1], m[2], m[3], r));
    } else {
#pragma unroll
      for (int f = 0; f < kStatSums; ++f) big[f] += (double)m[f];
      vmax = fmaxf(vmax, speed64(m[1], m[2], m[3], r));
    }
  }
  // the block's row: warp f < 4 adds the threads' sums of field f, warp 4 their maxima and counts
  __shared__ double sh[kStatSums][kAuxBlock];
  __shared__ float shmax[kAuxBlock / 32];
  __shared__ int shbad[kAuxBlock / 32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int f = 0; f < kStatSums; ++f) sh[f][threadIdx.x] = acc[f].value() + big[f];
  // (vmax >= 0: its bits order like integers)
  const unsigned wmax = __reduce_max_sync(0xffffffffu, __float_as_uint(vmax));
  const int wbad = __reduce_add_sync(0xffffffffu, bad);
  if (lane == 0) {
    shmax[wid] = __uint_as_float(wmax);
    shbad[wid] = wbad;
  }
  __syncthreads();
  double* const row = partials + (int64_t)blockIdx.x * kStatOutFields;
  if (wid < kStatSums) {
    double v = 0.0;
    for (int k = lane; k < kAuxBlock; k += 32) v += sh[wid][k];
    v = warp_sum(v);
    if (lane == 0) row[wid] = v;
  } else if (wid == kStatSums && lane == 0) {
    float m = 0.0f;
    int c = 0;
    for (int w = 0; w < kAuxBlock / 32; ++w) {
      m = fmaxf(m, shmax[w]);
      c += shbad[w];
    }
    row[4] = (double)m;
    row[5] = (double)c;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (wid < kStatOutFields) {
    double v = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) {
      const double p = __ldcg(partials + (int64_t)b * kStatOutFields + wid);
      v = (wid == 4) ? fmax(v, p) : v + p;
    }
    v = (wid == 4) ? warp_max(v) : warp_sum(v);
    if (lane == 0) out[wid] = v;
  }
  if (threadIdx.x == 0) *done = 0u;  // ready for the next call
}

// ---------------------------------------------------------------- noise tests
__global__ void k_philox(const uint32_t* __restrict__ ctr, uint32_t k0, uint32_t k1,
                         uint32_t* __restrict__ out, int64_t n) {
  const int64_t j = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (j >= n) return;
  const uint4 w = philox4x32_10(make_uint4(ctr[4 * j], ctr[4 * j + 1], ctr[4 * j + 2], ctr[4 * j + 3]), k0, k1);
  out[4 * j] = w.x; out[4 * j + 1] = w.y; out[4 * j + 2] = w.z; out[4 * j + 3] = w.w;
}

__global__ void k_site_normals(uint32_t k0, uint32_t k1, uint32_t step, uint32_t replica,
                               const uint32_t* __restrict__ sites, int64_t n,
                               float* __restrict__ out) {
  const int64_t j = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (j >= n) return;
  SiteNoise nz;
  site_noise(sites[j], step, replica, k0, k1, nz);
#pragma unroll
  for (int m = 0; m < 24; ++m) out[24 * j + m] = normal_at(nz, m);
}

// ---------------------------------------------------------------- state images
// One plane of a state image (pull layout) from the plane of population i of a buffer in
// the natural view: out[y] = plane[y + c_i] under periodic wrap, zeros in the padding.
template <class E>
__global__ void k_image_plane(Geometry g, const E* __restrict__ plane, int cx, int cy, int cz,
                              E* __restrict__ out) {
  const int64_t y = (int64_t)blockIdx.x * kAuxBlock + threadIdx.x;
  if (y >= g.ps) return;
  if (y >= g.n) {
    out[y] = E(0);
    return;
  }
  const Neighbours nb = neighbours((uint32_t)y, g);  // X[a], Y[b], Z[c]: coordinate - (a - 1)
  out[y] = plane[nb.X[1 - cx] + nb.Y[1 - cy] + nb.Z[1 - cz]];
}

// ---------------------------------------------------------------- launchers
static unsigned blocks_for(int64_t n) { return (unsigned)((n + kAuxBlock - 1) / kAuxBlock); }

#define RFLBM_STORE_DISPATCH(kind, CALL)                                   \
  switch (kind) {                                                          \
    case kStoreF32: { constexpr int K = kStoreF32; CALL; } break;          \
    case kStoreF16: { constexpr int K = kStoreF16; CALL; } break;          \
    case kStoreBF16: { constexpr int K = kStoreBF16; CALL; } break;        \
    default: return cudaErrorInvalidValue;                                 \
  }

template <int K>
using ST = typename Storage<K>::T;

cudaError_t launch_init_field(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                              const double* rho, const double* u, void* dst, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_init_field<K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, rho0, ss, rho, u, (ST<K>*)dst)));
  return cudaGetLastError();
}
cudaError_t launch_set_populations_f64(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                                       const double* f, void* dst, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_set_populations<double, K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, rest_pops<double>(rho0), ss, f, (ST<K>*)dst)));
  return cudaGetLastError();
}
cudaError_t launch_set_populations_f32(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                                       const float* f, void* dst, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_set_populations<float, K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, rest_pops<float>(rho0), ss, f, (ST<K>*)dst)));
  return cudaGetLastError();
}
cudaError_t launch_get_populations_f64(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                                       const void* src, double* f, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_get_populations<double, K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, rest_pops<double>(rho0), ss, (const ST<K>*)src, f)));
  return cudaGetLastError();
}
cudaError_t launch_get_populations_f32(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                                       const void* src, float* f, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_get_populations<float, K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, rest_pops<float>(rho0), ss, (const ST<K>*)src, f)));
  return cudaGetLastError();
}
cudaError_t launch_get_sites(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                             const void* src, const int64_t* sites, int64_t n, double* f,
                             cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_get_sites<K><<<blocks_for(n), kAuxBlock, 0, st>>>(g, rho0, ss, (const ST<K>*)src, sites, n, f)));
  return cudaGetLastError();
}
cudaError_t launch_moments(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                           const void* src, double* rho, double* u, double* pi, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_moments<K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, (double)rho0, ss, (const ST<K>*)src, rho, u, pi)));
  return cudaGetLastError();
}
int stats_partial_blocks(const Geometry& g, int num_sms) {
  const int64_t want = (g.n + kAuxBlock - 1) / kAuxBlock;
  const int64_t cap = 3 * (int64_t)num_sms;  // k_stats holds 3 blocks per SM
  return (int)(want < cap ? (want > 0 ? want : 1) : cap);
}
cudaError_t launch_stats(const Geometry& g, float rho0, const StoreScale& ss, int kind,
                         const void* src, double* partials, int nblocks, double* out, unsigned* done,
                         cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_stats<K><<<nblocks, kAuxBlock, 0, st>>>(g, rho0, ss, (const ST<K>*)src, partials, out, done)));
  return cudaGetLastError();
}
cudaError_t launch_image_plane(const Geometry& g, size_t elem, const void* plane, int cx, int cy, int cz,
                               void* out, cudaStream_t st) {
  if (elem == 4)
    k_image_plane<uint32_t><<<blocks_for(g.ps), kAuxBlock, 0, st>>>(g, (const uint32_t*)plane, cx, cy, cz, (uint32_t*)out);
  else if (elem == 2)
    k_image_plane<uint16_t><<<blocks_for(g.ps), kAuxBlock, 0, st>>>(g, (const uint16_t*)plane, cx, cy, cz, (uint16_t*)out);
  else
    return cudaErrorInvalidValue;
  return cudaGetLastError();
}
cudaError_t launch_init_thermal(const Geometry& g, float rho0, float kT, const StoreScale& ss, int kind,
                                uint32_t key0, uint32_t key1, uint32_t replica, void* dst, cudaStream_t st) {
  RFLBM_STORE_DISPATCH(kind, (k_init_thermal<K><<<blocks_for(g.n), kAuxBlock, 0, st>>>(g, rho0, kT, ss, key0, key1,
                                                                                        replica, (ST<K>*)dst)));
  return cudaGetLastError();
}
cudaError_t launch_philox(const uint32_t* ctr, uint32_t k0, uint32_t k1, uint32_t* out,
                          int64_t n, cudaStream_t st) {
  k_philox<<<blocks_for(n), kAuxBlock, 0, st>>>(ctr, k0, k1, out, n);
  return cudaGetLastError();
}
cudaError_t launch_site_normals(uint32_t k0, uint32_t k1, uint32_t step, uint32_t replica,
                                const uint32_t* sites, int64_t n, float* out, cudaStream_t st) {
  k_site_normals<<<blocks_for(n), kAuxBlock, 0, st>>>(k0, k1, step, replica, sites, n, out);
  return cudaGetLastError();
}

}  // namespace rflbm_dev
