// Power spectrum |F(k)|^2 of one real field per site (3-D, half spectrum kx = 0 .. nx/2), in sums of
// two float32 values.
//
// An FP64 transform of 128^3 sites does 55 M FP64 operations, at 1.9 per clock and SM some
// 100 us at best (cuFFT's D2Z: 241 us), while its data is 17 MB. Here every real number of the
// transform is an unevaluated sum of two float32 values (Pair32: an addition takes 8 float32
// operations, a product 4, at 128 per clock). Twiddle factors carry 48 bits and an addition 46, so
// the transform's error, near 1e-14 of the norm, stays far below the rounding of the float32
// field (6e-8).
//
// Three passes, one per axis, each on tiles of kCols lines in shared memory (Stockham stages of
// radix 8, 4, 2 and the odd primes up to 13, two buffers):
//   x: two real rows at a time as one complex line; the half spectra of both rows out
//   y: in place
//   z: the last transform, and |F|^2 out instead of the spectrum
// The spectrum between the passes is read and written once each and stays in L2 up to 192^3. The
// three passes of 128^3 took 24 + 21 + 23 us with the tile loaded to and stored from shared memory,
// and 16 + 16 + 17 us with the first stage loading and the last one storing in global memory.
#include "rflbm_spectrum.h"
#include "tma.cuh"
#include "wide.cuh"

#include <cmath>
#include <vector>

namespace rflbm_dev {

namespace {

constexpr int kCols = 8;             // lines of a tile: 128 bytes of one row of the spectrum
constexpr int kMaxLine = 768;        // two tile buffers and the twiddles in 206 KB of shared memory

struct Cpx {
  Pair32 re, im;
};
__device__ __forceinline__ Pair32 pneg(Pair32 a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ Pair32 psub(Pair32 a, Pair32 b) { return padd(a, pneg(b)); }
__device__ __forceinline__ Cpx cadd(Cpx a, Cpx b) { return {padd(a.re, b.re), padd(a.im, b.im)}; }
__device__ __forceinline__ Cpx csub(Cpx a, Cpx b) { return {psub(a.re, b.re), psub(a.im, b.im)}; }
__device__ __forceinline__ Cpx cmul(Cpx a, Cpx b) {
  return {psub(pmul(a.re, b.re), pmul(a.im, b.im)), padd(pmul(a.re, b.im), pmul(a.im, b.re))};
}
__device__ __forceinline__ Cpx minus_i(Cpx a) { return {a.im, pneg(a.re)}; }
__device__ __forceinline__ Cpx unpack(float4 v) { return {{v.x, v.y}, {v.z, v.w}}; }
__device__ __forceinline__ float4 pack(Cpx a) { return make_float4(a.re.hi, a.re.lo, a.im.hi, a.im.lo); }

template <int R>
__device__ __forceinline__ void dft(Cpx (&v)[R], const float4* tw, int step);

__device__ __forceinline__ void dft2(Cpx& a, Cpx& b) {
  const Cpx t = csub(a, b);
  a = cadd(a, b);
  b = t;
}
__device__ __forceinline__ void dft4(Cpx& a, Cpx& b, Cpx& c, Cpx& d) {
  dft2(a, c);
  dft2(b, d);
  d = minus_i(d);
  dft2(a, b);
  dft2(c, d);
  const Cpx t = b;  // outputs in order 0, 1, 2, 3
  b = c;
  c = t;
}

// v -> its discrete Fourier transform of length R; tw[j step] = exp(-2 pi i j / R).
template <int R>
__device__ __forceinline__ void dft(Cpx (&v)[R], const float4* tw, int step) {
  if constexpr (R == 2) {
    dft2(v[0], v[1]);
  } else if constexpr (R == 4) {
    dft4(v[0], v[1], v[2], v[3]);
  } else if constexpr (R == 8) {
    constexpr Pair32 h{0.70710678118654752440f, (float)(0.70710678118654752440 - (double)0.70710678118654752440f)};
    dft4(v[0], v[2], v[4], v[6]);
    dft4(v[1], v[3], v[5], v[7]);
    // times exp(-2 pi i j / 8) of the odd half
    v[3] = {pmul(h, padd(v[3].re, v[3].im)), pmul(h, psub(v[3].im, v[3].re))};
    v[5] = minus_i(v[5]);
    v[7] = {pmul(h, psub(v[7].im, v[7].re)), pneg(pmul(h, padd(v[7].re, v[7].im)))};
    Cpx e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      v[j] = cadd(e[j], o[j]);
      v[j + 4] = csub(e[j], o[j]);
    }
  } else {  // an odd prime, by sums and differences of opposite terms
    constexpr int M = R / 2;
    Cpx s[M], d[M];
    Cpx total = v[0];
#pragma unroll
    for (int j = 0; j < M; ++j) {
      s[j] = cadd(v[j + 1], v[R - 1 - j]);
      d[j] = csub(v[j + 1], v[R - 1 - j]);
      total = cadd(total, s[j]);
    }
    const Cpx first = v[0];
    v[0] = total;
#pragma unroll 1
    for (int k = 1; k <= M; ++k) {
      Cpx a = first, b{{0.0f, 0.0f}, {0.0f, 0.0f}};
      int m = 0;
#pragma unroll
      for (int j = 0; j < M; ++j) {
        m += k;
        m -= m >= R ? R : 0;
        const Cpx w = unpack(tw[m * step]);  // cos, -sin
        a = {padd(a.re, pmul(w.re, s[j].re)), padd(a.im, pmul(w.re, s[j].im))};
        b = {psub(b.re, pmul(w.im, d[j].im)), padd(b.im, pmul(w.im, d[j].re))};
      }
      // (k is not a compile-time index: select the two outputs)
#pragma unroll
      for (int q = 1; q <= M; ++q)
        if (q == k) {
          v[q] = cadd(a, b);
          v[R - q] = csub(a, b);
        }
    }
  }
}

// One Stockham stage of radix R over a tile of kCols lines: `before` is the product of the radices
// done so far; load(position, line) and store(position, line, value) reach the tile. Consecutive
// threads take consecutive lines.
template <int R, class Load, class Store>
__device__ __forceinline__ void stage(const Load& load, const Store& store, const float4* tw, int n, int before) {
  const int m = n / R;
  for (int b = threadIdx.x; b < m * kCols; b += blockDim.x) {
    const int c = b % kCols, j = b / kCols;
    const int q = j / before, k = j - q * before;
    Cpx v[R];
    const int tstep = k * (m / before);  // twiddle exp(-2 pi i r k / (before R))
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = load(j + r * m, c);
    if (before > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], unpack(tw[r * tstep]));
    }
    dft<R>(v, tw, m);
    const int o = q * before * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) store(o + r * before, c, v[r]);
  }
}

template <int kOdd, class Load, class Store>
__device__ __forceinline__ void stage_of(int r, const Load& load, const Store& store, const float4* tw, int n, int before) {
  if (r == 8) stage<8>(load, store, tw, n, before);
  else if (r == 4) stage<4>(load, store, tw, n, before);
  else if (r == 2) stage<2>(load, store, tw, n, before);
  if constexpr (kOdd > 0) {
    if (r == 3) stage<3>(load, store, tw, n, before);
    if (r == 5) stage<5>(load, store, tw, n, before);
    if (r == 7) stage<7>(load, store, tw, n, before);
  }
  if constexpr (kOdd > 1) {
    if (r == 11) stage<11>(load, store, tw, n, before);
    if (r == 13) stage<13>(load, store, tw, n, before);
  }
}

// The lines of a tile through all stages: the first one loads from global memory, the last one
// stores there (they keep no copy of the tile in shared memory, and their accesses overlap with
// the butterflies); between stages the values go through the buffers a and b in turn. kOdd: 1 with
// the radices 3, 5 and 7, 2 with 11 and 13 too.
template <int kOdd, class Load, class Store>
__device__ __forceinline__ void transform(float4* a, float4* b, const float4* tw, const SpectrumAxis& ax, const Load& load,
                                          const Store& store) {
  const int n = ax.n, last = ax.nfactors - 1;
  if (last < 0) {  // n = 1
    if (threadIdx.x < kCols) store(0, (int)threadIdx.x, load(0, (int)threadIdx.x));
    return;
  }
  if (kOdd > 0) __syncthreads();  // odd radices read the twiddles in their first stage
  if (last == 0) {
    stage_of<kOdd>(ax.factors[0], load, store, tw, n, 1);
    return;
  }
  stage_of<kOdd>(ax.factors[0], load, [&](int i, int c, const Cpx& v) { a[i * kCols + c] = pack(v); }, tw, n, 1);
  __syncthreads();
  int before = ax.factors[0];
  for (int f = 1; f < last; ++f) {
    stage_of<kOdd>(ax.factors[f], [&](int i, int c) { return unpack(a[i * kCols + c]); },
                   [&](int i, int c, const Cpx& v) { b[i * kCols + c] = pack(v); }, tw, n, before);
    before *= ax.factors[f];
    float4* const t = a;
    a = b;
    b = t;
    __syncthreads();
  }
  stage_of<kOdd>(ax.factors[last], [&](int i, int c) { return unpack(a[i * kCols + c]); }, store, tw, n, before);
}

__device__ __forceinline__ void load_twiddles(float4* tw, const SpectrumAxis& ax) {
  for (int j = threadIdx.x; j < ax.n; j += blockDim.x) tw[j] = __ldg(ax.twiddles + j);
}

// Rows 2 p and 2 p + 1 of the field (of `rows` rows of n values) as the real and imaginary parts of
// line p; their half spectra to spec[row][kx], kx <= n / 2.
template <int kOdd>
__global__ void __launch_bounds__(256) k_spectrum_x(const __grid_constant__ SpectrumAxis ax,
                                                     const float* field, int64_t rows,
                                                     float4* __restrict__ spec) {
  extern __shared__ float4 smem[];
  const int n = ax.n, nh = n / 2 + 1;
  float4 *a = smem, *b = smem + n * kCols, *tw = smem + 2 * n * kCols;
  grid_launch_dependents();
  load_twiddles(tw, ax);
  grid_dependency_wait();
  const int64_t row0 = (int64_t)blockIdx.x * 2 * kCols;
  // (the last stage stores into the buffer that it does not read)
  float4* const out = ax.nfactors % 2 ? a : b;
  transform<kOdd>(a, b, tw, ax,
                  [&](int x, int c) {
                    const int64_t r = row0 + 2 * c;
                    return Cpx{{r < rows ? field[r * n + x] : 0.0f, 0.0f},
                               {r + 1 < rows ? field[(r + 1) * n + x] : 0.0f, 0.0f}};
                  },
                  [&](int i, int c, const Cpx& v) { out[i * kCols + c] = pack(v); });
  __syncthreads();
  for (int i = threadIdx.x; i < nh * kCols; i += blockDim.x) {
    const int c = i % kCols, k = i / kCols;
    const int64_t r = row0 + 2 * c;
    if (r >= rows) continue;
    const Cpx p = unpack(out[k * kCols + c]), q = unpack(out[(k == 0 ? 0 : n - k) * kCols + c]);
    const auto half = [](Pair32 v) { return Pair32{0.5f * v.hi, 0.5f * v.lo}; };
    spec[r * nh + k] = pack(Cpx{half(padd(p.re, q.re)), half(psub(p.im, q.im))});
    if (r + 1 < rows) spec[(r + 1) * nh + k] = pack(Cpx{half(padd(p.im, q.im)), half(psub(q.re, p.re))});
  }
}

// Lines of n values `inner` apart: line l = (l / inner, l % inner) starts at (l / inner) n inner +
// l % inner. In place, or |F|^2 (hi, lo) to `power`.
template <int kOdd, bool kPower>
__global__ void __launch_bounds__(256) k_spectrum_lines(const __grid_constant__ SpectrumAxis ax, float4* spec,
                                                         uint32_t lines, FastDiv inner, float2* __restrict__ power,
                                                         unsigned* __restrict__ range) {
  extern __shared__ float4 smem[];
  const int n = ax.n;
  float4 *a = smem, *b = smem + n * kCols, *tw = smem + 2 * n * kCols;
  grid_launch_dependents();
  load_twiddles(tw, ax);
  grid_dependency_wait();
  // (blockDim.x is a multiple of kCols: a thread stays with one line)
  const uint32_t l = blockIdx.x * (uint32_t)kCols + threadIdx.x % kCols;
  const uint32_t o = fastdiv(l, inner);
  const bool mine = l < lines;
  const int64_t at = (int64_t)o * n * inner.d + (l - o * inner.d);
  unsigned seen = 0u;
  transform<kOdd>(a, b, tw, ax,
                  [&](int i, int) { return unpack(mine ? spec[at + (int64_t)i * inner.d] : make_float4(0.0f, 0.0f, 0.0f, 0.0f)); },
                  [&](int i, int, const Cpx& f) {
                    if (!mine) return;
                    if (!kPower) {
                      spec[at + (int64_t)i * inner.d] = pack(f);
                      return;
                    }
                    const Pair32 q = padd(pmul(f.re, f.re), pmul(f.im, f.im));
                    power[at + (int64_t)i * inner.d] = make_float2(q.hi, q.lo);
                    const float x = f.re.hi, y = f.im.hi, most = fmaxf(fabsf(x), fabsf(y));
                    // (a NaN is lost by fmaxf: its sum is not)
                    seen |= (x + y < 0x1p60f && x + y > -0x1p60f && most < 0x1p60f ? 0u : kSpectrumLarge) |
                            (most >= 0x1p-30f ? kSpectrumUsual : 0u) | (most > 0.0f ? kSpectrumNonzero : 0u);
                  });
  if (kPower) {
    seen = __reduce_or_sync(0xffffffffu, seen);
    if ((threadIdx.x & 31) == 0 && (seen & ~*(volatile unsigned*)range)) atomicOr(range, seen);
  }
}

int line_threads(int n) {
  int t = (n / 8) * kCols;
  t = t < 64 ? 64 : (t > 256 ? 256 : (t + 31) / 32 * 32);
  return t;
}
size_t line_smem(int n) { return sizeof(float4) * ((size_t)2 * n * kCols + n); }

template <class Kernel>
cudaError_t allow_smem(Kernel* k, size_t bytes) {
  return bytes <= 48 * 1024 ? cudaSuccess
                            : cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

}  // namespace

bool spectrum_axis(int n, SpectrumAxis* ax) {
  ax->n = n;
  ax->nfactors = 0;
  ax->odd = 0;
  ax->twiddles = nullptr;
  if (n < 1 || n > kMaxLine) return false;
  const int radices[8] = {8, 4, 2, 3, 5, 7, 11, 13};
  for (int r : radices)
    while (n % r == 0) {
      if (r == 3 || r == 5 || r == 7) ax->odd = ax->odd > 1 ? ax->odd : 1;
      if (r > 8) ax->odd = 2;
      ax->factors[ax->nfactors++] = r;
      n /= r;
    }
  return n == 1;
}

std::vector<float> spectrum_twiddles(int n) {
  std::vector<float> t((size_t)4 * n);
  for (int j = 0; j < n; ++j) {
    const double a = -2.0 * 3.14159265358979323846 * j / n;
    const double v[2] = {std::cos(a), std::sin(a)};
    for (int k = 0; k < 2; ++k) {
      t[(size_t)4 * j + 2 * k] = (float)v[k];
      t[(size_t)4 * j + 2 * k + 1] = (float)(v[k] - (double)(float)v[k]);
    }
  }
  return t;
}

cudaError_t launch_power_spectrum(const Geometry& g, const SpectrumAxis (&ax)[3], const float* field, void* spec,
                                  float2* power, unsigned* range, cudaStream_t st) {
  const int64_t rows = (int64_t)g.ny * g.nz;
  const uint32_t nh = g.nx / 2 + 1;
  float4* const s = static_cast<float4*>(spec);
  const auto lines = [&](auto* kernel, const SpectrumAxis& a, uint32_t nlines, uint32_t inner) {
    const size_t smem = line_smem(a.n);
    if (cudaError_t e = allow_smem(kernel, smem)) return e;
    return launch_chained(kernel, (nlines + kCols - 1) / kCols, (unsigned)line_threads(a.n), smem, st, a, s, nlines,
                          make_fastdiv(inner), power, range);
  };
  const auto first = [&](auto* kernel) {
    const size_t smem = line_smem(ax[0].n);
    if (cudaError_t e = allow_smem(kernel, smem)) return e;
    return launch_chained(kernel, (unsigned)((rows + 2 * kCols - 1) / (2 * kCols)), (unsigned)line_threads(ax[0].n), smem,
                          st, ax[0], field, rows, s);
  };
  cudaError_t e = ax[0].odd == 0   ? first(&k_spectrum_x<0>)
                  : ax[0].odd == 1 ? first(&k_spectrum_x<1>)
                                   : first(&k_spectrum_x<2>);
  if (e == cudaSuccess)
    e = ax[1].odd == 0   ? lines(&k_spectrum_lines<0, false>, ax[1], nh * g.nz, nh)
        : ax[1].odd == 1 ? lines(&k_spectrum_lines<1, false>, ax[1], nh * g.nz, nh)
                         : lines(&k_spectrum_lines<2, false>, ax[1], nh * g.nz, nh);
  if (e == cudaSuccess)
    e = ax[2].odd == 0   ? lines(&k_spectrum_lines<0, true>, ax[2], nh * g.ny, nh * g.ny)
        : ax[2].odd == 1 ? lines(&k_spectrum_lines<1, true>, ax[2], nh * g.ny, nh * g.ny)
                         : lines(&k_spectrum_lines<2, true>, ax[2], nh * g.ny, nh * g.ny);
  return e;
}

}  // namespace rflbm_dev
