// Equilibrium-statistics diagnostics (off the timed path): per-mode sums for the
// fluctuation-dissipation check of every Table II mode, and the static structure factor
// S(|k|) of the hydrodynamic fields by FFT and spherical shell averaging (Sec. III).
#include <cufft.h>

#include "rflbm_diag.h"
#include "tma.cuh"
#include "wide.cuh"

namespace rflbm_dev {

constexpr int kDiagBlock = 256;

// All 27 Hermite moments of the shifted populations of one tile G[a][b][c] (Eq. 5 with
// the tensor-product basis of Table II): M[p][q][r] = sum g h_p(c_x) h_q(c_y) h_r(c_z).
__device__ __forceinline__ void all_moments(const float (&G)[3][3][3], float (&M)[3][3][3]) {
  float X[3][3][3];  // [p][b][c]
#pragma unroll
  for (int b = 0; b < 3; ++b)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float s0 = G[0][b][c] + G[1][b][c] + G[2][b][c];
      X[0][b][c] = s0;
      X[1][b][c] = G[2][b][c] - G[0][b][c];
      X[2][b][c] = fmaf(-1.0f / 3.0f, s0, G[2][b][c] + G[0][b][c]);
    }
  float Y[3][3][3];  // [p][q][c]
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float s0 = X[p][0][c] + X[p][1][c] + X[p][2][c];
      Y[p][0][c] = s0;
      Y[p][1][c] = X[p][2][c] - X[p][0][c];
      Y[p][2][c] = fmaf(-1.0f / 3.0f, s0, X[p][2][c] + X[p][0][c]);
    }
#pragma unroll
  for (int p = 0; p < 3; ++p)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float s0 = Y[p][q][0] + Y[p][q][1] + Y[p][q][2];
      M[p][q][0] = s0;
      M[p][q][1] = Y[p][q][2] - Y[p][q][0];
      M[p][q][2] = fmaf(-1.0f / 3.0f, s0, Y[p][q][2] + Y[p][q][0]);
    }
}

template <int kStore>
__device__ __forceinline__ void gather_tile(const typename Storage<kStore>::T* __restrict__ src,
                                            const Geometry& g, const StoreScale& ss, uint32_t s,
                                            float (&G)[3][3][3]) {
  const PopSlots slots(s, g);
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] =
        Storage<kStore>::load(src[slots(i)], class_of(i), ss);
}

// Each thread accumulates up to kDiagSitesPerThread sites in float32, then the block sums
// its 54 values into one FP64 partial slot: eight threads per column, each adding 32 of the
// block's 256 values as a RunningSum, so that a column takes 40 FP64 operations per block.
// (Warp shuffles in FP64 took 270 lane operations per value of a block and bound the kernel:
// 128^3 float32 took 170 us, and takes 59 us.) Bound by the 108 bytes read per site.
constexpr int kModePitch = kDiagBlock + 8;  // columns of a warp's four groups of eight in distinct banks
template <int kStore>
__global__ void __launch_bounds__(kDiagBlock, 2) k_mode_sums(Geometry g, StoreScale ss,
                                                          const typename Storage<kStore>::T* __restrict__ src,
                                                          double* __restrict__ partials) {
  float acc[2 * kQ];
#pragma unroll
  for (int k = 0; k < 2 * kQ; ++k) acc[k] = 0.0f;
  const int64_t base = (int64_t)blockIdx.x * kDiagBlock * kDiagSitesPerThread;
#pragma unroll 1
  for (int j = 0; j < kDiagSitesPerThread; ++j) {
    const int64_t s = base + (int64_t)j * kDiagBlock + threadIdx.x;
    if (s >= g.n) break;
    float G[3][3][3], M[3][3][3];
    gather_tile<kStore>(src, g, ss, (uint32_t)s, G);
    all_moments(G, M);
#pragma unroll
    for (int p = 0; p < 3; ++p)
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int k = mode_of(p, q, r);
          acc[k] += M[p][q][r];
          acc[kQ + k] = fmaf(M[p][q][r], M[p][q][r], acc[kQ + k]);
        }
  }
  __shared__ float sh[kQ][kModePitch];
#pragma unroll
  for (int half = 0; half < 2; ++half) {
    if (half) __syncthreads();
#pragma unroll
    for (int k = 0; k < kQ; ++k) sh[k][threadIdx.x] = acc[half * kQ + k];
    __syncthreads();
    const int col = threadIdx.x >> 3, part = threadIdx.x & 7;
    double v = 0.0;
    if (col < kQ) {
      RunningSum r;
      bool big = false;
#pragma unroll 8
      for (int j = 0; j < kDiagBlock / 8; ++j) {
        const float x = sh[col][part + 8 * j];
        r.add(x);
        big = big || !(fabsf(x) < 0x1p100f);
      }
      v = r.value();
      if (big) {  // infinities, NaN and sums that could overflow float32
        v = 0.0;
        for (int j = 0; j < kDiagBlock / 8; ++j) v += (double)sh[col][part + 8 * j];
      }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (col < kQ && part == 0) partials[(int64_t)blockIdx.x * 2 * kQ + half * kQ + col] = v;
  }
}

// Column sums of a row-major array in a fixed order: a block per column, thread t adds rows
// t, t + 256, ..., then a fixed tree.
__global__ void __launch_bounds__(kDiagBlock) k_reduce_columns(const double* partials, int64_t rows, int cols,
                                 double* __restrict__ out, unsigned* range = nullptr,
                                 unsigned* range_out = nullptr) {
  __shared__ double sh[kDiagBlock / 32];
  grid_dependency_wait();
  const int col = blockIdx.x;
  if (range && col == 0 && threadIdx.x == 0) {
    *range_out = *range;
    *range = 0u;
  }
  double v = 0.0;
  for (int64_t r = threadIdx.x; r < rows; r += kDiagBlock) v += partials[r * cols + col];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kDiagBlock / 32; ++w) v += sh[w];
    out[col] = v;
  }
}

// Field value of one site, float32 sums of the shifted populations (out in float32, or in FP64 for
// cuFFT):
// 0 rho - rho0, 1..3 rho u, 4..9 Pi = a^(2) (xx, yy, zz, xy, xz, yz). One instance per field,
// its weights compiled in (selected per population at run time they took 92 us at 128^3
// float32); bound by the 108 bytes read and 8 written per site.
template <int kStore, int kField, class Out>
__global__ void __launch_bounds__(kDiagBlock) k_field(Geometry g, StoreScale ss,
                                                      const typename Storage<kStore>::T* src,
                                                      Out* __restrict__ out) {
  grid_launch_dependents();
  grid_dependency_wait();
  const int64_t s = (int64_t)blockIdx.x * kDiagBlock + threadIdx.x;
  if (s >= g.n) return;
  const PopSlots slots((uint32_t)s, g);
  float v = 0.0f, drho = 0.0f;
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    const float x = Storage<kStore>::load(src[slots(i)], class_of(i), ss);
    const int c[3] = {cx_of(i), cy_of(i), cz_of(i)};
    const float w = kField == 0  ? 1.0f
                    : kField < 4 ? (float)c[(kField - 1) % 3]
                    : kField < 7 ? (float)(c[(kField - 4) % 3] * c[(kField - 4) % 3])
                                 : (float)(c[kField == 9 ? 1 : 0] * c[kField == 7 ? 1 : 2]);
    v = fmaf(w, x, v);
    drho += x;
  }
  // Pi_aa = sum g c_a^2 - drho / 3 (the rest state drops out)
  if (kField >= 4 && kField <= 6) v -= drho * (1.0f / 3.0f);
  out[s] = (Out)v;
}

// Shell of a wave vector: round(L |k| / 2 pi) with L |k| / 2 pi = L sqrt(fx^2 + fy^2 + fz^2), k_a / L_a =
// f_a, rounded as the FP64 expression does. The float32 value decides unless it lies within
// its error (a few 2^-24 relative) of a boundary between shells.
__device__ __forceinline__ int shell_of(int kx, int ky, int kz, const Geometry& g, double L) {
  const float Lf = (float)L;
  const float x = (float)kx * (Lf / (float)g.nx), y = (float)ky * (Lf / (float)g.ny), z = (float)kz * (Lf / (float)g.nz);
  const float t = sqrtf(fmaf(x, x, fmaf(y, y, z * z)));
  const float n = rintf(t);
  if (fabsf(fabsf(t - n) - 0.5f) > fmaf(t, 2e-6f, 1e-6f)) return (int)n;
  const double fx = (double)kx / g.nx, fy = (double)ky / g.ny, fz = (double)kz / g.nz;
  return (int)llrint(L * sqrt(fx * fx + fy * fy + fz * fz));
}

// |F|^2 of one entry of a spectrum and the sums of a scan: float32 pairs where they are given, FP64
// for cuFFT's complex values.
__device__ __forceinline__ double power_of(const cufftDoubleComplex& c) { return fma(c.x, c.x, c.y * c.y); }
__device__ __forceinline__ Pair32 power_of(float2 p) { return {p.x, p.y}; }
__device__ __forceinline__ double twice(double v) { return 2.0 * v; }
__device__ __forceinline__ Pair32 twice(Pair32 v) { return {2.0f * v.hi, 2.0f * v.lo}; }
__device__ __forceinline__ double scan_add(double a, double b) { return a + b; }
__device__ __forceinline__ Pair32 scan_add(Pair32 a, Pair32 b) { return padd(a, b); }
__device__ __forceinline__ double from_lane(double v, int o) { return __shfl_up_sync(0xffffffffu, v, o); }
__device__ __forceinline__ Pair32 from_lane(Pair32 v, int o) {
  return {__shfl_up_sync(0xffffffffu, v.hi, o), __shfl_up_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double fp64_of(double v) { return v; }
__device__ __forceinline__ double fp64_of(Pair32 v) { return (double)v.hi + (double)v.lo; }

// Shell sums of |F(k)|^2 / N over the half spectrum of a real transform (kx = 0 .. nx/2),
// each non-redundant vector counted twice. Shell n = round(|k| L / 2 pi) with
// L = max(nx, ny, nz). The vectors (kx, +-ky, +-kz) lie in one shell: a thread adds these up to
// four entries first, and shells, scan and bins take a quarter of the work (128^3: 17.5 -> 10.8 us).
// The sums are reproducible bit for bit: each warp owns a row of
// shell bins in shared memory. Along a spectrum row (ky, kz) the shell grows with kx, so the
// vectors of one shell are neighbours: a segmented scan over the warp's lanes adds them up
// (a fixed tree of float32 pairs), and the last lane of each run adds the run to its FP64 bin, one
// spectrum row after another. The rows are then summed in warp order into the block's partial
// row. (Counts are integers, exact in any order.) Four FP64 operations per warp of vectors. Before the
// four were added first, 128^3 took 190 us with the shell computed in FP64 (three quotients and a root) and
// the lanes adding to the bins one after another, 28 us with the scan in FP64. (Four blocks per SM: the
// grid's, in one wave.)
template <class Entry>
__global__ void __launch_bounds__(kDiagBlock, 4) k_shell_bins(Geometry g, FastDiv div_nxh, FastDiv div_nyh,
                                                           const Entry* spec, int nshell,
                                                           double* __restrict__ partials) {
  constexpr int kWarps = kDiagBlock / 32;
  extern __shared__ double bins[];  // [kWarps][nshell] sums, then [nshell] counts
  unsigned* const counts = reinterpret_cast<unsigned*>(bins + (size_t)kWarps * nshell);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int j = threadIdx.x; j < kWarps * nshell; j += kDiagBlock) bins[j] = 0.0;
  for (int j = threadIdx.x; j < nshell; j += kDiagBlock) counts[j] = 0u;
  grid_launch_dependents();
  __syncthreads();
  grid_dependency_wait();
  double* const mine = bins + (size_t)wid * nshell;
  const int nxh = g.nx / 2 + 1;
  const int nyh = g.ny / 2 + 1, nzh = g.nz / 2 + 1;
  const int64_t total = (int64_t)nzh * nyh * nxh;
  const double L = (double)max(g.nx, max(g.ny, g.nz));
  const unsigned upto = 0xffffffffu >> (31 - lane);  // lanes 0 .. lane
  const int64_t stride = (int64_t)gridDim.x * kDiagBlock;
  for (int64_t wbase = (int64_t)blockIdx.x * kDiagBlock + 32 * wid; wbase < total; wbase += stride) {
    const int64_t idx = wbase + lane;  // warp-uniform trip count
    int shell = nshell;
    uint32_t row = 0xffffffffu;
    decltype(power_of(Entry())) v{};
    bool self = false;
    unsigned images = 1;
    if (idx < total) {
      row = fastdiv((uint32_t)idx, div_nxh);
      const int kx = (int)((uint32_t)idx - row * (uint32_t)nxh);
      const int kz = (int)fastdiv(row, div_nyh);
      const int ky = (int)(row - (uint32_t)kz * nyh);
      const int my = ky ? (int)g.ny - ky : 0, mz = kz ? (int)g.nz - kz : 0;  // of -ky and -kz
      const auto at = [&](int y, int z) { return power_of(spec[((int64_t)z * g.ny + y) * nxh + kx]); };
      v = at(ky, kz);
      if (my != ky) v = scan_add(v, at(my, kz));
      if (mz != kz) v = scan_add(v, my != ky ? scan_add(at(ky, mz), at(my, mz)) : at(ky, mz));
      images = (my != ky ? 2u : 1u) * (mz != kz ? 2u : 1u);
      shell = min(nshell, shell_of(kx, ky, kz, g, L));
      self = (kx == 0) || ((g.nx % 2 == 0) && kx == (int)g.nx / 2);
      if (!self) v = twice(v);
    }
    const int before = __shfl_up_sync(0xffffffffu, shell, 1);
    const uint32_t row_before = __shfl_up_sync(0xffffffffu, row, 1);
    const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || before != shell || row_before != row);
    const unsigned selfs = __ballot_sync(0xffffffffu, self);
    const int start = 31 - __clz(heads & upto);  // first lane of this lane's run
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const auto t = from_lane(v, o);
      if (lane - o >= start) v = scan_add(v, t);
    }
    const bool tail = (lane == 31 || ((heads >> (lane + 1)) & 1u)) && shell < nshell;
    if (tail) {
      const unsigned run = upto & ~((1u << start) - 1u);
      atomicAdd(&counts[shell], images * (2u * (unsigned)__popc(run) - (unsigned)__popc(run & selfs)));
    }
    // runs of one spectrum row are of different shells
    const uint32_t first = __shfl_sync(0xffffffffu, row, 0);
    const uint32_t end = min(fastdiv((uint32_t)min(wbase + 31, total - 1), div_nxh), first + 31u);
    const double run_sum = fp64_of(v);
    for (uint32_t r = first; r <= end; ++r) {
      if (tail && row == r) mine[shell] += run_sum;
      __syncwarp();
    }
  }
  __syncthreads();
  const double inv_n = 1.0 / (double)g.n;
  for (int j = threadIdx.x; j < nshell; j += kDiagBlock) {
    double sum = 0.0;
    for (int k = 0; k < kWarps; ++k) sum += bins[(size_t)k * nshell + j];
    sum *= inv_n;
    partials[(int64_t)blockIdx.x * 2 * nshell + j] = sum;
    partials[(int64_t)blockIdx.x * 2 * nshell + nshell + j] = (double)counts[j];
  }
}

int64_t mode_sum_blocks(const Geometry& g) {
  const int64_t per = (int64_t)kDiagBlock * kDiagSitesPerThread;
  return (g.n + per - 1) / per;
}

template <int K>
using DT = typename Storage<K>::T;

cudaError_t launch_mode_sums(const Geometry& g, const StoreScale& ss, int kind, const void* src,
                             double* partials, double* out54, cudaStream_t st) {
  const int64_t blocks = mode_sum_blocks(g);
  switch (kind) {
    case kStoreF32: k_mode_sums<kStoreF32><<<(unsigned)blocks, kDiagBlock, 0, st>>>(g, ss, (const DT<kStoreF32>*)src, partials); break;
    case kStoreF16: k_mode_sums<kStoreF16><<<(unsigned)blocks, kDiagBlock, 0, st>>>(g, ss, (const DT<kStoreF16>*)src, partials); break;
    case kStoreBF16: k_mode_sums<kStoreBF16><<<(unsigned)blocks, kDiagBlock, 0, st>>>(g, ss, (const DT<kStoreBF16>*)src, partials); break;
    default: return cudaErrorInvalidValue;
  }
  if (cudaError_t e = cudaGetLastError()) return e;
  return launch_chained(&k_reduce_columns, 2u * kQ, kDiagBlock, 0, st, partials, blocks, 2 * kQ, out54, nullptr, nullptr);
}

template <int kStore, int kField, class Out>
static cudaError_t launch_field_at(const Geometry& g, const StoreScale& ss, const void* src, int field, Out* out,
                                   cudaStream_t st) {
  if constexpr (kField > 9) {
    return cudaErrorInvalidValue;
  } else {
    if (field != kField) return launch_field_at<kStore, kField + 1>(g, ss, src, field, out, st);
    const unsigned blocks = (unsigned)(((int64_t)g.n + kDiagBlock - 1) / kDiagBlock);
    return launch_chained(&k_field<kStore, kField, Out>, blocks, kDiagBlock, 0, st, g, ss, (const DT<kStore>*)src, out);
  }
}

template <class Out>
static cudaError_t launch_field_as(const Geometry& g, const StoreScale& ss, int kind, const void* src, int field, Out* out,
                                   cudaStream_t st) {
  switch (kind) {
    case kStoreF32: return launch_field_at<kStoreF32, 0>(g, ss, src, field, out, st);
    case kStoreF16: return launch_field_at<kStoreF16, 0>(g, ss, src, field, out, st);
    case kStoreBF16: return launch_field_at<kStoreBF16, 0>(g, ss, src, field, out, st);
    default: return cudaErrorInvalidValue;
  }
}
cudaError_t launch_field(const Geometry& g, const StoreScale& ss, int kind, const void* src, int field, float* out,
                         cudaStream_t st) {
  return launch_field_as(g, ss, kind, src, field, out, st);
}
cudaError_t launch_field(const Geometry& g, const StoreScale& ss, int kind, const void* src, int field, double* out,
                         cudaStream_t st) {
  return launch_field_as(g, ss, kind, src, field, out, st);
}

template <class Entry>
static cudaError_t launch_bins(const Geometry& g, const Entry* spec, int nshell, int blocks, double* partials, double* out,
                               unsigned* range, unsigned* range_out, cudaStream_t st) {
  // kDiagBlock / 32 rows of sums + one row of counts: up to 221 KB at nshell = 3072
  const size_t smem = sizeof(double) * (size_t)(kDiagBlock / 32 + 1) * (size_t)nshell;
  if (smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_shell_bins<Entry>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (cudaError_t e = launch_chained(&k_shell_bins<Entry>, (unsigned)blocks, kDiagBlock, smem, st, g,
                                     make_fastdiv(g.nx / 2 + 1), make_fastdiv(g.ny / 2 + 1), spec, nshell, partials))
    return e;
  return launch_chained(&k_reduce_columns, 2u * nshell, kDiagBlock, 0, st, partials, (int64_t)blocks, 2 * nshell, out, range,
                        range_out);
}
cudaError_t launch_shell_bins(const Geometry& g, const void* spec, int nshell, int blocks,
                              double* partials, double* out, cudaStream_t st) {
  return launch_bins(g, (const cufftDoubleComplex*)spec, nshell, blocks, partials, out, nullptr, nullptr, st);
}
cudaError_t launch_power_bins(const Geometry& g, const float2* power, int nshell, int blocks, double* partials,
                              double* out, unsigned* range, unsigned* range_out, cudaStream_t st) {
  return launch_bins(g, power, nshell, blocks, partials, out, range, range_out, st);
}

}  // namespace rflbm_dev
