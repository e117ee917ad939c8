// The fused stream-and-collide step with TMA staging in flat tiles: for whole boxes of any
// row length from 16 sites, where the row segments of step_tma.cuh do not fit the rows.
//
// A buffer plane is one run of n sites, s = x + nx (y + ny z), and away from the box edges the
// source x - c of site s is s - (c_x + nx c_y + nx ny c_z): a tile of 128 consecutive sites,
// whatever rows they lie in, pulls each population from 128 consecutive sites. So the buffer
// is described to TMA as a 2-D tensor (site, plane), a tile's three populations of one source
// row (c_y, c_z) are one box of three planes, starting at the 16-byte boundary at or before the
// first site needed (a runtime offset of up to 3 or 7 elements into shared memory), and its
// 27 results are one box of 27 planes. No thread is idle but in the last tile, and a row
// length needs no alignment.
//
// What the run misses are the sites at box edges. The boxes are placed by the row (y, z) of the
// tile's middle site, wraps included. A site in a row whose own wraps differ (rows at the y
// edges, and z edges inside a tile) loads the values of the rows concerned into its own slots of
// the tile. The periodic x edge is at the ends of every row: the nine values that the
// first and the last site of a row take from its other end are loaded ahead, one per
// thread over the CTA, while the copies are in flight, and put in their slots. (Left to the
// two threads concerned, these loads would follow the copies in every warp that holds a
// row end.)
//
// The collision, the noise and the waits are those of step_tma.cuh; a site computes the same
// bits.
#pragma once

#include "step_tma.cuh"

namespace rflbm_dev {

constexpr int kFlatW = 128;          // sites per tile
constexpr uint32_t kFlatMinRow = 16;  // at most 9 rows in a tile, 162 values at row ends

// Flat offset from row (y, z) to the row (y - cy, z - cz), with the periodic wraps.
__device__ __forceinline__ int row_shift(int y, int z, int cy, int cz, const Geometry& g) {
  int ys = y - cy, zs = z - cz;
  ys += ys < 0 ? (int)g.ny : 0;
  ys -= ys >= (int)g.ny ? (int)g.ny : 0;
  zs += zs < 0 ? (int)g.nz : 0;
  zs -= zs >= (int)g.nz ? (int)g.nz : 0;
  return (int)g.nx * (ys - y) + (int)g.nxy * (zs - z);
}

// Row coordinates of site s.
struct FlatSite {
  int x, y, z;
};
__device__ __forceinline__ FlatSite flat_site(uint32_t s, const Geometry& g) {
  const uint32_t z = fastdiv(s, g.div_nxy);
  const uint32_t rem = s - z * g.nxy;
  const uint32_t y = fastdiv(rem, g.div_nx);
  return {(int)(rem - y * g.nx), (int)y, (int)z};
}

// Where site 0 of a tile lies in a copy shifted by `shift`: the copy starts at the 16-byte boundary
// at or before the site left of it.
template <int kH>
__device__ __forceinline__ int flat_origin(int shift) {
  return ((shift - 1) & (kH - 1)) + 1;
}

// One tile's input: the copies and the values they miss. Group g = 3 (c_y + 1) + (c_z + 1) and
// position a of its three planes hold plane 3 g + a of the buffer in the pull view; kMirror: the
// planes 26 - (3 g + a) of the flipped view.
template <int kStore, int kThreads, bool kMirror>
struct FlatInput {
  using L = TmaLayout<kStore, kFlatW>;
  using T = typename L::T;
  static constexpr int kH = L::kH;
  static constexpr int kEnds = (2 * 9 * kGroups + kThreads - 1) / kThreads;
  static constexpr uint32_t kCopyBytes = (uint32_t)(kGroups * 3 * L::kSeg * sizeof(T));
  const int* origin;  // per group: element of site 0 in its first plane (shared memory, kGroups values)
  int mid_y, mid_z;   // row of the middle site: the copies' wraps
  bool edge;          // rows at a y edge in the tile (their wraps may differ)
  T end[kEnds];
  int end_at[kEnds];

  static __device__ __forceinline__ int plane(int p) { return kMirror ? kQ - 1 - p : p; }
  // Element of site 0 in position a of group gr, from the group's origin.
  static __device__ __forceinline__ int slot(int gr, int a, int origin) {
    return gr * L::kGroup + (kMirror ? 2 - a : a) * L::kSeg + origin;
  }

  // Issues the copies (threads 0..8) and the loads of the row ends; table: kGroups ints of shared
  // memory, filled when the next barrier has passed.
  __device__ __forceinline__ void start(T* sm, int* table, const CUtensorMap* map, uint64_t* bar, const T* src,
                                        uint32_t s0, uint32_t extra_tx, const Geometry& g) {
    const int t = threadIdx.x;
    origin = table;
    const uint32_t mid = min(s0 + kFlatW / 2, g.n - 1);
    const FlatSite m = flat_site(mid, g);
    mid_y = m.y;
    mid_z = m.z;
    if (t < kGroups) {
      if (t == 0) mbar_arrive_expect_tx(bar, kCopyBytes + extra_tx);
      const int shift = row_shift(mid_y, mid_z, t / 3 - 1, t % 3 - 1, g);
      table[t] = flat_origin<kH>(shift);
      // mirrored: planes 26 - 3 t - 2 .. 26 - 3 t hold positions a = 2, 1, 0
      tma_load_2d(sm + t * L::kGroup, map, (int)s0 + shift - flat_origin<kH>(shift), kMirror ? kQ - 3 - 3 * t : 3 * t,
                  bar);
    }
    const uint32_t row0 = fastdiv(s0, g.div_nx), row1 = fastdiv(min(s0 + kFlatW, g.n) - 1, g.div_nx);
    const int rmid = mid_y + mid_z * (int)g.ny;
    edge = mid_y - (rmid - (int)row0) < 1 || mid_y + ((int)row1 - rmid) > (int)g.ny - 2;
    const int items = (int)(row1 - row0 + 1) * 2 * kGroups;
#pragma unroll
    for (int e = 0; e < kEnds; ++e) {
      const int k = t + e * kThreads;
      end_at[e] = -1;
      end[e] = T();
      if (k >= items) continue;
      const int side = k / kGroups, gr = k - side * kGroups;  // even sides: x = 0, odd: x = nx - 1
      const uint32_t row = row0 + (uint32_t)(side >> 1);
      const int pos = (int)(row * g.nx + ((side & 1) ? g.nx - 1 : 0u) - s0);
      if (pos >= 0 && pos < kFlatW) {
        const int z = (int)fastdiv(row * g.nx, g.div_nxy), y = (int)row - z * (int)g.ny;
        const int cy = gr / 3 - 1, cz = gr % 3 - 1;
        // c_x = +1 pulls x = nx - 1 into x = 0, c_x = -1 pulls x = 0 into x = nx - 1
        const int cx = (side & 1) ? -1 : 1;
        const int64_t from = (int64_t)((int)(row * g.nx) + row_shift(y, z, cy, cz, g)) + ((side & 1) ? 0 : (int)g.nx - 1);
        end[e] = src[(int64_t)plane(3 * gr + cx + 1) * g.ps + from];
        end_at[e] = slot(gr, cx + 1, flat_origin<kH>(row_shift(mid_y, mid_z, cy, cz, g))) + pos - cx;
      }
    }
  }

  // After the copies: the values at the row ends into their slots.
  __device__ __forceinline__ void put_ends(T* sm) const {
#pragma unroll
    for (int e = 0; e < kEnds; ++e)
      if (end_at[e] >= 0) sm[end_at[e]] = end[e];
  }

  // After the copies: site s at tile position pos loads the values of the rows where its wraps are
  // not the middle site's, nine (three source rows of three planes) at a time.
  __device__ __forceinline__ void put_wrapped(T* sm, const T* src, uint32_t s, int pos, const Geometry& g) const {
    if (!edge || s >= g.n) return;
    const FlatSite v = flat_site(s, g);
    const int64_t row = (int64_t)v.z * g.nxy + (int64_t)v.y * g.nx;
#pragma unroll 1
    for (int kind = 0; kind < 4; ++kind) {  // c_y = -1, c_y = +1, c_z = -1, c_z = +1
      const bool of_y = kind < 2;
      const int c = kind & 1 ? 1 : -1;
      const int at = of_y ? v.y : v.z, mid = of_y ? mid_y : mid_z, last = (of_y ? (int)g.ny : (int)g.nz) - 1;
      const int wraps = c > 0 ? 0 : last;
      if ((at == wraps) == (mid == wraps)) continue;
      T val[9];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int cy = of_y ? c : u - 1, cz = of_y ? u - 1 : c, gr = 3 * (cy + 1) + cz + 1;
        const int64_t from = row + row_shift(v.y, v.z, cy, cz, g);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          int xs = v.x - (a - 1);
          xs += xs < 0 ? (int)g.nx : 0;
          xs -= xs >= (int)g.nx ? (int)g.nx : 0;
          val[3 * u + a] = src[(int64_t)plane(3 * gr + a) * g.ps + from + xs];
        }
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int gr = of_y ? 3 * (c + 1) + u : 3 * u + c + 1;
#pragma unroll
        for (int a = 0; a < 3; ++a) sm[slot(gr, a, origin[gr]) + pos - (a - 1)] = val[3 * u + a];
      }
    }
  }

  // Element of population i for tile position 0 (add the position).
  __device__ __forceinline__ int at(int i) const { return at(cx_of(i) + 1, cy_of(i) + 1, cz_of(i) + 1); }
  __device__ __forceinline__ int at(int a, int b, int c) const { return slot(3 * b + c, a, origin[3 * b + c]) - (a - 1); }
};

template <int kStore, int kModel, bool kNoise, bool kGhostNeq, bool kPhiRho0>
__global__ void __launch_bounds__(kFlatW, kModel == kModelBgk || kGhostNeq ? 8 : 9) step_flat(const __grid_constant__ CUtensorMap load_map,
                                                                               const __grid_constant__ CUtensorMap store_map,
                                                                               const StepParams p) {
  using S = Storage<kStore>;
  using In = FlatInput<kStore, kFlatW, false>;
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int table[kGroups];
  T* const sm = reinterpret_cast<T*>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));

  const int t = threadIdx.x;
  const uint32_t s0 = blockIdx.x * (uint32_t)kFlatW, s = s0 + t;
  grid_launch_dependents();
  SiteNoise noise;
  if (kNoise) site_noise_part<0, kPreWaitCalls>(s, p.step, p.replica, p.rk, noise);
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  grid_dependency_wait();

  const T* const src = static_cast<const T*>(p.src);
  In in;
  in.start(sm, table, &load_map, &bar, src, s0, p.test_extra_tx, p.geo);
  if (kNoise) site_noise_part<kPreWaitCalls, 6>(s, p.step, p.replica, p.rk, noise);

  const bool ok = mbar_wait_bounded(&bar, 0, kMaxPolls);
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(p.err, 1);
    mbar_wait_bounded(&bar, 0, kMaxPolls);
    return;
  }
  in.put_ends(sm);
  in.put_wrapped(sm, src, s, t, p.geo);
  __syncthreads();

  float G[3][3][3];
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = S::load(sm[in.at(i) + t], class_of(i), p.ss);
  if (kModel == kModelBgk) {
    const auto reload = [&](int a, int b, int c, float) {
      return S::load(sm[in.at(a, b, c) + t],
                     class_at(a, b, c), p.ss);
    };
    collide_site<kModel, kNoise, kGhostNeq, kPhiRho0>(G, p.cp, noise, reload);
  } else {
    collide_site<kModel, kNoise, kGhostNeq, kPhiRho0>(G, p.cp, noise);
  }

  __syncthreads();  // every input is read: the tile takes the outputs
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    sm[plane_of(i) * kFlatW + t] = S::store(G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1], class_of(i), p.ss);
  fence_proxy_async_smem();
  __syncthreads();
  if (t == 0) {
    tma_store_2d(&store_map, sm, (int)s0, 0);  // clipped at n
    bulk_commit();
    bulk_wait_read();
  }
}

// Two sites per thread (see step_tma_pair). kEven: rows of an even number of sites, where both
// sites of a thread lie in one row and plane c_x = 0 starts at an even element of its copy (one
// aligned pair per read); otherwise every plane is read as two elements.
// Held to 10 CTAs per SM with noise (96 registers; at the 108 the compiler would take, 9 CTAs,
// float16 232x128x64 68.8 against 65.8 us).
template <int kStore, bool kNoise, bool kEven>
__global__ void __launch_bounds__(kFlatW / 2, kNoise ? 10 : 0) step_flat_pair(const __grid_constant__ CUtensorMap load_map,
                                                              const __grid_constant__ CUtensorMap store_map,
                                                              const StepParams p) {
  using S = Storage<kStore>;
  using In = FlatInput<kStore, kFlatW / 2, false>;
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int table[kGroups];
  T* const sm = reinterpret_cast<T*>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));

  const int t = threadIdx.x;
  const uint32_t s0 = blockIdx.x * (uint32_t)kFlatW, s = s0 + 2u * t;
  grid_launch_dependents();
  const PhiloxKey key{p.key0, p.key1};
  PairNoise<kPairPreDrawn, PhiloxKey> noise{s, p.step, p.replica, key};
  if (kNoise) noise.draw();
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  grid_dependency_wait();

  const T* const src = static_cast<const T*>(p.src);
  In in;
  in.start(sm, table, &load_map, &bar, src, s0, p.test_extra_tx, p.geo);
  const bool ok = mbar_wait_bounded(&bar, 0, kMaxPolls);
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(p.err, 1);
    mbar_wait_bounded(&bar, 0, kMaxPolls);
    return;
  }
  in.put_ends(sm);
  in.put_wrapped(sm, src, s, 2 * t, p.geo);
  in.put_wrapped(sm, src, s + 1, 2 * t + 1, p.geo);
  __syncthreads();

  float2 G[3][3][3];
  if constexpr (S::kScaled && !kNoise) {  // (with noise it spills at 96 registers: 300x128x64 84.6 against 83.0 us)
    collide_stored<kStore, kNoise>(
        [&](int a, int b, int c, T (&v)[2]) { stored_pair(sm + in.at(a, b, c) + 2 * t, kEven && a == 1, v); }, p.ss, G,
        p.cp, noise, ScaledWeight<kStore>{p.ss});
  } else {
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const T* const from = sm + in.at(i) + 2 * t;
      float2 v = kEven && cx_of(i) == 0 ? S::load2(from) : S::load1x2(from);
      if (S::kScaled) v = kmul(p.ss.inv_scale[class_of(i)], v);
      G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = v;
    }
    collide_tile<kModelReg, kNoise, false, false>(G, p.cp, noise, ScaledWeight<kStore>{p.ss});
  }

  __syncthreads();
  T* out = sm + 2 * t;
#pragma unroll
  for (int i = 0; i < kQ; ++i) S::store2(out + plane_of(i) * kFlatW, G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1]);
  fence_proxy_async_smem();
  __syncthreads();
  if (t == 0) {
    tma_store_2d(&store_map, sm, (int)s0, 0);
    bulk_commit();
    bulk_wait_read();
  }
}

// ---- the AA pattern in flat tiles (see step_aa.cuh for the two forms)

// Even form: a tile's own 27 planes in, the results back into the slots of the opposite
// directions. No site needs another's values, so there are no box edges.
template <int kStore, int kModel, bool kNoise>
__global__ void __launch_bounds__(kFlatW, kModel == kModelBgk ? 8 : 9) step_flat_aa_even(const __grid_constant__ CUtensorMap map,
                                                                                       const StepParams p) {
  using S = Storage<kStore>;
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  T* const sm = reinterpret_cast<T*>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));

  const int t = threadIdx.x;
  const uint32_t s0 = blockIdx.x * (uint32_t)kFlatW, s = s0 + t;
  grid_launch_dependents();
  SiteNoise noise;
  if (kNoise) site_noise_part<0, kPreWaitCalls>(s, p.step, p.replica, p.rk, noise);
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  grid_dependency_wait();
  if (t == 0) {
    mbar_arrive_expect_tx(&bar, (uint32_t)(kQ * kFlatW * sizeof(T)) + p.test_extra_tx);
    tma_load_2d(sm, &map, (int)s0, 0, &bar);
  }
  if (kNoise) site_noise_part<kPreWaitCalls, 6>(s, p.step, p.replica, p.rk, noise);
  const bool ok = mbar_wait_bounded(&bar, 0, kMaxPolls);
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(p.err, 1);
    mbar_wait_bounded(&bar, 0, kMaxPolls);
    return;
  }

  float G[3][3][3];
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = S::load(sm[plane_of(i) * kFlatW + t], class_of(i), p.ss);
  if (kModel == kModelBgk) {
    const auto reload = [&](int a, int b, int c, float) {
      return S::load(sm[(9 * b + 3 * c + a) * kFlatW + t], class_at(a, b, c), p.ss);
    };
    collide_site<kModel, kNoise, false, false>(G, p.cp, noise, reload);
  } else {
    collide_site<kModel, kNoise, false, false>(G, p.cp, noise);
  }

  __syncthreads();
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    sm[(kQ - 1 - plane_of(i)) * kFlatW + t] =
        S::store(G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1], class_of(i), p.ss);
  fence_proxy_async_smem();
  __syncthreads();
  if (t == 0) {
    tma_store_2d(&map, sm, (int)s0, 0);
    bulk_commit();
    bulk_wait_read();
  }
}

template <int kStore, bool kNoise>
__global__ void __launch_bounds__(kFlatW / 2) step_flat_aa_even_pair(const __grid_constant__ CUtensorMap map,
                                                                      const StepParams p) {
  using S = Storage<kStore>;
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  T* const sm = reinterpret_cast<T*>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));

  const int t = threadIdx.x;
  const uint32_t s0 = blockIdx.x * (uint32_t)kFlatW;
  grid_launch_dependents();
  const PhiloxKey key{p.key0, p.key1};
  PairNoise<kPairPreDrawn, PhiloxKey> noise{s0 + 2u * t, p.step, p.replica, key};
  if (kNoise) noise.draw();
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  grid_dependency_wait();
  if (t == 0) {
    mbar_arrive_expect_tx(&bar, (uint32_t)(kQ * kFlatW * sizeof(T)) + p.test_extra_tx);
    tma_load_2d(sm, &map, (int)s0, 0, &bar);
  }
  const bool ok = mbar_wait_bounded(&bar, 0, kMaxPolls);
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(p.err, 1);
    mbar_wait_bounded(&bar, 0, kMaxPolls);
    return;
  }

  float2 G[3][3][3];
  if constexpr (S::kScaled) {
    collide_stored<kStore, kNoise>(
        [&](int a, int b, int c, T (&v)[2]) { stored_pair(sm + (9 * b + 3 * c + a) * kFlatW + 2 * t, true, v); }, p.ss, G,
        p.cp, noise, ScaledWeight<kStore>{p.ss});
  } else {
#pragma unroll
    for (int i = 0; i < kQ; ++i)
      G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = S::load2(sm + plane_of(i) * kFlatW + 2 * t);
    collide_tile<kModelReg, kNoise, false, false>(G, p.cp, noise, ScaledWeight<kStore>{p.ss});
  }

  __syncthreads();
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    S::store2(sm + (kQ - 1 - plane_of(i)) * kFlatW + 2 * t, G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1]);
  fence_proxy_async_smem();
  __syncthreads();
  if (t == 0) {
    tma_store_2d(&map, sm, (int)s0, 0);
    bulk_commit();
    bulk_wait_read();
  }
}

// Site that population i of a site with neighbours nb is pushed to: x + c_i.
__device__ __forceinline__ uint32_t push_site(const Neighbours& nb, int i) {
  return nb.X[1 - cx_of(i)] + nb.Y[1 - cy_of(i)] + nb.Z[1 - cz_of(i)];
}

// Odd form: the mirrored planes in, the results straight to the neighbours x + c_i. The halo of a
// copy covers slots of other sites that their CTAs overwrite meanwhile; no site uses those.
template <int kStore, int kModel, bool kNoise>
__global__ void __launch_bounds__(kFlatW, kModel == kModelBgk ? 8 : 9) step_flat_aa_odd(const __grid_constant__ CUtensorMap load_map,
                                                                                      const StepParams p) {
  using S = Storage<kStore>;
  using In = FlatInput<kStore, kFlatW, true>;
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int table[kGroups];
  T* const sm = reinterpret_cast<T*>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));

  const int t = threadIdx.x;
  const uint32_t s0 = blockIdx.x * (uint32_t)kFlatW, s = s0 + t;
  grid_launch_dependents();
  SiteNoise noise;
  if (kNoise) site_noise_part<0, kPreWaitCalls>(s, p.step, p.replica, p.rk, noise);
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  grid_dependency_wait();

  T* const buf = static_cast<T*>(p.dst);
  In in;
  in.start(sm, table, &load_map, &bar, buf, s0, p.test_extra_tx, p.geo);
  if (kNoise) site_noise_part<kPreWaitCalls, 6>(s, p.step, p.replica, p.rk, noise);
  const bool ok = mbar_wait_bounded(&bar, 0, kMaxPolls);
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(p.err, 1);
    mbar_wait_bounded(&bar, 0, kMaxPolls);
    return;
  }
  in.put_ends(sm);
  in.put_wrapped(sm, buf, s, t, p.geo);
  __syncthreads();

  float G[3][3][3];
#pragma unroll
  for (int i = 0; i < kQ; ++i)
    G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = S::load(sm[in.at(i) + t], class_of(i), p.ss);
  if (kModel == kModelBgk) {
    const auto reload = [&](int a, int b, int c, float) {
      return S::load(sm[in.at(a, b, c) + t],
                     class_at(a, b, c), p.ss);
    };
    collide_site<kModel, kNoise, false, false>(G, p.cp, noise, reload);
  } else {
    collide_site<kModel, kNoise, false, false>(G, p.cp, noise);
  }
  if (s >= p.geo.n) return;
  const Neighbours nb = neighbours(s, p.geo);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    T* const plane = buf + plane_of(i) * p.geo.ps;
    plane[push_site(nb, i)] = S::store(G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1], class_of(i), p.ss);
  }
}

template <int kStore, bool kNoise, bool kEven>
__global__ void __launch_bounds__(kFlatW / 2) step_flat_aa_odd_pair(const __grid_constant__ CUtensorMap load_map,
                                                                     const StepParams p) {
  using S = Storage<kStore>;
  using In = FlatInput<kStore, kFlatW / 2, true>;
  using T = typename S::T;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ int table[kGroups];
  T* const sm = reinterpret_cast<T*>(smem_raw + ((128u - (smem_addr(smem_raw) & 127u)) & 127u));

  const int t = threadIdx.x;
  const uint32_t s0 = blockIdx.x * (uint32_t)kFlatW, s = s0 + 2u * t;
  grid_launch_dependents();
  const PhiloxKey key{p.key0, p.key1};
  PairNoise<kPairPreDrawn, PhiloxKey> noise{s, p.step, p.replica, key};
  if (kNoise) noise.draw();
  if (t == 0) {
    mbar_init(&bar, 1);
    mbar_init_fence();
  }
  __syncthreads();
  grid_dependency_wait();

  T* const buf = static_cast<T*>(p.dst);
  In in;
  in.start(sm, table, &load_map, &bar, buf, s0, p.test_extra_tx, p.geo);
  const bool ok = mbar_wait_bounded(&bar, 0, kMaxPolls);
  if (__syncthreads_or(!ok)) {
    if (t == 0) atomicOr(p.err, 1);
    mbar_wait_bounded(&bar, 0, kMaxPolls);
    return;
  }
  in.put_ends(sm);
  in.put_wrapped(sm, buf, s, 2 * t, p.geo);
  in.put_wrapped(sm, buf, s + 1, 2 * t + 1, p.geo);
  __syncthreads();

  float2 G[3][3][3];
  if constexpr (S::kScaled) {
    collide_stored<kStore, kNoise>(
        [&](int a, int b, int c, T (&v)[2]) { stored_pair(sm + in.at(a, b, c) + 2 * t, kEven && a == 1, v); }, p.ss, G,
        p.cp, noise, ScaledWeight<kStore>{p.ss});
  } else {
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      const T* const from = sm + in.at(i) + 2 * t;
      G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1] = kEven && cx_of(i) == 0 ? S::load2(from) : S::load1x2(from);
    }
    collide_tile<kModelReg, kNoise, false, false>(G, p.cp, noise, ScaledWeight<kStore>{p.ss});
  }

  if (s >= p.geo.n) return;
  const Neighbours n0 = neighbours(s, p.geo);
  if (kEven) {
    // both sites in one row: x + 1 never wraps from x, x - 1 wraps when x = 0, x + 2 when x + 2 = nx
    const uint32_t x = n0.X[1], xp2 = x + 2u == p.geo.nx ? 0u : x + 2u;
#pragma unroll
    for (int i = 0; i < kQ; ++i) {
      T* const plane = buf + plane_of(i) * p.geo.ps;
      const uint32_t row = n0.Y[1 - cy_of(i)] + n0.Z[1 - cz_of(i)];
      const float2 v = G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1];
      if (cx_of(i) == 0) {
        S::store2(plane + (row + x), v);
      } else {
        plane[row + (cx_of(i) > 0 ? x + 1u : n0.X[2])] = S::pack(v.x);
        plane[row + (cx_of(i) > 0 ? xp2 : x)] = S::pack(v.y);
      }
    }
    return;
  }
  const bool two = s + 1 < p.geo.n;
  const Neighbours n1 = neighbours(two ? s + 1 : s, p.geo);
#pragma unroll
  for (int i = 0; i < kQ; ++i) {
    T* const plane = buf + plane_of(i) * p.geo.ps;
    const float2 v = G[cx_of(i) + 1][cy_of(i) + 1][cz_of(i) + 1];
    plane[push_site(n0, i)] = S::pack(v.x);
    if (two) plane[push_site(n1, i)] = S::pack(v.y);
  }
}

template <class Kernel, class... Args>
cudaError_t launch_flat(Kernel* kernel, int threads, size_t smem, const StepParams& p, cudaStream_t st, const Args&... args) {
  return launch_chained(kernel, (p.geo.n + kFlatW - 1) / kFlatW, (unsigned)threads, smem, st, args..., p);
}

template <int kStore, int kModel, bool kNoise, bool kGhostNeq, bool kPhiRho0>
cudaError_t launch_flat_one(const TmaMaps& m, const StepParams& p, cudaStream_t st) {
  return launch_flat(&step_flat<kStore, kModel, kNoise, kGhostNeq, kPhiRho0>, kFlatW, TmaLayout<kStore, kFlatW>::kBytes, p,
                     st, *m.load, *m.store);
}
template <int kStore, bool kNoise>
cudaError_t launch_flat_pair(const TmaMaps& m, const StepParams& p, cudaStream_t st) {
  return launch_flat(p.geo.nx % 2 ? &step_flat_pair<kStore, kNoise, false> : &step_flat_pair<kStore, kNoise, true>,
                     kFlatW / 2, TmaLayout<kStore, kFlatW>::kBytes, p, st, *m.load, *m.store);
}

template <int kStore, int kModel, bool kNoise>
cudaError_t launch_flat_aa_one(const TmaMaps& m, const StepParams& p, bool odd, cudaStream_t st) {
  if (odd)
    return launch_flat(&step_flat_aa_odd<kStore, kModel, kNoise>, kFlatW, TmaLayout<kStore, kFlatW>::kBytes, p, st, *m.load);
  return launch_flat(&step_flat_aa_even<kStore, kModel, kNoise>, kFlatW, kQ * kFlatW * storage_bytes(kStore) + 128, p, st,
                     *m.store);
}
template <int kStore, bool kNoise>
cudaError_t launch_flat_aa_pair(const TmaMaps& m, const StepParams& p, bool odd, cudaStream_t st) {
  if (odd)
    return launch_flat(
        p.geo.nx % 2 ? &step_flat_aa_odd_pair<kStore, kNoise, false> : &step_flat_aa_odd_pair<kStore, kNoise, true>,
        kFlatW / 2, TmaLayout<kStore, kFlatW>::kBytes, p, st, *m.load);
  return launch_flat(&step_flat_aa_even_pair<kStore, kNoise>, kFlatW / 2, kQ * kFlatW * storage_bytes(kStore) + 128, p, st,
                     *m.store);
}
template <int kStore>
cudaError_t launch_flat_aa(const TmaMaps& m, const StepParams& p, const StepVariant& v, bool odd, cudaStream_t st) {
  if (v.ghost_neq || v.phi_rho0) return cudaErrorInvalidValue;
  if (v.model == kModelBgk)
    return v.noise ? launch_flat_aa_one<kStore, kModelBgk, true>(m, p, odd, st)
                   : launch_flat_aa_one<kStore, kModelBgk, false>(m, p, odd, st);
  if (flat_aa_uses_pairs(v, odd, p.geo.nx))
    return v.noise ? launch_flat_aa_pair<kStore, true>(m, p, odd, st) : launch_flat_aa_pair<kStore, false>(m, p, odd, st);
  return launch_flat_aa_one<kStore, kModelReg, true>(m, p, odd, st);
}

}  // namespace rflbm_dev
