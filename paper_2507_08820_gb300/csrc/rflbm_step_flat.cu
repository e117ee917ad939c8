// Flat-tile step kernels (step_flat.cuh) for float32 storage, and the dispatch for all storage
// formats.
#include "step_flat.cuh"

namespace rflbm_dev {

// Whole boxes that run in flat tiles. Microseconds per step, float32 with noise unless said, "rows"
// the row-segment kernels, "ragged" those with a ragged last segment, "gather" the general kernel:
//  - rows that no segment width divides, from the size where the tiles' longer latency is hidden
//    (56^3: flat 8.8, gather 7.6; without noise 72^3 12.9 and 9.7, 80^3 15.0 and 15.7; 16-bit without
//    noise 60^3 8.3 and 7.5, 66^3 8.6 and 9.0): 100^3 flat 38.0, ragged 42.7, gather 42.3, float16
//    39.7, -, 43.8; 200^3 269, 326, 316, float16 272, 537, 340; 150x110x70 42.9, -, 48.3. Ragged segments
//    stay where they are wide and nearly full (376x128x64 102.9 against 103.6, 248x128x64 69.7 and 69.9, AA
//    75.3 and 76.0; 232x128x64, 10 % idle threads, 69.1 and 65.7), wide with 16-bit storage without
//    noise (120x128x128 34.5 against 36.8), and for smaller fluctuating ping-pong boxes (60^3: ragged 9.7,
//    flat 10.5).
//  - rows in segments of 32 sites, one warp or half of one: 160x128x128 flat 90.7, rows 98.4, float16
//    93.8 against 159.8, AA 97.3 against 138.3
//  - rows in segments of 96 sites where two sites per thread leave a warp and a half:
//    96x128x128 float16 58.5 against 67.0, 288x96x96 AA 98.1 against 107.2 (its odd steps)
//  - rows in several segments of 64 sites, the fluctuating ping-pong step: 320x128x128 176.8
//    against 186.0; rows of one segment are as fast (64x128x128 39.3 against 39.2)
bool flat_pays(const Geometry& g, const StepVariant& v, bool aa) {
  if (g.nx < kFlatMinRow) return false;
  const bool f32 = v.storage == kStoreF32;
  switch (tma_segment_width(g.nx)) {
    case 0: {
      const uint64_t nx = g.nx, w = (uint64_t)tma_ragged_width(g.nx, storage_bytes(v.storage));
      const bool wide = w >= 128, full = wide && (nx + w - 1) / w * w * 30 <= nx * 31;
      if (full || (wide && !f32 && !v.noise && !aa)) return false;
      if (!v.noise) return g.n >= (f32 ? 450000u : 230000u);
      return g.n >= (w && f32 && !aa ? 250000u : 200000u);
    }
    case 32: return g.n >= 200000u;
    case 64: return g.n >= 200000u && f32 && v.noise && !aa && g.nx > 64;
    case 96: return g.n >= 200000u && v.noise && v.model == kModelReg && (f32 ? aa && g.nx > 96 : true);
    default: return false;
  }
}

bool flat_aa_uses_pairs(const StepVariant& v, bool odd, uint32_t nx) {
  if (tma_uses_pairs(v)) return true;
  // the fluctuating float32 odd steps, as in the row-segment form (aa_uses_pairs): 300x300x100
  // 315.0 against 323.8 us per step
  return odd && nx % 2 == 0 && v.model == kModelReg && !v.ghost_neq && !v.phi_rho0 && v.noise;
}

uint32_t flat_load_sites(int storage) {
  return kFlatW + 2 * (storage == kStoreF32 ? Storage<kStoreF32>::kHalo : Storage<kStoreF16>::kHalo);
}
uint32_t flat_store_sites() { return kFlatW; }

cudaError_t launch_step_flat(const TmaMaps& m, const StepParams& p, const StepVariant& v, cudaStream_t st) {
  if (v.storage != kStoreF32) return launch_step_flat_16(m, p, v, st);
  constexpr int F = kStoreF32;
  if (tma_uses_pairs(v)) return launch_flat_pair<F, false>(m, p, st);  // kT = 0
  if (v.model == kModelBgk) {
    if (!v.noise) return launch_flat_one<F, kModelBgk, false, false, false>(m, p, st);
    return v.phi_rho0 ? launch_flat_one<F, kModelBgk, true, false, true>(m, p, st)
                      : launch_flat_one<F, kModelBgk, true, false, false>(m, p, st);
  }
  if (!v.noise) return launch_flat_one<F, kModelReg, false, true, false>(m, p, st);  // (omega_g != 1)
  if (v.ghost_neq) {
    return v.phi_rho0 ? launch_flat_one<F, kModelReg, true, true, true>(m, p, st)
                      : launch_flat_one<F, kModelReg, true, true, false>(m, p, st);
  }
  return v.phi_rho0 ? launch_flat_one<F, kModelReg, true, false, true>(m, p, st)
                    : launch_flat_one<F, kModelReg, true, false, false>(m, p, st);
}

}  // namespace rflbm_dev
