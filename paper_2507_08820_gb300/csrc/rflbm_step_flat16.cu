// Flat-tile step kernels (step_flat.cuh) for 16-bit storage, the paper's configuration only.
#include "step_flat.cuh"

namespace rflbm_dev {

template <int kStore>
static cudaError_t launch_store(const TmaMaps& m, const StepParams& p, const StepVariant& v, cudaStream_t st) {
  if (v.model == kModelBgk)
    return v.noise ? launch_flat_one<kStore, kModelBgk, true, false, false>(m, p, st)
                   : launch_flat_one<kStore, kModelBgk, false, false, false>(m, p, st);
  return v.noise ? launch_flat_pair<kStore, true>(m, p, st) : launch_flat_pair<kStore, false>(m, p, st);
}

cudaError_t launch_step_flat_16(const TmaMaps& m, const StepParams& p, const StepVariant& v, cudaStream_t st) {
  if (v.ghost_neq || v.phi_rho0) return cudaErrorInvalidValue;
  if (v.storage == kStoreF16) return launch_store<kStoreF16>(m, p, v, st);
  if (v.storage == kStoreBF16) return launch_store<kStoreBF16>(m, p, v, st);
  return cudaErrorInvalidValue;
}

}  // namespace rflbm_dev
