// The in-place AA steps in flat tiles (step_flat.cuh), all storage formats.
#include "step_flat.cuh"

namespace rflbm_dev {

cudaError_t launch_step_flat_aa(const TmaMaps& m, const StepParams& p, const StepVariant& v, bool odd, cudaStream_t st) {
  switch (v.storage) {
    case kStoreF32: return launch_flat_aa<kStoreF32>(m, p, v, odd, st);
    case kStoreF16: return launch_flat_aa<kStoreF16>(m, p, v, odd, st);
    case kStoreBF16: return launch_flat_aa<kStoreBF16>(m, p, v, odd, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace rflbm_dev
