// Results of the synchronous calls in page-locked host memory (rflbm_host.cu).
#pragma once

#include <cuda_runtime.h>

#include "rflbm_aux.h"

namespace rflbm_dev {

// What the kernels of one handle write in place, so that a synchronous call ends with one
// synchronisation and no copy.
struct HostResults {
  int err;  // set by bounded waits in kernels
  unsigned spectrum_range;
  double stats[kStatOutFields];
  double modes[2 * kQ];
};

// A zeroed block for one handle, and its return. Safe from several threads; a region of blocks is
// freed with its last one.
cudaError_t acquire_host_results(HostResults** out);
void release_host_results(HostResults* p);

}  // namespace rflbm_dev
