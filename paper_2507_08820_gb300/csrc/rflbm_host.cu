// Page-locked result blocks of the handles, from regions shared by them: allocating page-locked
// memory for one handle costs 170 us, a tenth of creating a small box.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>
#include <vector>

#include "rflbm_host.h"

namespace rflbm_dev {

namespace {

constexpr int kBlocks = 64;  // per region (one bit each)
constexpr size_t kBlockBytes = (sizeof(HostResults) + 127) / 128 * 128;

struct Region {
  char* base;
  unsigned long long used;
};
std::mutex g_mutex;
std::vector<Region> g_regions;

// False after the device that a region was allocated on has been reset: its memory is gone.
bool alive(const Region& r) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, r.base) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeHost;
}

}  // namespace

cudaError_t acquire_host_results(HostResults** out) {
  *out = nullptr;
  std::lock_guard<std::mutex> lock(g_mutex);
  for (size_t k = 0; k < g_regions.size();) {
    Region& r = g_regions[k];
    if (!alive(r)) {
      g_regions.erase(g_regions.begin() + (ptrdiff_t)k);
      continue;
    }
    if (~r.used) {
      const int b = __builtin_ctzll(~r.used);
      r.used |= 1ull << b;
      *out = reinterpret_cast<HostResults*>(r.base + b * kBlockBytes);
      break;
    }
    ++k;
  }
  if (!*out) {
    Region r{nullptr, 1ull};
    if (cudaError_t e = cudaHostAlloc((void**)&r.base, kBlocks * kBlockBytes, cudaHostAllocPortable)) return e;
    g_regions.push_back(r);
    *out = reinterpret_cast<HostResults*>(r.base);
  }
  std::memset(*out, 0, sizeof(HostResults));
  return cudaSuccess;
}

void release_host_results(HostResults* p) {
  if (!p) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  for (size_t k = 0; k < g_regions.size(); ++k) {
    Region& r = g_regions[k];
    const char* const c = reinterpret_cast<const char*>(p);
    if (c < r.base || c >= r.base + kBlocks * kBlockBytes) continue;
    r.used &= ~(1ull << ((size_t)(c - r.base) / kBlockBytes));
    if (!r.used) {
      cudaFreeHost(r.base);
      g_regions.erase(g_regions.begin() + (ptrdiff_t)k);
    }
    return;
  }
}

}  // namespace rflbm_dev
