// The power spectrum of one field per site (rflbm_spectrum.cu).
#pragma once

#include <vector>

#include "rflbm_internal.h"

namespace rflbm_dev {

// One axis of the transform: its length, the radices of its stages and its table of twiddle
// factors exp(-2 pi i j / n) (device memory, n x (re hi, re lo, im hi, im lo)).
struct SpectrumAxis {
  int n, nfactors;
  int factors[12];
  int odd;   // 0: powers of two, 1: radices 3, 5 or 7 among them, 2: 11 or 13
  const float4* twiddles;
};

// Fills *ax for length n (no table yet); false when n is above 768 or has a prime factor above 13.
bool spectrum_axis(int n, SpectrumAxis* ax);
std::vector<float> spectrum_twiddles(int n);

// What *range tells after a transform, as bits: some |F| is 2^60 or more or not finite; some |F| is
// 2^-30 or more; some |F| is not zero. With kSpectrumLarge, or with kSpectrumNonzero alone, the
// squares leave the range of float32 and the spectrum has to be taken in FP64 (spectrum_usable).
enum : unsigned { kSpectrumLarge = 1u, kSpectrumUsual = 2u, kSpectrumNonzero = 4u };
inline bool spectrum_usable(unsigned range) {
  return !(range & kSpectrumLarge) && ((range & kSpectrumUsual) || !(range & kSpectrumNonzero));
}

// |F|^2 (hi, lo) of the half spectrum, [kz][ky][kx], kx <= nx / 2, from the field (one float per site). spec
// holds 16 bytes per value; power may be the field's memory.
cudaError_t launch_power_spectrum(const Geometry& g, const SpectrumAxis (&ax)[3], const float* field, void* spec,
                                  float2* power, unsigned* range, cudaStream_t st);

}  // namespace rflbm_dev
