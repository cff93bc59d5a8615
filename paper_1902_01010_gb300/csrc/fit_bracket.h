// Bracket of an FP64 distance |x - med| known by the leading bits of its FP32 value |x - med_f|,
// used by the fit's MAD (ellfit.cu). Host and device code.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define VR_HD __host__ __device__ __forceinline__
#else
#define VR_HD inline
#endif

namespace vr {

// A key is the 22 leading bits below the sign of a non-negative FP32 number: a slice of 2^-14 of
// its size. Infinity's:
constexpr int kDistBits = 22, kDistDrop = 9;
constexpr uint32_t kDistInf = 0x7f800000u >> kDistDrop;

VR_HD double dist_of_key(uint32_t key) {
  const uint32_t b = key << kDistDrop;
  float f;
  memcpy(&f, &b, sizeof(f));
  return (double)f;
}

// [*lo, *hi] holds every FP64 distance whose FP32 form has the key `top`, and with *err, the
// bound on |d_f - d| from the rounding of med and of the difference, some room on either side.
// False where the slice's upper end is infinite, or not wide against *err (med far from the
// distances' size).
VR_HD bool dist_bracket(uint32_t top, double med, double *lo, double *hi, double *err) {
  if (top + 1u >= kDistInf) return false;
  const double blo = dist_of_key(top), bhi = dist_of_key(top + 1u);
  *err = 1.2e-7 * (fabs(med) + bhi);
  *lo = blo - 4.0 * *err;
  *hi = bhi + 4.0 * *err;
  return *err < 0.25 * (bhi - blo);
}

}  // namespace vr
