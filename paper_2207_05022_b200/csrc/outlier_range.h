// The outlier test of a unit (Section 6: log-likelihood under its Gaussian below -4) and the fp32 values that pass it.
// Plain arithmetic, also compiled for the host by the tests.
#pragma once
#include <math.h>

#include "host_device.h"

namespace sti {

// inv2var = 1 / (2 var); with zero variance c0 is +inf and 0 * inf is NaN, which compares false: no outliers
STI_HOST_DEVICE bool is_outlier(float x, double mu, double inv2var, double c0) {
  const double d = static_cast<double>(x) - mu;
  const double ll = c0 - d * d * inv2var;
  return ll < -4.0;
}

// The test is monotone in |x - mu|, so the values that pass it are one run of fp32 numbers, and its ends lie at the rounded
// thresholds mu +- radius, give or take a few units in the last place.  An end is looked for among the kEndCandidates
// consecutive fp32 numbers around a threshold, numbered away from the mean, by testing all of them at once (a lane each):
// the last inlier if an outlier follows it, else the answer is -1 and the caller has to test every weight - the run
// is empty (fp32 numbers near the mean are wider apart than the interval), the radius has cancelled (deviations near 21.8,
// where c0 reaches -4), or the threshold is so close to zero that its rounding error spans very many fp32 numbers.
constexpr int kEndCandidates = 16;

// Number `i` around threshold `t` of the side `sign` (+1: the largest inlier is looked for, -1: the smallest).
STI_HOST_DEVICE float end_candidate(float t, int i, int sign) {
  union { float f; unsigned u; } v;
  v.f = t;
  unsigned key = (v.u & 0x80000000u) ? ~v.u : (v.u | 0x80000000u);         // ascending with the value
  key += static_cast<unsigned>(sign * (i - kEndCandidates / 2));
  v.u = (key & 0x80000000u) ? (key & 0x7fffffffu) : ~key;
  return v.f;
}
// `inliers`: bit i = candidate i is one.
STI_HOST_DEVICE int end_index(unsigned inliers) {
  if (inliers == 0u || inliers >> (kEndCandidates - 1) != 0u) return -1;
#if defined(__CUDA_ARCH__)
  return 31 - __clz(static_cast<int>(inliers));
#else
  return 31 - __builtin_clz(inliers);
#endif
}

}  // namespace sti
