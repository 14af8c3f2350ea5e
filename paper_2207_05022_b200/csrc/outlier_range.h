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

// The test is monotone in |x - mu|, so the values that pass it are one run of fp32 numbers.  From `t`, the rounded
// threshold mu +- radius, to the end of that run on the side of `away` (+-INFINITY): towards the mean while t is an outlier,
// then away from it while the next value is not.
// The threshold is good to a few units in its last place, so this is a step or two - unless the run is empty (fp32 numbers
// near the mean are wider apart than the interval), the radius has cancelled (deviations near 21.8, where c0 reaches -4)
// or the threshold lies so close to zero that its rounding error spans very many fp32 numbers.  Then the steps run out and
// the answer is false: the caller has to test every weight instead.
constexpr int kThresholdSteps = 32;
STI_HOST_DEVICE bool extreme_inlier(float away, double mu, double inv2var, double c0, float& t) {
  int left = kThresholdSteps;
  while (is_outlier(t, mu, inv2var, c0)) {
    if (left-- == 0) return false;
    t = nextafterf(t, -away);
  }
  for (float further = nextafterf(t, away); fabsf(further) < INFINITY && !is_outlier(further, mu, inv2var, c0);
       further = nextafterf(t, away)) {
    if (left-- == 0) return false;
    t = further;
  }
  return true;
}

}  // namespace sti
