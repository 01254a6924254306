// The projector's convergence measure and what follows from it (host only).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <limits>

namespace bst {

// `worst` raised to the largest of n residuals; infinite as soon as one of
// them is not finite (a maximum would pass over a NaN: every comparison with
// it is false), so that a round whose vectors or values overflowed counts as
// diverged and not as converged.
inline double raise_worst(double worst, const double* res, std::size_t n) {
  for (std::size_t j = 0; j < n; ++j) {
    if (!std::isfinite(res[j])) return std::numeric_limits<double>::infinity();
    if (res[j] > worst) worst = res[j];
  }
  return worst;
}

// Plain steps that bring a residual `worst` to half the tolerance when each
// multiplies it by `decay`: at least `iters`, at most 6 iters, and `iters` when
// the decay says nothing (not below one, or a residual that is not finite).
inline int plain_steps(int iters, double worst, double tol, double decay) {
  if (!(worst > 0) || !std::isfinite(worst) || !(decay > 0 && decay < 1)) return iters;
  const double need = std::log(0.5 * tol / worst) / std::log(decay);
  return int(std::min<double>(6.0 * iters, std::max<double>(iters, std::ceil(need))));
}

}  // namespace bst
