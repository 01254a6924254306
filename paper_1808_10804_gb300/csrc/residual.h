// The projector's convergence measure (host only).
#pragma once

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

}  // namespace bst
