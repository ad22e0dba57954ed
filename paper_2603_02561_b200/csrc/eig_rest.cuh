// What the rows that the tridiagonal reduction leaves out may carry for its result to count as complete.
#pragma once

#include <cuda_runtime.h>

namespace solar {

// rest: trace of the rows left out, trace: of G, theta_last: the smallest kept eigenvalue found, all of the scaled
// matrix.  The residuals say that the kept vectors are eigenvectors, not that they belong to the largest eigenvalues.  G is
// positive semi-definite, so no eigenvalue of the rest is above its trace: below theta_last nothing is missing.  (The end on
// a decoupled tail leaves at most theta_last / 2.)  A trace of 1e-4 of G's is what the comparison of trace(T) with trace(G)
// allows anyway; histories of lower rank than r end there, with theta_last at the rounding level.  False for a NaN.
__host__ __device__ __forceinline__ bool rest_keeps_result(float rest, float trace, float theta_last) {
  return rest <= (theta_last > 1e-4f * trace ? theta_last : 1e-4f * trace);
}

}  // namespace solar
