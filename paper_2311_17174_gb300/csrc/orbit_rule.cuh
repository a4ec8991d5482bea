// orbit_rule.cuh -- when the orbit's Newton iteration (k_orbit.cu) has settled,
// callable on the host as well.
#pragma once
#include <cuda_runtime.h>

namespace emri {

// u1, u2, ...: sizes of the updates (relative for v, absolute for e) that the
// evaluations apply, largest of the walker's segments; each is the error
// before it, so u_{k+1} / u_k measures the contraction and the error left by
// the last update u is about u times it.  Measured contraction: 5e-5 to 7e-4
// over the configurations' orbits, up to 3e-2 for the fastest ones (1e5 solar
// masses, e > 0.8 at the LSO), where the FP32 linearisation is worst.

// What may be left, in v: one ulp of a double, as the sequential solver leaves.
// Over 1e5 cycles it moves the phase by 4e-10 rad.
constexpr float kOrbitLeft = 2e-16f;

// A fourth evaluation after updates u1 and u2: where three would leave more
// than a tenth of kOrbitLeft at the contraction u2 / u1 (a later one can be
// three times weaker), or u2 is large.
__host__ __device__ __forceinline__ bool orbit_again(float u1, float u2) {
  return !(u2 <= 1e-9f && u2 * u2 * u2 <= 0.1f * kOrbitLeft * (u1 * u1));
}

// Whether the last update leaves less than kOrbitLeft, at the worse of the last
// two contractions last / prev and prev / prev2.  False for NaN.
__host__ __device__ __forceinline__ bool orbit_settled(float prev2, float prev, float last) {
  if (last <= 1e-16f) return true;   // at rounding level, where the ratios say nothing
  return last <= 1e-12f && last * last <= kOrbitLeft * prev && last * prev <= kOrbitLeft * prev2;
}

}  // namespace emri
