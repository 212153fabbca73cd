// The two vectors a pair's score is formed from, shared by all score kernels:
// a = sqrt(vol2) Z2 - sqrt(vol1) Z1 and b = sqrt(vol2) Z2 + sqrt(vol1) Z1 in
// float64.
#pragma once

namespace cdl {

// The compiler contracts w - v to fma(-s1, Z1, w), which leaves the rounding of w
// where the two products are equal: equal (opposite) embeddings under equal volumes
// get their a = 0 (b = 0) apart, and with it scores of exactly 0 (NaN for infinities,
// as from w - v). The test of the volumes comes first and is one for all threads: the
// kernels are bound by float64 instructions.
__device__ __forceinline__ void score_ab(const double* __restrict__ Z1, const double* __restrict__ Z2, double s1,
                                         double s2, size_t o, double& a, double& b) {
  const double z1 = Z1[o], z2 = Z2[o], w = s2 * z2, v = s1 * z1;
  a = w - v;
  b = w + v;
  if (s1 == s2) {
    if (z1 == z2) a = z2 - z1;
    if (z1 == -z2) b = z2 + z1;
  }
}

}  // namespace cdl
