// Nearest neighbours by exact FP64 distances, found with float copies of the positions.
//
// One pass over the candidates keeps the two smallest float squared distances and the candidate of
// the smallest: 15 FP32 and integer instructions a candidate. If the second is farther than the
// first by more than both can err, the first is the nearest in FP64 as well and its exact distance
// is the only one needed; otherwise (about one vertex in a thousand of a Plummer sphere) the
// candidates within the error of the first are compared exactly.
//
// Errors: with float copies of the coordinates a difference errs by at most e + 2^-24 |dx|, where
// e = e_i + e_j and e_k = 2^-23 max|coordinate_k| + 1e-37, so the float distance s is within
// 2^-20 s + sqrt(3) e of the true one (the squares' and sums' rounding included while s^2 is normal),
// and the FP64 squared distance within 2^-50 of the true one.
#pragma once

#include "device.cuh"

namespace mstar {

struct NearestScan {
  float m1, m2;  // the two smallest float squared distances
  int j1;        // the candidate of m1
  __device__ __forceinline__ void clear() {
    m1 = m2 = __int_as_float(0x7f800000);
    j1 = -1;
  }
  __device__ __forceinline__ void add(float dx, float dy, float dz, bool take, int j) {
    float r2 = fmaf(dz, dz, fmaf(dy, dy, dx * dx));
    r2 = take ? fminf(r2, 3e38f) : __int_as_float(0x7f800000);  // (an overflow or NaN counts as 3e38)
    m2 = fminf(m2, fmaxf(m1, r2));
    j1 = r2 < m1 ? j : j1;
    m1 = fminf(m1, r2);
  }
  __device__ __forceinline__ bool none() const { return m1 > 3.2e38f; }  // no candidate was taken
  // The first is certainly the nearest; e bounds e_i + e_j over the candidates.
  __device__ __forceinline__ bool certain(float e) const {
    const float s1 = sqrtf(m1), s2 = sqrtf(m2);
    return m1 > 1e-30f && m1 < 1e30f && s2 * (1.0f - 0x1p-18f) - 1.75f * e > s1 * (1.0f + 0x1p-18f) + 1.75f * e;
  }
  // Candidates whose float squared distance exceeds this are certainly not the nearest (inf: unknown).
  __device__ __forceinline__ float limit(float e) const {
    const float t = sqrtf(fmaxf(m1, 1e-30f)) * (1.0f + 0x1p-17f) + 3.75f * e;
    return m1 < 1e30f ? t * t * (1.0f + 0x1p-16f) : __int_as_float(0x7f800000);
  }
};

}  // namespace mstar
