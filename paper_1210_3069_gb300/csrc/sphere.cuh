// Vectors and tangent frames on the unit sphere shared by the ray recursion,
// the image search and the spectra: products, the (theta-hat, phi-hat) basis and
// the change of basis of a 2x2 matrix.
#pragma once

#include <cuda_runtime.h>

namespace clc {

// Tangent basis (theta-hat, phi-hat) at the unit vector n; on a pole (where
// it is undefined) its limit along phi = 0.
__device__ __forceinline__ void tangent_basis(const double n[3], double t[3], double p[3]) {
  const double r2 = n[0] * n[0] + n[1] * n[1];
  if (r2 == 0.0) {
    t[0] = n[2] >= 0.0 ? 1.0 : -1.0; t[1] = 0.0; t[2] = 0.0;
    p[0] = 0.0; p[1] = 1.0; p[2] = 0.0;
    return;
  }
  const double ir = rsqrt(r2), rho = r2 * ir;
  t[0] = n[2] * n[0] * ir; t[1] = n[2] * n[1] * ir; t[2] = -rho;
  p[0] = -n[1] * ir; p[1] = n[0] * ir; p[2] = 0.0;
}

__device__ __forceinline__ void cross3(const double a[3], const double b[3], double c[3]) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

__device__ __forceinline__ double dot3(const double a[3], const double b[3]) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}

// o = Q A Q^T (row-major 2x2)
__device__ __forceinline__ void qaqt(const double Q[4], const double A[4], double o[4]) {
  const double m0 = Q[0] * A[0] + Q[1] * A[2], m1 = Q[0] * A[1] + Q[1] * A[3];
  const double m2 = Q[2] * A[0] + Q[3] * A[2], m3 = Q[2] * A[1] + Q[3] * A[3];
  o[0] = m0 * Q[0] + m1 * Q[1];
  o[1] = m0 * Q[2] + m1 * Q[3];
  o[2] = m2 * Q[0] + m3 * Q[1];
  o[3] = m2 * Q[2] + m3 * Q[3];
}

}  // namespace clc
