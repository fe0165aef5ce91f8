// Square root of a Cholesky pivot and quotients by it from one reciprocal square
// root, for device and host.
#pragma once

#include <math.h>

#ifndef GENEO_HD
#ifdef __CUDACC__
#define GENEO_HD __host__ __device__ __forceinline__
#else
#define GENEO_HD inline
#endif
#endif

namespace geneo {

// r = p^(-1/2) to an ulp or so.  A step of the Newton iteration each: without it
// the product p r is off by up to 1.5 * 2^-53 (the square root by 2^-53) and a r by
// more on average than the quotient.
template <typename T>
GENEO_HD T pivot_root(T p, T r) {
  const T d = p * r;
  return fma(T(0.5) * r, fma(-d, d, p), d);
}
// a / d, d = pivot_root(p, r)
template <typename T>
GENEO_HD T pivot_quotient(T a, T d, T r) {
  const T q = a * r;
  return fma(r, fma(-q, d, a), q);
}

}  // namespace geneo
