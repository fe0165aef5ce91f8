// The FP64 Jacobi rotation from FP32 starting values, for device and host.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#ifndef GENEO_HD
#ifdef __CUDACC__
#define GENEO_HD __host__ __device__ __forceinline__
#else
#define GENEO_HD inline
#endif
#endif

namespace geneo {

// Conversions by integer operations: they run on the FP64 pipe otherwise, which
// bounds these kernels (setup on 64 x 64 elements in FP64 20.8 -> 20.1 ms).  FP32
// truncated, 0 below its normal numbers; values of 2^128 and above are for
// jacobi_f32_inf, which gives infinity for them (and for NaN).
GENEO_HD uint32_t jacobi_hi(double x) {
#ifdef __CUDA_ARCH__
  return (uint32_t)__double2hiint(x);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  return (uint32_t)(u >> 32);
#endif
}
GENEO_HD float jacobi_f32(double x) {
  const uint32_t hi = jacobi_hi(x), m = hi & 0x7fffffffu;
#ifdef __CUDA_ARCH__
  const uint32_t v = __funnelshift_l((uint32_t)__double2loint(x), m - (896u << 20), 3) | (hi & 0x80000000u);
  return __uint_as_float(m < (897u << 20) ? 0u : v);
#else
  uint64_t u;
  memcpy(&u, &x, 8);
  uint32_t v = (uint32_t)((((uint64_t)(m - (896u << 20)) << 32) | (uint32_t)u) >> 29) | (hi & 0x80000000u);
  if (m < (897u << 20)) v = 0u;
  float f;
  memcpy(&f, &v, 4);
  return f;
#endif
}
GENEO_HD float jacobi_f32_inf(double x) {
  return (jacobi_hi(x) & 0x7fffffffu) < (1151u << 20) ? jacobi_f32(x) : (float)HUGE_VAL;
}
GENEO_HD double jacobi_f64(float f) {
#ifdef __CUDA_ARCH__
  const uint32_t u = __float_as_uint(f), m = u & 0x7fffffffu;
  const uint32_t h = (u & 0x80000000u) | ((m >> 3) + (896u << 20));
  return m < 0x00800000u ? 0.0 : __hiloint2double((int)h, (int)(u << 29));
#else
  return fabsf(f) < 0x1p-126f ? 0.0 : (double)f;
#endif
}

// The rotation that annihilates a_pq has the tangent t, the root of apq t^2 + dd t -
// apq = 0 (dd = a_qq - a_pp) of at most 1 in size, and the cosine c = (1 +
// t^2)^(-1/2).
//
// The divisions and square roots of t = 1 / (|theta| + sqrt(theta^2 + 1)), theta = dd
// / (2 apq), and of c are dependent chains on a pipe of 1/64 of the FP32 rate.  So
// both start in FP32 (t0, y0 about c, g about the reciprocal of the derivative 2 apq
// t + dd, each good to a few 1e-7) and end in FP64 multiply-adds: t by two Newton
// steps with FP64 residuals (the first leaves about 1e-13, the second FP64
// rounding), c by one third-order step.  Largest errors over a million pivots: t
// 2.1e-16 (3.3e-16 by the formula in FP64), c 1.5e-16 (3.0e-16).  Setup on 64 x 64
// elements 20.1 ms, by the formula 24.4; on 48^3 385 and 404.
GENEO_HD void jacobi_refine(double dd, double apq, float t0, float y0, float g, double& t, double& c) {
  const double y = jacobi_f64(y0), y2 = y * y;   // exact
  double x = jacobi_f64(t0);
  x -= jacobi_f64(jacobi_f32(fma(fma(apq, x, dd), x, -apq)) * g);
  x -= jacobi_f64(jacobi_f32(fma(fma(apq, x, dd), x, -apq)) * g);
  t = x;
  const double e = fma(-fma(x, x, 1.0), y2, 1.0);
  c = fma(y, fma(0.375, e, 0.5) * e, y);
}

// Whether the FP32 values, residuals and steps above stay in range (entries of
// nearly converged matrices lie inside: a narrower range, 1e-15 and 1e15, sent many
// of their rotations to the formula, and setup on 64 x 64 elements took 21.6 ms).
GENEO_HD bool jacobi_in_range(float theta, float af) {
  return fabsf(af) > 1e-22f && fabsf(af) < 1e15f && fabsf(theta) < 1e22f;
}
GENEO_HD double jacobi_tangent_formula(double dd, double apq) {
  const double theta = dd / (2.0 * apq);
  return (theta >= 0.0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
}

}  // namespace geneo
