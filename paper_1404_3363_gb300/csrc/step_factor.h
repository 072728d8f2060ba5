// Step control of the FP64 integrator for groups of lanes (k_coop64.cuh), in
// plain C++ so that it also runs on the host.
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define IVV_STEP_HD __host__ __device__ __forceinline__
#else
#define IVV_STEP_HD inline
#endif

namespace ivv {

// fac = 0.9 (tol / err)^(1/3), the FP32 cube root refined by one Newton step
// (relative error 1e-13) without a double division.  An error that FP32 does
// not hold takes the plain form, as the one-lane kernel: at a point where
// det J = 0 the slope is infinite and so is the error (factor 0, and the
// step is retried at a fifth); its FP32 reciprocal would make that a NaN.
IVV_STEP_HD double coop_step_factor(double tol, double err) {
  if (!(err > 1e-36 && err < 1e36)) return 0.9 * cbrt(tol / err);
  const float ri = 1.f / (float)err;
  const double inv = (double)ri * fma(-err, (double)ri, 2.0);
  const double x = tol * inv;
  const float xf = (float)x;
  if (!(xf > 1e-30f && xf < 1e30f)) return 0.9 * cbrt(x);
  const float r = cbrtf(xf);
  const double rd = (double)r;
  return 0.9 * fma(-fma(rd * rd, rd, -x), (double)(1.f / (3.f * r * r)), rd);
}

}  // namespace ivv
