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

// fac = 0.9 (tol / err)^(1/3) to double precision (relative error below 4e-16,
// as the cube root's own) without a double division: the FP32 cube root, and
// two Newton steps on err r^3 = tol, which take it from 1e-7 over 1e-14 to the
// last bit.  Numbers whose quotient FP32 may not hold take the plain form, as
// the one-lane kernel: at a point where det J = 0 the slope is infinite and so
// is the error (factor 0, and the step is retried at a fifth), which would be a
// NaN here.
IVV_STEP_HD double coop_step_factor(double tol, double err) {
  if (!(err > 1e-24 && err < 1e12 && tol > 1e-24 && tol < 1e12)) return 0.9 * cbrt(tol / err);
  const float ef = (float)err, rf = cbrtf((float)tol / ef);
  const double c = (double)(-1.f / (3.f * ef * rf * rf));       // -1 / f'(r) of f = err r^3 - tol
  double r = (double)rf;
  r = fma(fma(err * r, r * r, -tol), c, r);
  r = fma(fma(err * r, r * r, -tol), c, r);
  return 0.9 * r;
}

}  // namespace ivv
