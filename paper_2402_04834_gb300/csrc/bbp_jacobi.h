// Scalar step of the one-sided Jacobi rotation, for device and host code.
#pragma once

#include <math.h>

#include "bbp_geometry.h"

namespace bbp {

// Tangent of the Jacobi rotation of two columns whose squared norms differ by
// d and whose product is c: the root of c t^2 + d t - c = 0 with |t| <= 1 (c
// and max(|d|, |c|) representable in FP32).  An FP32 root (1e-7) takes two
// simplified Newton steps: the residual in FP64, the derivative's reciprocal
// in FP32 and the same for both, so that each step gains seven digits and the
// last one leaves two FP64 roundings.  One step with an FP32 correction, which
// this replaced, costs as many FP64 instructions (conversions are such, too)
// and stops at 2e-14.
BBP_HD double jacobi_tangent(double d, double c) {
  const float df = (float)d, cf = (float)c, z = df / (2.f * cf), az = fabsf(z);
  const float tf = copysignf(az > 1e4f ? 0.5f / az : 1.f / (az + sqrtf(fmaf(az, az, 1.f))), z);
  const double inv = (double)(1.f / fmaf(2.f * cf, tf, df));
  double t = (double)tf;
  t = fma(-fma(fma(c, t, d), t, -c), inv, t);
  return fma(-fma(fma(c, t, d), t, -c), inv, t);
}

}  // namespace bbp
