// FP64 roots and quotients along serial chains (internal header).
//
// A dependent FP64 instruction takes about 100 cycles on this chip, and the
// library's root and division are chains of ten and more, so the solvers'
// serial parts take a float seed, one Newton step on the reciprocal (root) and
// one on the residual of the result itself: a fused multiply-add gives that
// residual with one rounding, so the result is the exact value rounded once (to
// within 2^-85; Markstein, IBM J. Res. Dev. 34, 1990).  Two Newton steps on the
// reciprocal and a product, as short, are off by up to 2.7 units of 2^-53.
#pragma once

#include "ed_internal.h"

namespace ed {

// Binary exponent field of a double; magnitudes with fields in (920, 1120) lie
// well inside the range of a normal float, and so do their reciprocals.
__device__ __forceinline__ int exp_field(double v) { return __double2hiint(v) & 0x7ff00000; }
__device__ __forceinline__ bool float_range(double v) {
  const int e = exp_field(v);
  return e > (920 << 20) && e < (1120 << 20);
}

// root = sqrt(v), inv = 1 / root, v > 0.
__device__ __forceinline__ void root_inverse(double v, double& root, double& inv) {
  if (!float_range(v)) {
    root = sqrt(v);
    inv = 1.0 / root;
    return;
  }
  double y = (double)rsqrtf((float)v);
  y = y * fma(-0.5 * v, y * y, 1.5);   // 1 / sqrt(v) to 2^-42
  const double g = v * y;
  root = fma(fma(-g, g, v), 0.5 * y, g);
  inv = fma(fma(-root, y, 1.0), y, y);
}

// a / d from y, the reciprocal of d to 2^-46.
__device__ __forceinline__ double quot_step(double a, double d, double y) {
  const double g = a * y;
  return fma(fma(-d, g, a), y, g);
}
// Reciprocal of d to 2^-46, d in float_range.
__device__ __forceinline__ double rcp_seed(double d) {
  const double y = (double)(1.0f / (float)d);
  return fma(y, fma(-d, y, 1.0), y);
}

// a / d for |a| <= |d|.
__device__ __forceinline__ double quotient(double a, double d) {
  return float_range(d) ? quot_step(a, d, rcp_seed(d)) : a / d;
}

}  // namespace ed
