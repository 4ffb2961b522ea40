// ddouble.cuh -- double-double (hi + lo, ~2^-104 relative) arithmetic of the
// plan-time table kernels.
#pragma once
#include <cuda_runtime.h>

namespace nusht {

struct dd {
  double hi, lo;
};
__device__ __forceinline__ dd dd_fast(double a, double b) {
  const double s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ dd dd_mul(dd a, double b) {
  const double p = a.hi * b;
  return dd_fast(p, fma(a.lo, b, fma(a.hi, b, -p)));
}
__device__ __forceinline__ dd dd_div(dd a, double b) {
  const double q = a.hi / b;
  const double r = fma(-q, b, a.hi) + a.lo;
  return dd_fast(q, r / b);
}
__device__ __forceinline__ dd dd_quot(double a, double b) { return dd_div({a, 0.0}, b); }
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  const double s = a.hi + b.hi, bb = s - a.hi;
  return dd_fast(s, ((a.hi - (s - bb)) + (b.hi - bb)) + (a.lo + b.lo));
}
__device__ __forceinline__ double dd_root(dd a) {
  const double s = sqrt(a.hi);
  return s + (fma(-s, s, a.hi) + a.lo) / (2.0 * s);
}

__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const double p = a.hi * b.hi;
  return dd_fast(p, fma(a.hi, b.lo, fma(a.lo, b.hi, fma(a.hi, b.hi, -p))));
}
// the value `off` lanes below
__device__ __forceinline__ dd dd_up(dd v, int off) {
  return {__shfl_up_sync(0xffffffffu, v.hi, off), __shfl_up_sync(0xffffffffu, v.lo, off)};
}

}  // namespace nusht
