// mt_ff.cuh -- float-float (binary32 pair) arithmetic from the published
// error-free transforms: Knuth's TwoSum, Dekker's FastTwoSum and the
// FMA-based TwoProd.  ~48-bit accurate; used where a binary64 result is not
// needed but binary32 is not enough (the descents' anchor orbits, the
// quotients of the fixed-point tier).
#pragma once
#include <cmath>
#include <cuda_runtime.h>

namespace mt {

struct ff { float hi, lo; };

__host__ __device__ __forceinline__ ff ff_from(double x) {
  ff r;
  r.hi = (float)x;
  r.lo = (float)(x - (double)r.hi);
  return r;
}
__host__ __device__ __forceinline__ ff ff_norm(float s, float e) {  // FastTwoSum, |s| >= |e|
  ff r;
  r.hi = s + e;
  r.lo = e - (r.hi - s);
  return r;
}
__host__ __device__ __forceinline__ ff ff_add(ff a, ff b) {
  const float s = a.hi + b.hi;  // TwoSum
  const float bb = s - a.hi;
  const float e = (a.hi - (s - bb)) + (b.hi - bb) + (a.lo + b.lo);
  return ff_norm(s, e);
}
__host__ __device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = a.hi * b.hi;  // TwoProd
  const float e = fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, fmaf(a.hi, b.hi, -p)));
  return ff_norm(p, e);
}
__host__ __device__ __forceinline__ ff ff_neg(ff a) { return ff{-a.hi, -a.lo}; }
__host__ __device__ __forceinline__ ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
__host__ __device__ __forceinline__ ff ff_twice(ff a) { return ff{a.hi + a.hi, a.lo + a.lo}; }
// s a power of two
__host__ __device__ __forceinline__ ff ff_scale(ff a, float s) { return ff{a.hi * s, a.lo * s}; }
// 1 / a: an approximate binary32 reciprocal and one Newton correction in the low part
__host__ __device__ __forceinline__ ff ff_rcp(ff a) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a.hi));
#else
  const float r = 1.0f / a.hi;
#endif
  const float e = fmaf(-a.lo, r, fmaf(-a.hi, r, 1.f));
  return ff_norm(r, r * e);
}

// The square of the radius within which A d + B d^2 + C d^3 stands for p_K
// around an anchor: |C| rho^2 = 1e-4 |A| and |B| rho = 1e-2 |A| (in the
// maximum norm: C ~ A^3 passes 2^64, its square binary32's range).  Negative,
// so that not even the anchor itself is within it, where a coefficient leaves
// binary32's range.
__host__ __device__ __forceinline__ float series_rho2(float Ax, float Ay, float Bx, float By, float Cx, float Cy) {
  const float a = fmaxf(fabsf(Ax), fabsf(Ay)), b = fmaxf(fabsf(Bx), fabsf(By)), c = fmaxf(fabsf(Cx), fabsf(Cy)),
              ab = a / b;
  const float r = fminf(1e-4f * a / c, 1e-4f * ab * ab);
  // 0 only where all six are finite (fmaxf passes over a NaN)
  const float f = 0.f * (((Ax + Ay) + (Bx + By)) + (Cx + Cy));
  return f == 0.f && c < 1e37f && r > 0.f ? r : -1.f;
}

}  // namespace mt
