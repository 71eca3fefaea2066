// mt_descent.cuh -- one binary64 Newton descent in fixed point (mt_fix.cuh),
// shared by the single-polynomial kernels (mt_newton.cu) and the batched
// one (mt_batch.cu).
#pragma once
#include "mt_common.cuh"
#include "mt_fix.cuh"

namespace mt {

constexpr int FXB = 28;  // fraction bits of the high limb: |Re|, |Im| < 4
// waiting lanes that trigger a refill of the persistent kernels (p_24: 1 13.66
// ms, 3 13.54, 5 13.60, 8 13.99; every s_{l,n} to order 16: 1.13, 1.09, 1.09, 1.10)
constexpr unsigned DESC_REFILL = 3;

// z as X, Y at 2^-60, or as the bits of its binary64 coordinates (wide:
// outside the fixed range, or a polynomial kept in binary64), and the squares of the last step and of the
// divergence radius.
struct Descent {
  long long X, Y;
  float rdiv2, prev2;
  int it;
  bool wide, fx;
};

__device__ __forceinline__ void descent_set(Descent& d, double x, double y) {
  d.wide = !(d.fx && fx_fits<FXB>(x) && fx_fits<FXB>(y));
  d.X = d.wide ? __double_as_longlong(x) : fx_from_f64<FXB>(x);
  d.Y = d.wide ? __double_as_longlong(y) : fx_from_f64<FXB>(y);
}
__device__ __forceinline__ void descent_start(Descent& d, double2 z0, bool fx) {
  d.fx = fx;
  d.it = 0;
  d.prev2 = 3.0e38f;
  // long jump: beyond twice the start radius and outside D(0, 4)
  const float ax = f32_trunc(z0.x), ay = f32_trunc(z0.y);
  d.rdiv2 = fmaxf(16.f, 4.f * fmaf(ax, ax, ay * ay));
  descent_set(d, z0.x, z0.y);
}
__device__ __forceinline__ double2 descent_point(const Descent& d) {
  return d.wide ? make_double2(__longlong_as_double(d.X), __longlong_as_double(d.Y))
                : make_double2(fx_to_f64<FXB>(d.X), fx_to_f64<FXB>(d.Y));
}

// One binary64 Newton step, for the points outside the fixed range (starts of
// polynomials of a small degree), at a zero of P', or of a polynomial kept in
// binary64; NaN where it is not
// finite.  s2 receives |step|^2.
static __device__ __noinline__ double2 newton_step_f64(int m, int lcap, double2 z, float& s2) {
  double vr, vi, dr, di, qr, qi;
  orbit_f64(m, lcap, 1.0, z.x, z.y, vr, vi, dr, di);
  cdiv_f64(vr, vi, dr, di, qr, qi);
  const float fr = f32_trunc(qr), fi = f32_trunc(qi);
  s2 = fmaf(fr, fr, fi * fi);
  return make_double2(z.x - qr, z.y - qi);
}

// Roots next to the real axis.  A fixed-point coordinate is off by some 2e-18
// however small it is; in binary64 the error of a small Im shrinks with it (and
// at the root 0 that of Re as well).  rms of Im over the roots of p_20 with |Im|
// below 1e-6: 1.4e-18 fixed, 1.8e-19 binary64; in [1e-6, 1e-4) 2.2e-18 and
// 4.7e-19; from 1e-4 on the fixed point is the closer (2.3e-18 and 7.3e-18).
// So the components below 2^-13 of a converged point are taken from one more
// step with the value in binary64 (P' in binary32: the step is ~1e-16, its
// relative error of 1e-6 is nothing); the others keep the fixed point's digits.
constexpr int AXIS_EXP = -13;
static __device__ __noinline__ double2 axis_step(int m, int lcap, double2 z) {
  double vr, vi;
  float dr, di, qr, qi;
  orbit_f64_d32(m, lcap, z.x, z.y, vr, vi, dr, di);
  if (!cdiv_f32s(f32_trunc(vr), f32_trunc(vi), dr, di, qr, qi)) return z;
  if (fx_below(z.x, AXIS_EXP)) z.x -= f64_of_f32(qr);
  if (fx_below(z.y, AXIS_EXP)) z.y -= f64_of_f32(qi);
  return z;
}
// A point that the caller will fold to the real axis (|Im| < eps / 2: a real root,
// one in ten) needs no step unless it is the root 0: axis_floor is the high word of
// eps / 4, from which on Im counts (0: always; the step moves Im by some 1e-17, so
// an eps below 1e-16 takes every point).  The finish of p_24: 0.305 -> 0.282 ms,
// descents of s_{4,22} 52.4 -> 51.9.
inline unsigned axis_floor(double eps) {
  const double q = 0.25 * eps;
  unsigned long long b;
  __builtin_memcpy(&b, &q, 8);
  return eps >= 1e-16 ? (unsigned)(b >> 32) : 0u;
}
__device__ __forceinline__ bool axis_near(double2 z, unsigned floor_hi) {
  return fx_below(z.y, AXIS_EXP) &&
         ((unsigned)(__double2hiint(z.y) & 0x7fffffff) >= floor_hi || fx_below(z.x, AXIS_EXP));
}
// A warp gathers such points (their indices in cand) and steps 32 of them
// together, since a binary64 step costs it the same for one.  buf: its 64
// entries of shared memory; n: entries waiting (warp-uniform).
template <class T>
__device__ __forceinline__ void axis_push(T* buf, unsigned& n, bool mine, T at) {
  const unsigned b = __ballot_sync(0xffffffffu, mine);
  if (mine) buf[n + __popc(b & lanemask_lt())] = at;
  n += __popc(b);
}
// the last (up to 32) entries: true for the lanes that received one (*at)
template <class T>
__device__ __forceinline__ bool axis_pop(const T* buf, unsigned& n, T& at) {
  __syncwarp();  // the entries, and the candidates they name, are written
  const unsigned c = n < 32u ? n : 32u;
  n -= c;
  const bool mine = (threadIdx.x & 31) < c;
  if (mine) at = buf[n + (threadIdx.x & 31)];
  __syncwarp();  // read before the next push
  return mine;
}

// One Newton step and its outcome: -1 go on, 0 converged, 1 divergent, 2 cap.
template <bool CAP>
__device__ __forceinline__ int descent_step(int m, int lcap, Descent& d, float tol2, int cap) {
  float s2 = 0.f;
  bool ok = false;
  if (!d.wide) {
    FxVal o;
    const FxTarget T{0, 0, ff{0.f, 0.f}, ff{0.f, 0.f}, true};
    fx_eval<FXB, CAP>(m, lcap, 8, d.X, d.Y, T, o);
    ff qr, qi;
    fx_cmul(o.nr, o.ni, o.ir, o.ii, o.sc, qr, qi);
    ok = fabsf(qr.hi) < 4.f && fabsf(qi.hi) < 4.f;  // false for NaN too
    if (o.over) {  // P or P' beyond binary64
      d.X = d.Y = 0x7ff8000000000000ll;
      d.wide = true;
      ok = true;
    } else if (ok) {
      s2 = fmaf(qr.hi, qr.hi, qi.hi * qi.hi);
      d.X -= fx_from_ff<FXB>(qr);
      d.Y -= fx_from_ff<FXB>(qi);
      if (!(fx_in<FXB>(d.X) && fx_in<FXB>(d.Y))) {
        d.X = __double_as_longlong(fx_to_f64<FXB>(d.X));
        d.Y = __double_as_longlong(fx_to_f64<FXB>(d.Y));
        d.wide = true;
      }
    }
  }
  if (!ok) {
    const double2 z = newton_step_f64(m, lcap, descent_point(d), s2);
    descent_set(d, z.x, z.y);
  }
  float ax, ay;
  bool lost = false;
  if (d.wide) {  // beyond binary32 (2^64 for |z|^2) inf, as the radius of such a start
    const double2 z = descent_point(d);
    lost = !finite2(z.x, z.y);
    ax = f32_trunc(z.x);
    ay = f32_trunc(z.y);
  } else {
    ax = (float)fx_hi(d.X) * (1.f / (1 << FXB));
    ay = (float)fx_hi(d.Y) * (1.f / (1 << FXB));
  }
  ++d.it;
  int outcome = -1;
  const float fl = (1.f + fabsf(ax) + fabsf(ay)) * 3.552713678800501e-15f;  // 16 ulp of binary64
  const float z2 = fmaf(ax, ax, ay * ay);
  if (lost || !(z2 <= d.rdiv2)) outcome = 1;
  else if (s2 < tol2) outcome = 0;  // the step that met tol also squared the error
  // binary64 rounding floor: steps stopped shrinking within a few ulp of z
  // (between two close roots Newton also stalls, at |step| ~ their
  // separation^2 / distance, far above this floor)
  else if (s2 >= 0.25f * d.prev2 && s2 < fl * fl) outcome = 0;
  else if (d.it >= cap) outcome = 2;
  d.prev2 = s2;
  return outcome;
}

// tol^2 in binary32 (not below its smallest positive value, so that a step
// of zero always meets it)
inline float tol2_f(double tol) { return std::max((float)(tol * tol), 1.4e-45f); }

}  // namespace mt
