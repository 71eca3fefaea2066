// mt_fix.cuh -- the critical orbit and the Newton quotient of the binary64
// tier in 64-bit fixed point, on the integer and binary32 pipes.
//
// Why.  GB300 issues binary64 arithmetic at 2 lanes per SM per clock, so a
// warp's binary64 instruction takes 16 clocks of the SM; a 32 x 32 + 64 bit
// multiply-add takes 1.2, a shift or an add 0.5 (measured).  An orbit step of
// P and P' is 7 binary64 instructions, 112 clocks of the SM a warp, or 19
// multiply-adds and ~50 shifts and adds, 35 clocks measured (the value alone
// 15); a dependent binary64 operation waits 64 clocks, an integer one 4 to 10.
// No step needs a wide exponent range: on and inside the level line |p_k|
// stays below sqrt(lambda0 + 3), and outside it the descent is still far from
// every root.  Bound: issue and the integer pipes (k_descend at p_20: 63 % issue,
// 50 % ALU pipe, half of the measured multiply-add rate).  Tried and not kept: the
// derivative in float-float (37 clocks, packed pairs 35), its cross terms in
// binary32 (37), a normalisation every step (39).  Split of p_20: descents
// 2.70 -> 0.84 ms, walk 2.32 -> 0.62, seeds 0.60 -> 0.33.
//
// Numbers.  A coordinate is an integer X of 64 bits, value X 2^-(FB+32), held
// as two signed limbs h 2^32 + l: FB bits of fraction in the high limb, the
// components below 2^(30 - FB) (FB = 28: 4, FB = 26: 16) by one unit of the
// high limb or more.  A product keeps 2 FB fractional bits: h h exactly plus the cross terms h l + l h, rounded
// to nearest (the l l term, below a quarter of the last place, is dropped),
// so a step z^2 + c is off by at most 3/4 2^-2FB in each component: 1.04e-17
// for FB = 28, where two binary64 roundings of values in [1, 2) are 2.2e-16.
// The constant c enters with all its FB + 32 bits (its low bits join the
// cross terms).  The derivative is a pair of 64-bit integers with one common
// exponent, normalised every second step to 56 bits.
// Near a root the quotient P / P' is off by 3.5e-18 rms for FB = 28 (1e-17 for
// 27, 4e-17 for 26), in binary64 by 3.5e-17 (against binary128, p_5 to p_32
// and s_{l,n} to order 25).
// The errors are absolute: a component below 1e-4 is less exact than in binary64,
// whose error shrinks with it, and the descents take it from there (axis_step,
// mt_descent.cuh).
// Orbits that leave the fixed range before their last step go on in
// float-float (they are far from every root: |p_k| > 2 escapes), from |p_k|^2 =
// 2^60 on by halving P / P'; one past binary64's range is reported.
#pragma once
#include <cstdint>

#include "mt_ff.cuh"

namespace mt {

struct fx2 {
  int h, l;  // (h 2^32 + l) 2^-(FB+32)
};

__host__ __device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }
__host__ __device__ __forceinline__ int fx_hi(long long w) { return (int)(w >> 32); }
// w 2^s as limbs, 0 <= s <= 31
__host__ __device__ __forceinline__ fx2 fx_split(long long w, int s) {
  const unsigned lo = (unsigned)w;
#ifdef __CUDA_ARCH__
  const unsigned l = lo << s;
  const unsigned h = __funnelshift_l(lo, (unsigned)(w >> 32), s);
#else
  const unsigned long long v = (unsigned long long)w << s;
  const unsigned l = (unsigned)v, h = (unsigned)(v >> 32);
  (void)lo;
#endif
  return fx2{(int)(h + (l >> 31)), (int)l};
}
// (t >> 31) as 32 bits (|t| < 2^62)
__host__ __device__ __forceinline__ int fx_shr31(long long t) {
#ifdef __CUDA_ARCH__
  return (int)__funnelshift_l((unsigned)t, (unsigned)(t >> 32), 1);
#else
  return (int)(t >> 31);
#endif
}
__host__ __device__ __forceinline__ unsigned fx_shl0(unsigned a, int s) {  // 0 for s outside [0, 31]
#ifdef __CUDA_ARCH__
  unsigned r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(s));
  return r;
#else
  return (s < 0 || s > 31) ? 0u : a << s;
#endif
}
__host__ __device__ __forceinline__ int fx_flo(unsigned m) {  // index of the highest set bit, -1 for 0
#ifdef __CUDA_ARCH__
  int r;
  asm("bfind.u32 %0, %1;" : "=r"(r) : "r"(m));
  return r;
#else
  return m ? 31 - __builtin_clz(m) : -1;
#endif
}
// arithmetic shift right by any s >= 0
__host__ __device__ __forceinline__ long long fx_sar(long long w, int s) { return w >> (s < 63 ? s : 63); }

// A binary64 coordinate as X (round to nearest, |x| < 2^(31 - FB); the sign
// and exponent are read as integers) and back (round to nearest even).
template <int F>
__host__ __device__ __forceinline__ long long fx_int(double x) {  // x 2^F, |x| < 2^(63 - F)
#ifdef __CUDA_ARCH__
  const long long b = __double_as_longlong(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
#endif
  const int e = (int)((b >> 52) & 0x7ff);
  long long m = (b & 0x000fffffffffffffll) | (e ? 0x0010000000000000ll : 0ll);
  const int s = e - 1075 + F;  // X = m 2^s
  if (s >= 0) {
    m <<= (s < 10 ? s : 10);  // s <= 10 in range
  } else {
    const int r = -s;
    m = r > 54 ? 0 : (m + (1ll << (r - 1))) >> r;
  }
  return b < 0 ? -m : m;
}
template <int FB>
__host__ __device__ __forceinline__ long long fx_from_f64(double x) {
  return fx_int<FB + 32>(x);
}
template <int FB>
__host__ __device__ __forceinline__ double fx_to_f64(long long X) {
  const unsigned long long a = X < 0 ? 0ull - (unsigned long long)X : (unsigned long long)X;
  if (a == 0) return 0.0;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = __builtin_clzll(a);
#endif
  const unsigned long long n = a << lz;  // top bit set
  unsigned long long m = n >> 11;        // 53 bits
  const unsigned long long rest = n & 0x7ffull;
  m += (rest > 0x400ull || (rest == 0x400ull && (m & 1))) ? 1ull : 0ull;
  // value = m 2^(11 - lz - FB - 32); a carry out of the significand moves into the exponent
  const unsigned long long e = (unsigned long long)(1075 + 11 - lz - FB - 32 - 1);
  const unsigned long long bits = (e << 52) + m | (X < 0 ? 0x8000000000000000ull : 0ull);
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)bits);
#else
  double r;
  __builtin_memcpy(&r, &bits, 8);
  return r;
#endif
}
// |x| < 2^E (false for inf and NaN)
__host__ __device__ __forceinline__ bool fx_below(double x, int E) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
  const int hi = (int)(b >> 32);
#endif
  return (unsigned)(hi & 0x7fffffff) < (unsigned)(1023 + E) << 20;
}
// Every fixed-point operand: |X| < 2^62 - 2^32, so that a limb h, which rounds
// up, stays below 2^30 and neither 2 h nor a cross term shifted by 31 leaves 32
// bits.  In value |x| < 2^(30 - FB) less 2^-FB; binary64 points are taken up to
// 2^(30 - FB) (1 - 2^-21), one unit of their high word below.
template <int FB>
__host__ __device__ __forceinline__ bool fx_fits(double x) {
#ifdef __CUDA_ARCH__
  const int hi = __double2hiint(x);
#else
  long long b;
  __builtin_memcpy(&b, &x, 8);
  const int hi = (int)(b >> 32);
#endif
  return (unsigned)(hi & 0x7fffffff) < ((unsigned)(1023 + 30 - FB) << 20) - 1u;
}
template <int FB>
__host__ __device__ __forceinline__ bool fx_in(long long X) {
  const long long L = (1ll << 62) - (1ll << 32);
  return X > -L && X < L;
}
// The same for a product W at 2^-2FB, on its high word (unit 2^(32 - 2FB))
template <int FB>
__host__ __device__ __forceinline__ bool fx_out(long long Wr, long long Wi) {
  constexpr unsigned R = (1u << (FB - 2)) - 1u;
  const unsigned a = (unsigned)(int)(Wr >> 32) + R, b = (unsigned)(int)(Wi >> 32) + R;
  return (a > b ? a : b) >= 2u * R;
}

// w as a float-float, in units of 2^16 (exact to the pair's 48 bits)
__host__ __device__ __forceinline__ ff fx_to_ff(long long w) {
  const float a = (float)(int)(w >> 40);
  const float b = (float)((int)(w >> 16) & 0xffffff);
  const float c = (float)((int)w & 0xffff);
  ff r;
  r.hi = fmaf(a, 16777216.f, b);
  r.lo = fmaf(c, 1.52587890625e-05f, fmaf(a, 16777216.f, -r.hi) + b);
  return r;
}
__host__ __device__ __forceinline__ float fx_pow2f(int e) {  // 2^e, clamped to binary32's normal range
  e = e < -126 ? -126 : e > 127 ? 127 : e;
#ifdef __CUDA_ARCH__
  return __int_as_float((e + 127) << 23);
#else
  const unsigned b = (unsigned)(e + 127) << 23;
  float f;
  __builtin_memcpy(&f, &b, 4);
  return f;
#endif
}

__host__ __device__ __forceinline__ int fx_exp(float f) {  // floor(log2 |f|), f normal
#ifdef __CUDA_ARCH__
  const unsigned b = __float_as_uint(f);
#else
  unsigned b;
  __builtin_memcpy(&b, &f, 4);
#endif
  return (int)((b >> 23) & 0xff) - 127;
}

// What an evaluation leaves: P and P - T as float-floats in one unit, and
// 1 / P' as a float-float pair: (P - T) / P' = n * inv * 2^sc.  over: P or P'
// is beyond binary64's range.
struct FxVal {
  ff vr, vi, nr, ni, ir, ii;
  int sc;
  bool over;
};

// A target T of the residual P - T: integers at 2^-2FB where it fits (fix),
// else a float-float.
struct FxTarget {
  long long r, i;
  ff fr, fi;
  bool fix;
};

template <int FB>
__host__ __device__ __forceinline__ FxTarget fx_target(double tr, double ti) {
  FxTarget T{0, 0, ff{0.f, 0.f}, ff{0.f, 0.f}, true};
  T.fix = fx_below(tr, 61 - 2 * FB) && fx_below(ti, 61 - 2 * FB);
  if (T.fix) {
    T.r = fx_int<2 * FB>(tr);
    T.i = fx_int<2 * FB>(ti);
  } else {
    T.fr = ff_from(tr);
    T.fi = ff_from(ti);
  }
  return T;
}

// P_a = p_m + (a8 / 8) p_lcap (lcap < 1: p_m) at c = X 2^-(FB+32), and its
// residual to T.  |c| components in range (fx_in).
//
// The derivative is carried as e_k = p'_k / 2^k (e_{k+1} = p_k e_k +
// 2^-(k+1)), e = U 2^(Ex - B) with two integers U of one exponent.  Two steps
// share one normalisation: U starts a pair of steps with its larger
// component in [2^56, 2^57) (or [2^57, 2^58) when the pair before grew it by
// more than 11), the first step leaves it below 2^61 (|p_k| < 4 sqrt 2), the
// second is normalised again.  Ex >= -k keeps 2^-57 of the added 2^-k.
template <int FB, bool CAP>
__host__ __device__ __forceinline__ void fx_eval(int m, int lcap, int a8, long long X, long long Y,
                                                 const FxTarget& T, FxVal& o) {
  constexpr int S = 32 - FB;   // a product at 2^-2FB to limbs
  constexpr int B = 57;
  // c at 2^-2FB and the bits below, which join the cross terms (at 2^-2FB 2^-31)
  const long long CR = (X + (1ll << (S - 1))) >> S, CI = (Y + (1ll << (S - 1))) >> S;
  const long long tr0 = ((X - (CR << S)) << (31 - S)) + (1ll << 30);
  const long long ti0 = ((Y - (CI << S)) << (31 - S)) + (1ll << 30);
  fx2 x = fx_split(X, 0), y = fx_split(Y, 0);
  long long Wr = CR, Wi = CI;
  fx2 u{1 << 24, 0}, v{0, 0};  // e_1 = 1/2
  long long Du = 1ll << (56 - S), Dv = 0;  // e after a step: D 2^(Ex - B + S)
  int Ex = 0;
  long long cwr = 0, cwi = 0, cdu = 0, cdv = 0;
  int cex = 0;
  if (CAP && lcap == 1) { cwr = Wr; cwi = Wi; cdu = Du; cdv = Dv; }
  int k = 1;
  // one orbit step; true where the orbit ends here (k = m, or out of range)
  auto step = [&](long long one) -> bool {
    const int nyh = -y.h, nvh = -v.h;
    long long tu = fx_mad(x.h, u.l, 0x80000000ll);
    tu = fx_mad(x.l, u.h, tu);
    tu = fx_mad(nyh, v.l, tu);
    tu = fx_mad(y.l, nvh, tu);
    long long tv = fx_mad(x.h, v.l, 0x80000000ll);
    tv = fx_mad(x.l, v.h, tv);
    tv = fx_mad(y.h, u.l, tv);
    tv = fx_mad(y.l, u.h, tv);
    Du = fx_mad(nyh, v.h, fx_mad(x.h, u.h, one)) + fx_hi(tu);
    Dv = fx_mad(y.h, u.h, fx_mad(x.h, v.h, 0)) + fx_hi(tv);
    long long tr = fx_mad(x.h, x.l, tr0);
    tr = fx_mad(nyh, y.l, tr);
    long long ti = fx_mad(x.h, y.l, ti0);
    ti = fx_mad(x.l, y.h, ti);
    Wr = fx_mad(nyh, y.h, fx_mad(x.h, x.h, CR)) + fx_shr31(tr);
    Wi = fx_mad(x.h + x.h, y.h, CI) + fx_shr31(ti);
    ++k;
    if (CAP && k == lcap) { cwr = Wr; cwi = Wi; cdu = Du; cdv = Dv; cex = Ex; }
    return k >= m || fx_out<FB>(Wr, Wi);
  };
  if (m > 1) {
    for (;;) {
      const int a = B - S - 1 - k - Ex;  // 2^-(k+1) at D's unit
      const long long one = (long long)(((unsigned long long)fx_shl0(1u, a - 32) << 32) | fx_shl0(1u, a));
      if (step(one)) break;
      x = fx_split(Wr, S);
      y = fx_split(Wi, S);
      u = fx_split(Du, S);
      v = fx_split(Dv, S);
      if (step((long long)((unsigned long long)one >> 1))) break;
      x = fx_split(Wr, S);
      y = fx_split(Wi, S);
      const int uh = fx_hi(Du), vh = fx_hi(Dv);
      const int p = fx_flo((unsigned)((uh ^ (uh >> 31)) | (vh ^ (vh >> 31))));
      int s = 24 - p;
      s = s > 0 ? s : 0;
      s = s < Ex + S + k ? s : Ex + S + k;
      u = fx_split(Du, s);
      v = fx_split(Dv, s);
      Ex += S - s;
    }
  }
  // p_k = W 2^-2FB, p'_k = D 2^(Ex - B + S + k)
  ff dr, di;
  o.over = false;
  o.vr = fx_to_ff(Wr);
  o.vi = fx_to_ff(Wi);
  o.sc = B - S - Ex - k - 2 * FB;
  if (k >= m) {
    if (CAP && lcap >= 1) {
      long long eu = fx_sar(cdu, 3) * a8, ev = fx_sar(cdv, 3) * a8;
      Wr += fx_sar(cwr * a8, 3);
      Wi += fx_sar(cwi * a8, 3);
      const int dlt = (Ex + m) - (cex + lcap);
      if (dlt >= 0) {
        Du += fx_sar(eu, dlt);
        Dv += fx_sar(ev, dlt);
      } else {
        Du = fx_sar(Du, -dlt) + eu;
        Dv = fx_sar(Dv, -dlt) + ev;
        o.sc += dlt;
      }
      o.vr = fx_to_ff(Wr);
      o.vi = fx_to_ff(Wi);
    }
    if (T.fix) {
      o.nr = fx_to_ff(Wr - T.r);
      o.ni = fx_to_ff(Wi - T.i);
    } else {
      o.nr = ff_sub(o.vr, ff_scale(T.fr, fx_pow2f(2 * FB - 16)));
      o.ni = ff_sub(o.vi, ff_scale(T.fi, fx_pow2f(2 * FB - 16)));
    }
    dr = fx_to_ff(Du);
    di = fx_to_ff(Dv);
  } else {
    // Float-float from step k on, far from every root (|p_k| > 2 escapes).
    // Once |p_k|^2 is beyond 2^60, c and the 1 of p' no longer count and
    // every further step halves P / P' exactly.
    const float U = fx_pow2f(16 - 2 * FB), IU = fx_pow2f(2 * FB - 16);
    ff zr = ff_scale(o.vr, U), zi = ff_scale(o.vi, U);
    const ff cr = ff_scale(fx_to_ff(X), fx_pow2f(16 - FB - 32)), ci = ff_scale(fx_to_ff(Y), fx_pow2f(16 - FB - 32));
    dr = fx_to_ff(Du);  // in units of 2^(16 + Ex - B + S + k0)
    di = fx_to_ff(Dv);
    const int ed = 16 + Ex - B + S + k;
    const float one = fx_pow2f(-ed);
    ff xr{0.f, 0.f}, xi{0.f, 0.f}, er{0.f, 0.f}, ei{0.f, 0.f};  // captured
    if (CAP && lcap >= 1 && lcap <= k) {
      const float de = fx_pow2f(cex + lcap - (Ex + k));
      xr = ff_scale(fx_to_ff(cwr), U);
      xi = ff_scale(fx_to_ff(cwi), U);
      er = ff_scale(fx_to_ff(cdu), de);
      ei = ff_scale(fx_to_ff(cdv), de);
    }
    for (; k < m; ++k) {
      const float big = fmaxf(fabsf(zr.hi), fabsf(zi.hi));
      if (big > 1073741824.f) break;
      const ff tr = ff_sub(ff_mul(zr, dr), ff_mul(zi, di)), ti = ff_add(ff_mul(zr, di), ff_mul(zi, dr));
      dr = ff_add(ff_twice(tr), ff{one, 0.f});
      di = ff_twice(ti);
      const ff nr = ff_add(ff_sub(ff_mul(zr, zr), ff_mul(zi, zi)), cr);
      zi = ff_add(ff_twice(ff_mul(zr, zi)), ci);
      zr = nr;
      if (CAP && k + 1 == lcap) { xr = zr; xi = zi; er = dr; ei = di; }
    }
    float IUs = IU;
    if (k < m) {
      const int r = m - k;
      // |P| ~ |p_k|^(2^r) and |P'| ~ |p'_k| 2^r |p_k|^(2^r - 1): past binary64's
      // range from 2^1024 on
      const float lz = 0.5f * log2f(fmaf(zr.hi, zr.hi, zi.hi * zi.hi));
      const float ld = log2f(fmaxf(fabsf(dr.hi), fabsf(di.hi))) + (float)(ed + r);
      o.over = r > 6 || lz * (float)(1 << r) >= 1024.f || ld + lz * (float)((1 << r) - 1) >= 1024.f;
      IUs = 5.421010862427522e-20f;  // n = p_k 2^-64; the target and p_lcap no longer count
      o.sc += 64 - 16 + 2 * FB - r;
    } else if (CAP && lcap >= 1) {
      const float al = 0.125f * a8;
      zr = ff_add(zr, ff_scale(xr, al));
      zi = ff_add(zi, ff_scale(xi, al));
      dr = ff_add(dr, ff_scale(er, al));
      di = ff_add(di, ff_scale(ei, al));
    }
    o.vr = ff_scale(zr, IUs);
    o.vi = ff_scale(zi, IUs);
    if (k < m) {
      o.nr = o.vr;
      o.ni = o.vi;
    } else {
      o.nr = ff_sub(o.vr, T.fix ? fx_to_ff(T.r) : ff_scale(T.fr, IU));
      o.ni = ff_sub(o.vi, T.fix ? fx_to_ff(T.i) : ff_scale(T.fi, IU));
    }
    // |D| may have grown past 2^60: bring its square back into binary32
    const float big = fmaxf(fabsf(dr.hi), fabsf(di.hi));
    if (big > 1e15f) {
      const int e = (fx_exp(big) > 120) ? 100 : 64;
      const float s = fx_pow2f(-e);
      dr = ff_scale(dr, s);
      di = ff_scale(di, s);
      o.sc -= e;
    }
  }
  // 1 / D = conj(D) / |D|^2
  const ff den = ff_add(ff_mul(dr, dr), ff_mul(di, di));
  const ff r = ff_rcp(den);
  o.ir = ff_mul(dr, r);
  o.ii = ff_neg(ff_mul(di, r));
}

// w 2^-2FB in binary32, to its full relative precision (two exact halves)
template <int FB>
__host__ __device__ __forceinline__ float fx_to_f32(long long w) {
  return fmaf((float)fx_hi(w), fx_pow2f(32 - 2 * FB), (float)(unsigned)w * fx_pow2f(-2 * FB));
}

// orbit_f64_d32_k (mt_common.cuh) with the value in fixed point: P = (Wr, Wi)
// 2^-2FB, P' and the curvature P'' / (2 P') in binary32.  False where the
// orbit leaves the fixed range before its last step.  The value alone is a
// third of fx_eval's step; its binary32 companions run beside it.
template <int FB>
__host__ __device__ __forceinline__ bool fx_value_d32_k(int m, long long X, long long Y, long long& Wr, long long& Wi,
                                               float& dr, float& di, float& kr, float& ki) {
  constexpr int S = 32 - FB;
  const long long CR = (X + (1ll << (S - 1))) >> S, CI = (Y + (1ll << (S - 1))) >> S;
  const long long tr0 = ((X - (CR << S)) << (31 - S)) + (1ll << 30);
  const long long ti0 = ((Y - (CI << S)) << (31 - S)) + (1ll << 30);
  fx2 x = fx_split(X, 0), y = fx_split(Y, 0);
  long long wr = CR, wi = CI;
  float dzr = 1.f, dzi = 0.f;  // p'_1 = 1, p''_1 = 0
  float ur = 0.f, ui = 0.f;  // p''_k / 4^k
  float h = 0.5f;  // 2^-(k-1), k = 2
  bool in = true;
#pragma unroll 4
  for (int k = 2; k <= m; ++k) {
    const float fr = fx_to_f32<FB>(wr), fi = fx_to_f32<FB>(wi);
    const float sr = dzr * h, si = dzi * h;  // p'_{k-1} / 2^(k-1)
    h *= 0.5f;
    const float nur = 0.5f * (fmaf(sr, sr, -si * si) + fmaf(fr, ur, -fi * ui));
    const float nui = 0.5f * fmaf(sr + sr, si, fmaf(fr, ui, fi * ur));
    const float tfr = fr + fr, tfi = fi + fi;
    const float ndr = fmaf(tfr, dzr, fmaf(-tfi, dzi, 1.f));
    const float ndi = fmaf(tfr, dzi, tfi * dzr);
    dzr = ndr; dzi = ndi; ur = nur; ui = nui;
    in = in && !fx_out<FB>(wr, wi);
    const int nyh = -y.h;
    const long long tr = fx_mad(nyh, y.l, fx_mad(x.h, x.l, tr0));
    const long long ti = fx_mad(x.l, y.h, fx_mad(x.h, y.l, ti0));
    wr = fx_mad(nyh, y.h, fx_mad(x.h, x.h, CR)) + fx_shr31(tr);
    wi = fx_mad(x.h + x.h, y.h, CI) + fx_shr31(ti);
    x = fx_split(wr, S);
    y = fx_split(wi, S);
  }
  Wr = wr;
  Wi = wi;
  dr = dzr;
  di = dzi;
  // P''/(2P') = (u 2^(m-1)) / (P' 2^-m), both scalings exact
  const float up = fx_pow2f(m - 1), dn = fx_pow2f(-m);
  const float ar = ur * up, ai = ui * up, cr2 = dr * dn, ci2 = di * dn;
  const float inv = 1.f / fmaf(cr2, cr2, ci2 * ci2);
  kr = fmaf(ar, cr2, ai * ci2) * inv;
  ki = fmaf(ai, cr2, -ar * ci2) * inv;
  return in;
}

// (a + ib) (c + id) 2^sc
__host__ __device__ __forceinline__ void fx_cmul(ff a, ff b, ff c, ff d, int sc, ff& qr, ff& qi) {
  const float s = fx_pow2f(sc < -126 ? -126 : sc), s2 = sc < -126 ? fx_pow2f(sc + 126) : 1.f;
  qr = ff_scale(ff_scale(ff_sub(ff_mul(a, c), ff_mul(b, d)), s), s2);
  qi = ff_scale(ff_scale(ff_add(ff_mul(a, d), ff_mul(b, c)), s), s2);
}

// q as an integer at 2^-(FB+32), |q| < 2^(30 - FB)
template <int FB>
__host__ __device__ __forceinline__ long long fx_from_ff(ff q) {
  const float P = (float)(1 << FB), I = 1.f / P;
#ifdef __CUDA_ARCH__
  const int i1 = __float2int_rn(q.hi * P);
#else
  const int i1 = (int)rintf(q.hi * P);
#endif
  const float rem = fmaf(-(float)i1, I, q.hi) + q.lo;
  const float f0 = rem * (P * 4294967296.f);
#ifdef __CUDA_ARCH__
  const int i0 = __float2int_rn(f0);
#else
  const int i0 = f0 >= 2147483520.f ? 2147483647 : f0 <= -2147483648.f ? (int)0x80000000 : (int)rintf(f0);
#endif
  return ((long long)i1 << 32) + i0;
}

}  // namespace mt
