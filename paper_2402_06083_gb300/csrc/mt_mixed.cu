// mt_mixed.cu -- the mixed-precision tier (MT_MIXED): binary32 level-line
// tracking and early Newton steps around float-float anchors (binary64 ones
// in the seed lift), and a finish with the value in 64 bits: binary64, or fixed
// point (mt_fix.cuh) for p_23 to p_25.
//
// Why.  The paper runs everything in FP80 (Sec. 6.1) and notes that GPUs
// offer little beyond FP64 (Sec. 6.4.5).  On a GB300 the binary64 pipe is
// the bottleneck (about 1.2 TFLOP/s) while binary32 runs ~60x faster, so the
// bulk of the Newton steps -- which only need to stay in the right basin --
// move to binary32, and binary64 is spent where precision is decided.
//
// How.  Absolute binary32 coordinates cannot resolve the level line at the
// periods of interest (sub-step spacings reach 1e-11 near c = -2 at n = 20),
// so the binary32 work is done in perturbation form around an anchor c0
// (the published perturbation technique of deep-zoom Mandelbrot
// renderers): with Z_k = p_k(c0) (float-float, ~1e-14; binary64 in the seed
// lift) and c = c0 + delta,
//   e_{k+1} = (2 Z_k + e_k) e_k + delta,   p_k(c) = Z_k + e_k,
//   p'_{k+1}(c) = 2 (Z_k + e_k) p'_k(c) + 1            (binary32),
// so binary32 carries only the difference from the anchor and its relative
// precision applies to |delta|, not to |c|.  The residual P(c) - T is
// (Z_m - T) + e_m with Z_m split into binary32 hi + lo.
//   - Walk: the anchor is re-taken every K sub-steps (a few turns of the
//     phase) from the current point, so |delta| stays a few turns' length.
//   - Descent: the anchor is the start point (p_n from 23 on: one of four
//     consecutive starts); binary32 Newton steps run to the binary32 floor, then
//     64-bit Newton steps (1.08 a root at p_28), once per group of end points on
//     the same root, finish to the tolerance (eq. Newton).
// The anchors only steer the binary32 steps; every root's digits come from
// its 64-bit finishing steps.  The chunk-end check of the walk and the
// count check catch any tracking failure, and the host then repeats the
// split in plain binary64.
#include "mt_descent.cuh"
#include "mt_fix.cuh"
#include "mt_levelline.cuh"
#include "mt_pert.cuh"

namespace mt {

constexpr int MIX_MAXM = 41;
// Shorter orbits of p_n keep an anchor per start, the whole orbit and the
// binary64 finish and tip redo.  Not for their speed: all four of the long orbits'
// ways take p_20 from 1.36 to 1.30 ms (the walk's series alone is slower there, see
// WALK_SERIES_MIN).  The last digits of these roots are what nearest-neighbour
// distances at the tip rest on, and they stay those of binary64.
constexpr int MIX_LONG = 23;
inline bool mixed_short(const PolyDev& P) { return P.kind == 0 && P.m < MIX_LONG; }
// The binary64 finish in fixed point: p_23 to p_25.  Of p_28's 67 M roots some
// neighbours' real parts agree in every digit; their places in the sorted list
// hang on the last one, and the binary64 finish leaves those as they were (1e-10
// at the worst of 4 M sampled components, 9e-7 with the fixed one).  s_{l,n}
// keeps it too: at |s| = 100 its tip pairs rest on the same digits (q_{8,12}: 4411
// roots to redo in double-double with the fixed finish, over the 4096 places).
constexpr int FIN_FX_MAXM = 25;

// binary64 reference orbit at c0: zs[k * stride] = Z_k in binary32 for
// k = 0 .. m-1 (truncated on the integer pipe: the binary64 pipe keeps the
// orbit itself), and v = P(c0) = Z_m (+ Z_lcap) as binary32 hi (x, y) + lo (z, w).
__device__ __forceinline__ void ref_orbit(const PolyDev& P, double c0x, double c0y, float2* zs,
                                          int stride, float4& v) {
  double zx = 0.0, zy = 0.0, capx = 0.0, capy = 0.0;
  zs[0] = make_float2(0.f, 0.f);
  for (int k = 1; k <= P.m; ++k) {
    const double nx = fma(zx, zx, fma(-zy, zy, c0x));
    const double ny = fma(twice_f64(zx), zy, c0y);
    zx = nx;
    zy = ny;
    if (k < P.m) zs[k * stride] = make_float2(f32_trunc(zx), f32_trunc(zy));  // integer pipe
    if (k == P.lcap) { capx = zx; capy = zy; }
  }
  const double vx = zx + capx, vy = zy + capy;
  const float hx = (float)vx, hy = (float)vy;
  v = make_float4(hx, hy, (float)(vx - (double)hx), (float)(vy - (double)hy));
}

// binary32 perturbation orbit: e = P(c0 + delta) - P(c0), D = P'(c0 + delta).
// The derivative is carried as g_k = p'_k / 2^k (g_{k+1} = p_k g_k +
// 2^-(k+1)): the same binary32 roundings as p'_{k+1} = 2 p_k p'_k + 1 up to
// powers of two, without doubling p_k (12 binary32 operations a step, not 14).
__device__ __forceinline__ void pert_eval(const PolyDev& P, const float2* zs, int stride, float dx,
                                          float dy, float& ex, float& ey, float& Dx, float& Dy) {
  float e_x = 0.f, e_y = 0.f, g_x = 0.f, g_y = 0.f;
  float ce_x = 0.f, ce_y = 0.f, cg_x = 0.f, cg_y = 0.f;
  int hexp = (127 - 1) << 23;  // exponent field of 2^-(k+1), k = 0
#pragma unroll 2
  for (int k = 0; k < P.m; ++k) {
    const float2 Z = zs[k * stride];
    const float zx = Z.x + e_x, zy = Z.y + e_y;  // p_k(c)
    const float h = __int_as_float(hexp);
    hexp -= 1 << 23;
    const float ng_x = fmaf(zx, g_x, fmaf(-zy, g_y, h));
    const float ng_y = fmaf(zx, g_y, zy * g_x);
    const float sx = Z.x + zx, sy = Z.y + zy;  // 2 Z_k + e_k
    const float ne_x = fmaf(sx, e_x, fmaf(-sy, e_y, dx));
    const float ne_y = fmaf(sx, e_y, fmaf(sy, e_x, dy));
    e_x = ne_x; e_y = ne_y; g_x = ng_x; g_y = ng_y;
    if (k + 1 == P.lcap) { ce_x = e_x; ce_y = e_y; cg_x = g_x; cg_y = g_y; }
  }
  ex = e_x + ce_x;
  ey = e_y + ce_y;
  // p'_m + p'_lcap = 2^m (g_m + 2^(lcap-m) g_lcap), exact scalings
  const float a = P.lcap > 0 ? __int_as_float((127 + P.lcap - P.m) << 23) : 0.f;
  const float s = __int_as_float((127 + P.m) << 23);
  Dx = fmaf(a, cg_x, g_x) * s;
  Dy = fmaf(a, cg_y, g_y) * s;
}

// Newton with target in perturbation form: the binary32 twin of the walk's
// newton_target_f64, with the same predictor (pred: first step solves
// log P = log T from the previous target Tp, L = log(T / Tp)) and stop rule.
__device__ __forceinline__ int newton_target_pert(const PolyDev& P, const float2* zs, int stride,
                                                  const float4& v, float& dx, float& dy, float tx,
                                                  float ty, float rel, int cap, float* first,
                                                  bool pred, float tpx, float tpy, float Lr,
                                                  float Li, bool* bad) {
  float thr2 = 0.f, prev2 = 0.f, h2 = 0.f;
  int it = 0;
  while (it < cap) {
    float ex, ey, Dx, Dy;
    pert_eval(P, zs, stride, dx, dy, ex, ey, Dx, Dy);
    float nr, ni;
    if (it == 0 && pred) {  // P - Tp - L P
      const float Pr = v.x + (v.z + ex), Pi = v.y + (v.w + ey);
      nr = (Pr - tpx) - fmaf(Lr, Pr, -Li * Pi);
      ni = (Pi - tpy) - fmaf(Lr, Pi, Li * Pr);
    } else {
      nr = ((v.x - tx) + v.z) + ex;
      ni = ((v.y - ty) + v.w) + ey;
    }
    float qr, qi;
    if (!cdiv_f32(nr, ni, Dx, Dy, qr, qi)) { *bad = true; break; }
    dx -= qr;
    dy -= qi;
    ++it;
    const float s2 = fmaf(qr, qr, qi * qi);
    if (it == 1) {
      h2 = s2;
      thr2 = rel * rel * s2;
    } else if (s2 <= thr2 || (it >= 3 && s2 > 0.25f * prev2)) {
      break;
    }
    prev2 = s2;
  }
  if (first) *first = sqrtf(h2);
  return it;
}

// a1 + a2 in the mixed tier: the lift of k_seed_lift (Sec. 4.2) with each
// level's solves in perturbation form around the point reached at the
// previous level (one binary64 reference orbit of p_{k+1} per level instead
// of ~(1 + shrink) x 3 binary64 Newton steps).  The s_{l,n} homotopy at the
// last level stays binary64.
__global__ void k_seed_lift_mixed(PolyDev P, double lambda0, int64_t N0, int log2N0, int shrink,
                                  double2* seeds, uint8_t* __restrict__ seed_bad, DevCounters* ctr) {
  extern __shared__ float2 zsh[];
  float2* zs = zsh + threadIdx.x;
  const int stride = blockDim.x;
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long steps = 0, s32 = 0, fails = 0;
  if (j <= N0 / 2) {
    double c, s;
    unit_phase((uint64_t)j, (uint64_t)N0, c, s);
    double zr = lambda0 * c, zi = lambda0 * s;
    const float lam2 = (float)(lambda0 * lambda0);
    const float Lq = (float)(-log(lambda0) / shrink);
    double R[LIFT_RADII];
    const bool tab = shrink_radii(lambda0, shrink, R);
    bool bad = false;
    for (int k = 1; k < P.m; ++k) {
      const uint64_t num = (k >= log2N0) ? 0 : (((uint64_t)j << k) & (uint64_t)(N0 - 1));
      unit_phase(num, (uint64_t)N0, c, s);
      PolyDev Q;
      Q.kind = 0; Q.l = 0; Q.n = k + 1; Q.m = k + 1; Q.lcap = -1; Q.log2d = k;
      float4 v;
      ref_orbit(Q, zr, zi, zs, stride, v);
      float dx = 0.f, dy = 0.f;
      const float ec = (float)c, es = (float)s;
      int it = newton_target_pert(Q, zs, stride, v, dx, dy, lam2 * ec, lam2 * es, 1e-3f, 40, nullptr,
                                  false, 0.f, 0.f, 0.f, 0.f, &bad);
      for (int q = 1; q <= shrink; ++q) {
        const float rp = (float)shrink_radius(R, tab, lambda0, shrink, q - 1);
        const float r = (float)shrink_radius(R, tab, lambda0, shrink, q);
        it += newton_target_pert(Q, zs, stride, v, dx, dy, r * ec, r * es, 1e-3f, 40, nullptr, true,
                                 rp * ec, rp * es, Lq, 0.f, &bad);
      }
      steps += it;
      s32 += it;
      zr += (double)dx;
      zi += (double)dy;
    }
    if (P.kind == 1) {
      // binary64 homotopy p_m -> p_m + p_{l-1} (as in k_seed_lift)
      const int k = P.m - 1;
      const uint64_t num = (k >= log2N0) ? 0 : (((uint64_t)j << k) & (uint64_t)(N0 - 1));
      unit_phase(num, (uint64_t)N0, c, s);
      for (int a = 1; a <= 8; ++a) {
        const double alpha = a / 8.0;
        for (int t = 0; t < 40; ++t) {
          double vr, vi, dr, di, qr, qi;
          orbit_f64(P.m, P.lcap, alpha, zr, zi, vr, vi, dr, di);
          cdiv_f64(vr - lambda0 * c, vi - lambda0 * s, dr, di, qr, qi);
          if (!finite2(qr, qi)) break;
          zr -= qr;
          zi -= qi;
          ++steps;
          if (fma(qr, qr, qi * qi) <= 1e-24 * fma(zr, zr, zi * zi) + 1e-300) break;
        }
      }
    }
    if (j == 0 || j == N0 / 2) zi = 0.0;
    seeds[j] = make_double2(zr, zi);
    fails = bad ? 1 : 0;
    seed_bad[j] = bad ? 1 : 0;  // lifted again in binary64 by k_seed_repair
  }
  warp_add_u64(&ctr->walk_newton, steps);
  warp_add_u64(&ctr->seed_newton, steps);
  warp_add_u64(&ctr->steps_fp32, s32);
  warp_add_u64(&ctr->walk_fail, fails);
}

// Float-float reference orbit of the walk, anchored at c0' = the float-float
// value of c0 (hi + lo, exactly a binary64), so that no bit of the anchor is
// lost: the caller carries c0 - c0' (below 2^-47 |c0|) in delta.  Z_k
// (k < m) to shared memory in binary32, P(c0') as binary32 hi + lo.  Its
// ~1e-14 relative accuracy moves P by far less than the walk's tolerance
// (1e-2 of a sub-step) and keeps the walk off the binary64 pipe, where one
// binary64 anchor cost as much as the binary32 sub-steps it served.
template <bool CAP, int MC, int STRIDE>
__device__ __forceinline__ void ref_orbit_ff(const PolyDev& P, double c0x, double c0y, float2* zs, float4& v,
                                             double& ax, double& ay) {
  const ff cx = ff_from(c0x), cy = ff_from(c0y);
  ax = (double)cx.hi + (double)cx.lo;
  ay = (double)cy.hi + (double)cy.lo;
  ff zx{0.f, 0.f}, zy{0.f, 0.f}, capx{0.f, 0.f}, capy{0.f, 0.f};
  zs[0] = make_float2(0.f, 0.f);
  const int m = MC > 0 ? MC : P.m;
#pragma unroll 2
  for (int k = 1; k <= m; ++k) {
    const ff nx = ff_add(ff_add(ff_mul(zx, zx), ff_neg(ff_mul(zy, zy))), cx);
    const ff ny = ff_add(ff_twice(ff_mul(zx, zy)), cy);
    zx = nx;
    zy = ny;
    if (k < m) zs[k * STRIDE] = make_float2(zx.hi, zy.hi);
    if (CAP && k == P.lcap) { capx = zx; capy = zy; }
  }
  const ff vx = CAP ? ff_add(zx, capx) : zx, vy = CAP ? ff_add(zy, capy) : zy;
  v = make_float4(vx.hi, vy.hi, vx.lo, vy.lo);
}

// a3 in the mixed tier: one lane per chunk of L sub-steps, binary32
// perturbation around a float-float anchor re-taken every K sub-steps.
// Shared memory: each warp owns m rows of 32 binary32 pairs (row stride 32,
// a compile-time constant).  j0 / nch / sbase: chunks [j0, j0 + nch) only,
// start g / every written at g / every - sbase (a streamed split's piece;
// 0 / nchunks / 0 for the whole line).  MC as in k_descend_mixed.
template <bool CAP, int MC>
__global__ void k_walk_mixed(PolyDev P, double lambda0, int M, int every, int64_t L, int64_t nchunks,
                             int K, const double2* __restrict__ seeds, double2* __restrict__ starts,
                             uint8_t* __restrict__ chunk_fail, DevCounters* ctr, int64_t j0, int64_t nch,
                             int64_t sbase) {
  extern __shared__ float2 zsh[];
  __shared__ float2 ph[64];
  for (int q = threadIdx.x; q < M; q += blockDim.x) {
    double c, s;
    unit_phase((uint64_t)q, (uint64_t)M, c, s);
    ph[q] = make_float2((float)(lambda0 * c), (float)(lambda0 * s));
  }
  __syncthreads();
  const int m = MC > 0 ? MC : P.m;
  float2* zs = zsh + (threadIdx.x >> 5) * 32 * m + (threadIdx.x & 31);
  const int64_t jl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = j0 + jl;
  unsigned long long steps = 0, fails = 0;
  if (jl < nch && j < nchunks) {
    const double2 s0 = seeds[j];
    double c0x, c0y;
    float4 v;
    ref_orbit_ff<CAP, MC, 32>(P, s0.x, s0.y, zs, v, c0x, c0y);
    float dx = (float)(s0.x - c0x), dy = (float)(s0.y - c0y), h = 0.f;
    bool bad = false;
    const float Li = 6.2831853f / M;
    const int esh = __ffs(every) - 1;  // every is a power of two
    uint64_t g = (uint64_t)j * (uint64_t)L;
    int kc = K;  // sub-steps to the next anchor
    for (int64_t i = 0; i < L; ++i, ++g) {
      if ((g & (uint64_t)(every - 1)) == 0)
        starts[(int64_t)(g >> esh) - sbase] = make_double2(c0x + (double)dx, c0y + (double)dy);
      const float2 Tp = ph[g & (uint64_t)(M - 1)];
      const float2 T = ph[(g + 1) & (uint64_t)(M - 1)];
      // tight (1e-2) only on the sub-steps that end on a start, as in walk_chunk
      const float rel = (((g + 1) & (uint64_t)(every - 1)) == 0) ? 1e-2f : 1e-1f;
      steps += newton_target_walk<CAP, MC, 32>(P, zs, v, dx, dy, T.x, T.y, rel, 16, &h, Tp.x, Tp.y, Li, &bad);
      if (--kc == 0 && i + 1 < L) {  // re-anchor at the current point
        kc = K;
        const double px = c0x + (double)dx, py = c0y + (double)dy;
        ref_orbit_ff<CAP, MC, 32>(P, px, py, zs, v, c0x, c0y);
        dx = (float)(px - c0x);
        dy = (float)(py - c0y);
      }
    }
    const double cx = c0x + (double)dx, cy = c0y + (double)dy;
    if (j == nchunks - 1) starts[(int64_t)(g >> esh) - sbase] = make_double2(cx, 0.0);
    const double2 zn = seeds[j + 1];
    const double er = cx - zn.x, ei = cy - zn.y;
    const double hh = (double)h;
    if (bad || !(er * er + ei * ei <= 0.0625 * hh * hh + 1e-28)) fails = 1;
    chunk_fail[j] = (uint8_t)fails;  // walked again in binary64 by k_walk_repair
  }
  warp_add_u64(&ctr->walk_newton, steps);
  warp_add_u64(&ctr->steps_fp32, steps);
  warp_add_u64(&ctr->walk_fail, fails);
}

// The walk of p_n.  As k_walk_mixed, with fewer and shorter Newton steps:
//  - The first K orbit steps of each Newton step are the cubic of p_K around
//    the anchor (as in k_descend_mixed; here within the walk's own tolerance),
//    K the largest for which it holds within WALK_REACH sub-steps in every
//    lane of the warp (one vote a step of the anchor's orbit).  The warp
//    re-anchors early when a lane leaves that radius.
//  - The predictor extrapolates z' = P / P' along log P from the last three
//    sub-steps (Adams-Bashforth), and a sub-step that ends on no start stops
//    once the error left after a correction is small, not once a further
//    correction has shown it.
// Bound by issue (70 %) with 14 warps an SM.
// Shared memory: each warp owns m rows of 32 binary32 pairs.
constexpr float WALK_REACH = 9.5f;

struct WalkAnchor {
  float4 v;        // P(c0) as binary32 hi + lo
  float4 ab;       // A, B at K
  float cx, cy;    // C at K
  float rho2;      // the series' radius squared
  int K;           // warp-uniform
};

// The anchor's orbit at c0 (binary64) and the series for a reach R.
__device__ __forceinline__ void walk_anchor(unsigned mask, int m, double px, double py, float R2, float2* zs,
                                            WalkAnchor& w, double& ax, double& ay) {
  const ff cx = ff_from(px), cy = ff_from(py);
  ax = (double)cx.hi + (double)cx.lo;
  ay = (double)cy.hi + (double)cy.lo;
  ff zx = cx, zy = cy;
  float Ax = 1.f, Ay = 0.f, Bx = 0.f, By = 0.f, Cx = 0.f, Cy = 0.f;
  auto next = [&]() {
    const ff nx = ff_add(ff_add(ff_mul(zx, zx), ff_neg(ff_mul(zy, zy))), cx);
    const ff ny = ff_add(ff_twice(ff_mul(zx, zy)), cy);
    zx = nx;
    zy = ny;
  };
  const float R = sqrtf(R2);
  w.rho2 = 3.0e38f;
  int k = 1;
  for (; k < m - 1; ++k) {
    const float tx = zx.hi + zx.hi, ty = zy.hi + zy.hi;
    const float nCx = fmaf(tx, Cx, fmaf(-ty, Cy, 2.f * fmaf(Ax, Bx, -Ay * By)));
    const float nCy = fmaf(tx, Cy, fmaf(ty, Cx, 2.f * fmaf(Ax, By, Ay * Bx)));
    const float nBx = fmaf(tx, Bx, fmaf(-ty, By, fmaf(Ax, Ax, -Ay * Ay)));
    const float nBy = fmaf(tx, By, fmaf(ty, Bx, 2.f * Ax * Ay));
    const float nAx = fmaf(tx, Ax, fmaf(-ty, Ay, 1.f));
    const float nAy = fmaf(tx, Ay, ty * Ax);
    // |C| R^2 <= 6e-3 |A|, |B| R <= 8e-2 |A|: the dropped fourth term is ~5e-4 of
    // e at the reach, half of a start's tolerance of 1e-2 h
    const float a1 = fmaxf(fabsf(nAx), fabsf(nAy)), b1 = fmaxf(fabsf(nBx), fabsf(nBy)),
                c1 = fmaxf(fabsf(nCx), fabsf(nCy));
    const bool ok = c1 < 1e37f && b1 * R <= 8e-2f * a1 && (c1 * R) * R <= 6e-3f * a1;
    if (!__all_sync(mask, ok)) break;
    Ax = nAx; Ay = nAy; Bx = nBx; By = nBy; Cx = nCx; Cy = nCy;
    next();
  }
  w.K = k;
  if (k > 1) w.rho2 = R2;
  w.ab = make_float4(Ax, Ay, Bx, By);
  w.cx = Cx;
  w.cy = Cy;
#pragma unroll 2
  for (; k < m; ++k) {
    zs[(k - w.K) * 32] = make_float2(zx.hi, zy.hi);
    next();
  }
  w.v = make_float4(zx.hi, zy.hi, zx.lo, zy.lo);
}

// e_m and D = P' at c0 + d: the series at K, then the orbit steps K .. m-1.
__device__ __forceinline__ void walk_eval(int m, const WalkAnchor& w, const float2* zs, float dx, float dy, float& ex,
                                          float& ey, float& Dx, float& Dy) {
  const float d2x = fmaf(dx, dx, -dy * dy), d2y = 2.f * dx * dy;
  const float bx = fmaf(w.ab.z, dx, -w.ab.w * dy), by = fmaf(w.ab.z, dy, w.ab.w * dx);
  const float qx = fmaf(w.cx, d2x, -w.cy * d2y), qy = fmaf(w.cx, d2y, w.cy * d2x);
  const float tx = w.ab.x + (bx + qx), ty = w.ab.y + (by + qy);
  float e_x = fmaf(tx, dx, -ty * dy), e_y = fmaf(tx, dy, ty * dx);
  float h = __int_as_float((127 - w.K) << 23);  // 2^-K
  float g_x = h * fmaf(3.f, qx, fmaf(2.f, bx, w.ab.x)), g_y = h * fmaf(3.f, qy, fmaf(2.f, by, w.ab.y));
  auto step = [&](const float2 Z) {
    h *= 0.5f;
    const float zx = Z.x + e_x, zy = Z.y + e_y;  // p_k(c)
    const float ng_x = fmaf(zx, g_x, fmaf(-zy, g_y, h));
    const float ng_y = fmaf(zx, g_y, zy * g_x);
    const float sx = Z.x + zx, sy = Z.y + zy;  // 2 Z_k + e_k
    const float ne_x = fmaf(sx, e_x, fmaf(-sy, e_y, dx));
    const float ne_y = fmaf(sx, e_y, fmaf(sy, e_x, dy));
    e_x = ne_x; e_y = ne_y; g_x = ng_x; g_y = ng_y;
  };
  const float2* z = zs;
  const int T = m - w.K;
  for (int r = T & 3; r > 0; --r, z += 32) step(*z);
  for (int r = T >> 2; r > 0; --r, z += 128) {
    step(z[0]);
    step(z[32]);
    step(z[64]);
    step(z[96]);
  }
  const float sc = __int_as_float((127 + m) << 23);
  ex = e_x;
  ey = e_y;
  Dx = g_x * sc;
  Dy = g_y * sc;
}

__global__ void k_walk_series(PolyDev P, double lambda0, int M, int every, int64_t L, int64_t nchunks, int Kturn,
                              const double2* __restrict__ seeds, double2* __restrict__ starts,
                              uint8_t* __restrict__ chunk_fail, DevCounters* ctr, int64_t j0, int64_t nch,
                              int64_t sbase) {
  extern __shared__ float2 zsh[];
  __shared__ float2 ph[64];
  for (int q = threadIdx.x; q < M; q += blockDim.x) {
    double c, s;
    unit_phase((uint64_t)q, (uint64_t)M, c, s);
    ph[q] = make_float2((float)(lambda0 * c), (float)(lambda0 * s));
  }
  __syncthreads();
  const int m = P.m;
  float2* zs = zsh + (threadIdx.x >> 5) * 32 * m + (threadIdx.x & 31);
  const int64_t jl = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t j = j0 + jl;
  unsigned long long steps = 0, fails = 0;
  const bool mine = jl < nch && j < nchunks;
  const unsigned mask = __ballot_sync(0xffffffffu, mine);
  if (mine) {
    const double2 s0 = seeds[j];
    double c0x, c0y;
    WalkAnchor w;
    walk_anchor(mask, m, s0.x, s0.y, 3.0e37f, zs, w, c0x, c0y);  // no step length yet: the whole orbit
    float dx = (float)(s0.x - c0x), dy = (float)(s0.y - c0y), h2 = 0.f;
    bool bad = false;
    const float Li = 6.2831853f / M;
    const int esh = __ffs(every) - 1;  // every is a power of two
    uint64_t g = (uint64_t)j * (uint64_t)L;
    int kc = 1;  // sub-steps to the next anchor: the first one gives the step length
    float w1x = 0.f, w1y = 0.f, w2x = 0.f, w2y = 0.f;  // z' at the last two sub-steps
    for (int64_t i = 0; i < L; ++i, ++g) {
      if ((g & (uint64_t)(every - 1)) == 0)
        starts[(int64_t)(g >> esh) - sbase] = make_double2(c0x + (double)dx, c0y + (double)dy);
      const float2 Tp = ph[g & (uint64_t)(M - 1)];
      const float2 T = ph[(g + 1) & (uint64_t)(M - 1)];
      // a correction of r h leaves about r^2 h: r = 1e-2 on the sub-steps that
      // end on a start (as k_walk_mixed: the roots a line finds depend on its
      // starts to a few thousandths of a sub-step), r^2 = 1e-1 on the others
      const float rel2 = (((g + 1) & (uint64_t)(every - 1)) == 0) ? 1e-4f : 1e-1f;
      float prev2 = 0.f;
      int it = 0;
      while (it < 16) {
        float ex, ey, Dx, Dy, qr, qi;
        walk_eval(m, w, zs, dx, dy, ex, ey, Dx, Dy);
        bool ok;
        if (it == 0) {
          // -dz = (P - Tp) / P' - L z'_ext, L = i Li, z'_ext = z' and its extrapolation
          const float Pr = w.v.x + (w.v.z + ex), Pi = w.v.y + (w.v.w + ey);
          float er, ei, wr, wi;
          ok = cdiv_f32(((w.v.x - Tp.x) + w.v.z) + ex, ((w.v.y - Tp.y) + w.v.w) + ey, Dx, Dy, er, ei);
          ok = cdiv_f32(Pr, Pi, Dx, Dy, wr, wi) && ok;
          float gr = wr, gi = wi;
          if (i >= 2) {
            gr = fmaf(1.9166667f, wr, fmaf(-1.3333334f, w1x, 0.41666668f * w2x));
            gi = fmaf(1.9166667f, wi, fmaf(-1.3333334f, w1y, 0.41666668f * w2y));
          } else if (i == 1) {
            gr = fmaf(1.5f, wr, -0.5f * w1x);
            gi = fmaf(1.5f, wi, -0.5f * w1y);
          }
          qr = fmaf(gi, Li, er);
          qi = fmaf(-gr, Li, ei);
          w2x = w1x; w2y = w1y;
          w1x = wr; w1y = wi;
        } else {
          ok = cdiv_f32(((w.v.x - T.x) + w.v.z) + ex, ((w.v.y - T.y) + w.v.w) + ey, Dx, Dy, qr, qi);
        }
        if (!ok) { bad = true; break; }
        dx -= qr;
        dy -= qi;
        ++it;
        const float s2 = fmaf(qr, qr, qi * qi);
        if (it == 1) h2 = s2;
        else if (s2 <= rel2 * h2 || (it >= 3 && s2 > 0.25f * prev2)) break;
        prev2 = s2;
      }
      steps += it;
      const bool out = !(fmaf(dx, dx, dy * dy) <= w.rho2 * 0.7f);  // the next sub-step may leave the series
      if ((--kc == 0 || __any_sync(mask, out)) && i + 1 < L) {  // re-anchor at the current point
        kc = Kturn;
        const double px = c0x + (double)dx, py = c0y + (double)dy;
        walk_anchor(mask, m, px, py, WALK_REACH * WALK_REACH * h2, zs, w, c0x, c0y);
        dx = (float)(px - c0x);
        dy = (float)(py - c0y);
      }
    }
    const double cx = c0x + (double)dx, cy = c0y + (double)dy;
    if (j == nchunks - 1) starts[(int64_t)(g >> esh) - sbase] = make_double2(cx, 0.0);
    const double2 zn = seeds[j + 1];
    const double er = cx - zn.x, ei = cy - zn.y;
    if (bad || !(er * er + ei * ei <= 0.0625 * (double)h2 + 1e-28)) fails = 1;
    chunk_fail[j] = (uint8_t)fails;  // walked again in binary64 by k_walk_repair
  }
  warp_add_u64(&ctr->walk_newton, steps);
  warp_add_u64(&ctr->steps_fp32, steps);
  warp_add_u64(&ctr->walk_fail, fails);
}

using WalkMixedFn = void (*)(PolyDev, double, int, int, int64_t, int64_t, int, const double2*, double2*, uint8_t*,
                             DevCounters*, int64_t, int64_t, int64_t);
template <int MC>
WalkMixedFn walk_mixed_fixed(int m) {
  if constexpr (MC < 16) {
    (void)m;
    return nullptr;
  } else {
    return m == MC ? &k_walk_mixed<false, MC> : walk_mixed_fixed<MC - 1>(m);
  }
}
// ms of the walk, without and with the series: p_20 0.178 and 0.212, p_21 0.222
// and 0.246 (the line's lanes are too few, and the anchors' votes and the loop over
// a varying length add latency), p_22 0.408 and 0.365, p_24 1.63 and 1.50, p_28
// 24.9 and 19.6.  By time the line lies between p_21 and p_22; p_22 stays with the
// short orbits (MIX_LONG).
constexpr int WALK_SERIES_MIN = MIX_LONG;
WalkMixedFn walk_mixed_kernel(const PolyDev& P) {
  if (P.lcap >= 0) return &k_walk_mixed<true, 0>;
  if (P.m >= WALK_SERIES_MIN) return &k_walk_series;
  WalkMixedFn f = walk_mixed_fixed<WALK_SERIES_MIN - 1>(P.m);
  return f ? f : &k_walk_mixed<false, 0>;
}

// a4 in the mixed tier, anchors.  One reference orbit serves the descents of
// 2^gsh consecutive starts of the line (a turn for 4): the orbit of one of
// them, c0, in float-float, rounded to binary32 (Z_k), plus P(c0) as binary32
// hi + lo and the long-jump bound on |delta|.  The anchor only steers the
// binary32 descent into the basin of its root (the binary64 finish sets the
// digits), so float-float's ~1e-14 suffices and keeps this off the binary64
// pipe.
//
// The first K orbit steps of every Newton step are replaced by the cubic of
// p_K around c0: e_K = A d + B d^2 + C d^3 with A = p'_K, B = p''_K / 2, C =
// p^(3)_K / 6 at c0, carried along the anchor's orbit (A' = 2 Z A + 1, B' =
// 2 Z B + A^2, C' = 2 Z C + 2 A B).  e grows about twofold a step, to ~|P| at
// the end, so it is still small at K = m - DM_TAIL, where the dropped fourth
// term is 1e-6 of e inside |d| <= rho, |C| rho^2 = 1e-4 |A| and |B| rho =
// 1e-2 |A| (deep-zoom renderers' series approximation).  At p_28 the median
// descent needs 9 steps after the series, nine in ten 12.
//
// A warp computes the orbits of a queue range together, lane j the one of
// the j-th group, into its own slot of the buffer: Z_k of lane j at
// za[(k - K) * 32 + j] (each store instruction writes 256 contiguous bytes).
// The slots are small and are read back by the same warp moments later, so
// they stay in L2.
struct WarpSlot {
  float2* za;   // [m - K][32]
  float4* zv;   // [32] P(c0)
  float4* zab;  // [32] A, B
  float4* zcr;  // [32] C, rho^2, long-jump bound
  double2* c0;  // [32]
};
constexpr int SLOT_EXTRA = 32 * 8;  // float2 units of the four small arrays
__device__ __forceinline__ WarpSlot warp_slot(float2* wbuf, int rows, unsigned warp) {
  const size_t per = (size_t)32 * rows + SLOT_EXTRA;  // float2 units
  float2* b = wbuf + per * warp;
  WarpSlot w;
  w.c0 = (double2*)b;
  w.zv = (float4*)(b + 64);
  w.zab = (float4*)(b + 128);
  w.zcr = (float4*)(b + 192);
  w.za = b + SLOT_EXTRA;
  return w;
}
// Starts left of this go on the far list at once, and so get an anchor each.  By
// the left tip single pairs of real roots lie 5e-4 of the starts' spacing apart
// (p_24: 2.1e-13 at -2 + 8.8e-7), where binary32 around a start's own orbit just
// tells them apart and around a neighbour's does not: of 5000 levels of p_24, 276
// missed a root and had the split repeated in binary64, 144 with an anchor a start.
constexpr float DM_TIP = -1.999f;
template <bool CAP, int MC>
__device__ __forceinline__ void anchor_orbit(const PolyDev& P, int K, double2 c0, const WarpSlot& w, unsigned j) {
  const int m = MC > 0 ? MC : P.m;
  const ff cx = ff_from(c0.x), cy = ff_from(c0.y);
  ff zx = cx, zy = cy, capx{0.f, 0.f}, capy{0.f, 0.f};  // Z_1 = c0
  if (CAP && P.lcap == 1) { capx = zx; capy = zy; }
  float Ax = 1.f, Ay = 0.f, Bx = 0.f, By = 0.f, Cx = 0.f, Cy = 0.f;
  auto next = [&](int k) {  // Z_k -> Z_{k+1}
    const ff nx = ff_add(ff_add(ff_mul(zx, zx), ff_neg(ff_mul(zy, zy))), cx);
    const ff ny = ff_add(ff_twice(ff_mul(zx, zy)), cy);
    zx = nx;
    zy = ny;
    if (CAP && k + 1 == P.lcap) { capx = zx; capy = zy; }
  };
#pragma unroll 2
  for (int k = 1; k < K; ++k) {
    const float tx = zx.hi + zx.hi, ty = zy.hi + zy.hi;
    const float nCx = fmaf(tx, Cx, fmaf(-ty, Cy, 2.f * fmaf(Ax, Bx, -Ay * By)));
    const float nCy = fmaf(tx, Cy, fmaf(ty, Cx, 2.f * fmaf(Ax, By, Ay * Bx)));
    const float nBx = fmaf(tx, Bx, fmaf(-ty, By, fmaf(Ax, Ax, -Ay * Ay)));
    const float nBy = fmaf(tx, By, fmaf(ty, Bx, 2.f * Ax * Ay));
    const float nAx = fmaf(tx, Ax, fmaf(-ty, Ay, 1.f));
    const float nAy = fmaf(tx, Ay, ty * Ax);
    Ax = nAx; Ay = nAy; Bx = nBx; By = nBy; Cx = nCx; Cy = nCy;
    next(k);
  }
#pragma unroll 4
  for (int k = K; k < m; ++k) {
    w.za[(k - K) * 32 + j] = make_float2(zx.hi, zy.hi);
    next(k);
  }
  const ff vx = ff_add(zx, capx), vy = ff_add(zy, capy);
  w.zv[j] = make_float4(vx.hi, vy.hi, vx.lo, vy.lo);
  // rho^2; no bound where nothing is skipped, none for the starts at the tip
  const float rho2 = K <= 1 ? 3.0e38f : cx.hi < DM_TIP ? -1.f : series_rho2(Ax, Ay, Bx, By, Cx, Cy);
  // long jump (as in k_descend: |c| > max(4, 2|c0|)); |delta| beyond rdel implies it
  const float r0 = sqrtf(fmaf(cx.hi, cx.hi, cy.hi * cy.hi)) * 1.0001f;
  w.zab[j] = make_float4(Ax, Ay, Bx, By);
  w.zcr[j] = make_float4(Cx, Cy, rho2, fmaxf(4.f, 2.f * r0) + r0);
  w.c0[j] = c0;
}

// Newton quotient's e and D = P'(c0 + d) from the series at K and the orbit
// steps K .. m-1; z1 points to Z_K of the lane's column.
template <bool CAP, int MC, int KC, int STRIDE>
__device__ __forceinline__ void pert_eval_series(const PolyDev& P, int Kr, const float2* z1, const float4& ab, float cx,
                                                 float cy, float dx, float dy, float& ex, float& ey, float& Dx,
                                                 float& Dy) {
  const int m = MC > 0 ? MC : P.m, K = MC > 0 ? KC : Kr;
  float e_x, e_y, g_x, g_y;
  if (MC > 0 && KC == 1) {
    e_x = dx; e_y = dy; g_x = 0.5f; g_y = 0.f;
  } else {
    const float d2x = fmaf(dx, dx, -dy * dy), d2y = 2.f * dx * dy;
    // A + B d + C d^2, and A + 2 B d + 3 C d^2
    const float bx = fmaf(ab.z, dx, -ab.w * dy), by = fmaf(ab.z, dy, ab.w * dx);
    const float qx = fmaf(cx, d2x, -cy * d2y), qy = fmaf(cx, d2y, cy * d2x);
    const float sx = ab.x + (bx + qx), sy = ab.y + (by + qy);
    e_x = fmaf(sx, dx, -sy * dy);
    e_y = fmaf(sx, dy, sy * dx);
    const float h = __int_as_float((127 - K) << 23);  // 2^-K
    g_x = h * fmaf(3.f, qx, fmaf(2.f, bx, ab.x));
    g_y = h * fmaf(3.f, qy, fmaf(2.f, by, ab.y));
  }
  float ce_x = 0.f, ce_y = 0.f, cg_x = 0.f, cg_y = 0.f;
  if (CAP && P.lcap == K) { ce_x = e_x; ce_y = e_y; cg_x = g_x; cg_y = g_y; }
  auto step = [&](int k, float h) {
    const float2 Z = z1[(k - K) * STRIDE];
    const float zx = Z.x + e_x, zy = Z.y + e_y;  // p_k(c)
    const float ng_x = fmaf(zx, g_x, fmaf(-zy, g_y, h));
    const float ng_y = fmaf(zx, g_y, zy * g_x);
    const float sx = Z.x + zx, sy = Z.y + zy;  // 2 Z_k + e_k
    const float ne_x = fmaf(sx, e_x, fmaf(-sy, e_y, dx));
    const float ne_y = fmaf(sx, e_y, fmaf(sy, e_x, dy));
    e_x = ne_x; e_y = ne_y; g_x = ng_x; g_y = ng_y;
    if (CAP && k + 1 == P.lcap) { ce_x = e_x; ce_y = e_y; cg_x = g_x; cg_y = g_y; }
  };
  if constexpr (MC > 0) {
#pragma unroll
    for (int k = KC; k < MC; ++k) step(k, __int_as_float((126 - k) << 23));  // 2^-(k+1)
  } else {
    int hexp = (126 - K) << 23;  // exponent field of 2^-(k+1), k = K
#pragma unroll 4
    for (int k = K; k < P.m; ++k) {
      step(k, __int_as_float(hexp));
      hexp -= 1 << 23;
    }
  }
  const float sc = __int_as_float((127 + m) << 23);
  if (CAP) {
    ex = e_x + ce_x;
    ey = e_y + ce_y;
    const float a = P.lcap > 0 ? __int_as_float((127 + P.lcap - m) << 23) : 0.f;
    Dx = fmaf(a, cg_x, g_x) * sc;
    Dy = fmaf(a, cg_y, g_y) * sc;
  } else {
    ex = e_x;
    ey = e_y;
    Dx = g_x * sc;
    Dy = g_y * sc;
  }
}

// a4 in the mixed tier, binary32 phase (persistent, per-lane refill as in
// k_descend) over starts [0, cnt), or with LIST over list[0 ..
// *nlist).  Each lane keeps the end of its anchor's orbit (Z_K .. Z_{m-1})
// in its own column of shared memory (row k - K holds Z_k of every lane; the
// row stride DM_BS + 1 is odd, so the rows of one column fall in different
// banks).  Lanes that finished are refilled together once DM_REFILL of them
// wait (or none is running): they take the next start indices of the warp's
// range of the work queue, and a refilled lane copies its orbit from the
// warp's slot into its column (m - K independent loads, L2 hits).  When the
// range (32 groups of 2^gsh starts) runs out the warp takes the next one (one
// atomic) and computes its 32 anchor orbits with every lane (anchor_orbit):
// the orbits cost one full-width pass per 32 2^gsh starts and never travel
// through HBM.  The Newton loop is binary32 only.  Each descent runs binary32
// Newton steps to the binary32 floor and leaves (delta from its start, its
// largest squared step) in pack[] with status 3 ("finish in binary64"), or
// stops as divergent (1) / timed out (2).  One that leaves the series' radius
// goes on the far list with its state (status 5) and is continued there
// without a series (LIST, K = 1, its own start as the anchor), so that no warp
// runs the whole orbit for one of its lanes.  MC: the orbit length when fixed
// at compile time (p_n), else 0.
//
// Bound by issue (80 %) and the binary32 pipe (50 %).  p_28, 268 M starts: 53.4
// ms with an anchor a start and every orbit step, 29.6 now (29.0 if the starts
// left of DM_TIP shared too); p_24 2.93 -> 1.86.
constexpr int DM_BS = 128;     // threads per block of the binary32 descent
// Idle lanes that trigger a refill, and orbit steps after the series: the
// refill's pass (the end's record, the next orbit's copy) costs about a third of a
// Newton step.  p_28, ms of the kernel: 4 lanes 31.7, 6 30.1, 8 29.5, 11 29.1 at 12
// steps; 10 / 14 / 16 steps +5.0 / -0.3 / +0.5 at 4 lanes, 14 +0.3 at 8.
constexpr int DM_REFILL = 11;
constexpr int DM_MAX_WARPS = 16384;  // warp slots of the anchor buffer (grids are capped to fit)
constexpr int DM_TAIL = 12;
constexpr int DM_GSH = 2;  // log2 of the starts that share an anchor
// The work queue and the start indices are 32-bit.  A warp takes ranges of up to
// 32 << DM_GSH starts until one begins past the last start, so the queue ends
// below count + (warps + 1) ranges, which must not wrap: a wrapped queue would
// hand out its starts again, without an end.
constexpr int64_t DM_MAX_COUNT = 0xffd00000ll;
static_assert(DM_MAX_COUNT + (DM_MAX_WARPS + 1ll) * (32ll << DM_GSH) <= (1ll << 32), "the queue wraps");
template <bool CAP, int MC, bool LIST>
__global__ void __launch_bounds__(DM_BS) k_descend_mixed(PolyDev P, int Kr, int gsh,
                                                         const double2* __restrict__ starts, int64_t cnt,
                                                         float2* wbuf, int cap, float4* __restrict__ pack,
                                                         uint8_t* __restrict__ status, unsigned* queue,
                                                         uint32_t* list, unsigned long long* nlist,
                                                         DevCounters* ctr) {
  extern __shared__ float2 zsh[];
  constexpr int stride = DM_BS + 1;
  constexpr int KC = MC >= MIX_LONG ? MC - DM_TAIL : 1;
  const int K = MC > 0 ? KC : Kr;
  const float2* zs = zsh + threadIdx.x;  // row 0 (Z_K) of this lane's column
  const unsigned lane = threadIdx.x & 31;
  const int rows = (MC > 0 ? MC : P.m) - K;
  const unsigned n = LIST ? (unsigned)*nlist : (unsigned)cnt;
  const unsigned range = 32u << gsh;  // starts of a queue range
  const WarpSlot ws = warp_slot(wbuf, rows, (blockIdx.x * DM_BS + threadIdx.x) >> 5);
  unsigned idx = ~0u;  // this lane's start in the queue (~0u: none)
  unsigned at = 0;     // its index in starts
  float dx = 0.f, dy = 0.f, h1 = 0.f, prev2 = 0.f, rdelta = 0.f, d0x = 0.f, d0y = 0.f, rho2 = 0.f, Cx = 0.f, Cy = 0.f;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f), ab = v;
  int it = 0;
  unsigned s32 = 0, ndiv = 0, nto = 0;
  // the warp's range [pool_base, pool_base + range) and its next unused index
  // (warp-uniform; none taken yet: pool_next at the range's end)
  unsigned pool_base = 0, pool_next = range;
  bool drained = false;                   // the queue is empty (warp-uniform)
  // a refilled lane with start i of the range in the slot: its orbit into
  // its column, and the state of a new descent
  auto take_orbit = [&](unsigned i) {
    const unsigned j = (i - pool_base) >> gsh;
    float2* dst = zsh + threadIdx.x;
    if (MC > 0) {
#pragma unroll
      for (int k = 0; k < (MC > 0 ? MC - KC : 1); ++k) dst[k * stride] = ws.za[k * 32 + j];
    } else {
      for (int k = 0; k < rows; ++k) dst[k * stride] = ws.za[k * 32 + j];
    }
    v = ws.zv[j];
    ab = ws.zab[j];
    const float4 cr = ws.zcr[j];
    Cx = cr.x;
    Cy = cr.y;
    rho2 = cr.z;
    rdelta = cr.w;
    at = LIST ? list[i] : i;
    if (LIST) {  // go on from where the series ended
      const float4 q = pack[at];
      dx = q.x;
      dy = q.y;
      h1 = q.z;
      it = __float_as_int(q.w);
      prev2 = 3.0e38f;
      d0x = d0y = 0.f;
    } else {
      const double2 s0 = starts[at], c0 = ws.c0[j];
      // truncated to 2^-23 of the difference, the order of binary32's rounding of
      // the steps' delta; zero for the anchor itself
      d0x = f32_trunc(s0.x - c0.x);
      d0y = f32_trunc(s0.y - c0.y);
      dx = d0x;
      dy = d0y;
      it = 0;
      prev2 = 0.f;
      h1 = 0.f;
    }
  };
  int outcome = 0;  // >= 0: the lane has no running descent (its last one ended so)
  for (;;) {
    const unsigned wait = __ballot_sync(0xffffffffu, outcome >= 0);
    // write the ended descents and refill their lanes together
    if (__popc(wait) >= (drained ? 32 : DM_REFILL)) {
      if (outcome >= 0 && idx < n) {
        pack[at] = make_float4(dx - d0x, dy - d0y, h1, __int_as_float(it));
        status[at] = (uint8_t)outcome;
        ndiv += outcome == 1;
        nto += outcome == 2;
        if (!LIST && outcome == 5) list[atomicAdd(nlist, 1ull)] = at;
        idx = ~0u;
      }
      if (drained) break;
      const unsigned R = __popc(wait);
      // the r-th lane that needs a start takes the r-th unused index of the
      // range, then of the next range
      const bool mine = outcome >= 0;
      const unsigned r_me = __popc(wait & lanemask_lt());
      const unsigned rem = pool_base + range - pool_next;
      if (mine && r_me < rem) {
        idx = pool_next + r_me;
        if (idx < n) take_orbit(idx);
      }
      if (rem >= R) {
        pool_next += R;
      } else {
        __syncwarp();  // the copies above have read the slot
        unsigned g = 0;
        if (lane == 0) g = atomicAdd(queue, range);
        g = __shfl_sync(0xffffffffu, g, 0);
        // the group's anchor: its middle start (of those that exist)
        const unsigned first = g + (lane << gsh);
        if (first < n) {
          const unsigned a = min(first + ((1u << gsh) >> 1), n - 1u);
          anchor_orbit<CAP, MC>(P, K, starts[LIST ? list[a] : a], ws, lane);
        }
        __syncwarp();  // the slot is written before any lane reads it
        pool_base = g;
        pool_next = g + (R - rem);
        if (mine && r_me >= rem) {
          idx = g + (r_me - rem);
          if (idx < n) take_orbit(idx);
        }
      }
      // the queue is drained once a lane's index lies past its end
      if (mine) outcome = idx < n ? -1 : 0;
      drained = __any_sync(0xffffffffu, mine && idx >= n);
    }
    if (outcome < 0) {
      float ex, ey, Dx, Dy, qr, qi;
      if (!LIST && !(fmaf(dx, dx, dy * dy) <= rho2)) {
        outcome = 5;  // beyond the series: continued on the far list
      } else {
        pert_eval_series<CAP, MC, KC, stride>(P, K, zs, ab, Cx, Cy, dx, dy, ex, ey, Dx, Dy);
        const float nr = (v.x + v.z) + ex, ni = (v.y + v.w) + ey;
        if (!cdiv_f32(nr, ni, Dx, Dy, qr, qi)) {
          outcome = 3;  // out of binary32 range: binary64 decides
        } else {
          dx -= qr;
          dy -= qi;
          ++it;
          ++s32;
          const float s2 = fmaf(qr, qr, qi * qi);
          h1 = fmaxf(h1, s2);  // largest step so far
          if (!(fmaf(dx, dx, dy * dy) <= rdelta * rdelta)) outcome = 1;
          // binary32 floor: the step is 1e-5 of the descent's scale, or it
          // stopped shrinking once already below 1e-3 of it
          else if (s2 <= 1e-10f * h1 || (s2 <= 1e-6f * h1 && s2 > 0.25f * prev2)) outcome = 3;
          else if (it >= cap) outcome = 2;
          prev2 = s2;
        }
      }
    }
  }
  warp_add_u64(&ctr->desc_newton, s32);
  warp_add_u64(&ctr->desc_fp32, s32);
  warp_add_u64(&ctr->steps_fp32, s32);
  warp_add_u64(&ctr->n_diverge, ndiv);
  warp_add_u64(&ctr->n_timeout, nto);
}

using DescMixedFn = void (*)(PolyDev, int, int, const double2*, int64_t, float2*, int, float4*, uint8_t*, unsigned*,
                             uint32_t*, unsigned long long*, DevCounters*);

// The instantiation for a polynomial: p_n with 16 <= n <= 33 has its orbit
// length fixed at compile time; everything else runs the general loop.
template <int MC>
DescMixedFn desc_mixed_fixed(int m) {
  if constexpr (MC < 16) {
    (void)m;
    return nullptr;
  } else {
    return m == MC ? &k_descend_mixed<false, MC, false> : desc_mixed_fixed<MC - 1>(m);
  }
}
DescMixedFn desc_mixed_kernel(const PolyDev& P) {
  if (P.lcap >= 0) return &k_descend_mixed<true, 0, false>;
  DescMixedFn f = desc_mixed_fixed<33>(P.m);
  return f ? f : &k_descend_mixed<false, 0, false>;
}

// a4 in the mixed tier, binary64 finish, once per root.
//
// About three in four descents repeat a root (Table newtonSteps), and the
// repeats come from starts anywhere along the line, not only from the
// neighbouring ones.  The binary32 end points of two descents that reached
// the same root agree to the binary32 floor (~1e-5 of the descent's
// largest step), while distinct roots sit at distances comparable to that
// step.  So the end points, conjugate-folded, are sorted by Re, and an end
// point that lies within FINISH_SAME (1e-4) of the smaller of the two
// descent scales from one of its FINISH_SCAN sorted predecessors follows
// that predecessor: only the head of each group gets the binary64 Newton
// steps, and followers take the head's result (the root set would merge
// them anyway).  A wrong merge can only drop one of the c_L descents of a
// root; the count check then reports it and the tier falls back to
// binary64 (measured: 3e-3 instead of 1e-4 already merges distinct roots
// at p_24).  A group whose scan would run past FINISH_SCAN predecessors
// gets a head of its own: one more finish, never a wrong merge.
constexpr float FINISH_SAME2 = 1e-8f;  // (1e-4)^2 of the squared scale h1
constexpr int FINISH_SCAN = 32;

// The left tip c = -2 (Sec. 6.3.2): the real roots there close in on one
// another faster than the binary32 descents resolve (at p_30 two real roots
// 1.4e-12 apart near -2 + 3.9e-4, one of them reached by no binary32
// descent).  Descents that end within tip_box of -2 are redone in binary64
// from their start (status 4).  Near -2 the real roots of a degree-d
// polynomial of the family are spaced as sqrt(c + 2) / d, so the region of
// spacings below a fixed threshold shrinks as 1 / d^2: tip_box =
// 1e-3 (d / 2^29)^2, 2.5 times the p_30 case (0.8 % of the descents there).
inline double tip_box(const PolyDev& P) { return 1e-3 * exp2(2.0 * (P.log2d - 29)); }
// Sort keys of the binary32 end points: Re in fixed point, 2^-37 per unit
// over [-2.25, 1.75) (every root of the family lies in Re in [-2, 1/4]),
// FINISH_KEY_BITS = 40 bits, so that five radix passes order them.  The map
// c -> floor((c + 2.25) 2^37) is monotone (non-decreasing), so the sort
// orders the end points by Re up to one bucket, FINISH_BUCKET wide.
constexpr int FINISH_KEY_BITS = 40;
constexpr double FINISH_BUCKET = 7.275957614183426e-12;  // 2^-37
constexpr uint64_t TIP_KEY = (1ull << FINISH_KEY_BITS) - 2;  // above every finite key, below the rest
constexpr uint64_t REST_KEY = (1ull << FINISH_KEY_BITS) - 1;
// The key's bits above FINISH_KEY_BITS carry the descent's squared scale
// h1 (binary32, its low 8 bits dropped: rounded down, so the grouping test
// only tightens) through the sort, which orders the low 40 bits only: the
// group scan reads it from the sorted keys instead of gathering it.
__device__ __forceinline__ uint64_t with_scale(uint64_t key, float h1) {
  return key | ((uint64_t)(__float_as_uint(fmaxf(h1, 0.f)) >> 8) << FINISH_KEY_BITS);
}
__device__ __forceinline__ float key_scale(uint64_t key) {
  return __uint_as_float((unsigned)(key >> FINISH_KEY_BITS) << 8);
}
__device__ __forceinline__ uint64_t finish_key(double re) {
  // floor((re + 2.25) 2^37) = floor(re 2^37) + 2.25 2^37, the first term an
  // arithmetic shift of re's significand (integer pipe only: on GB300 the
  // binary64 pipe issues at 1/64 of the binary32 rate)
  const long long b = __double_as_longlong(re);
  const int E = (int)((b >> 52) & 0x7ff);
  const long long M = (b & 0x000fffffffffffffll) | (E ? 0x0010000000000000ll : 0ll);
  const int sh = min(63, 1038 - max(E, 1));  // re 2^37 = M 2^(E' - 1038), E' = max(E, 1)
  long long k;
  if (sh <= 0) k = b < 0 ? -0x7fffffffffffll : 0x7fffffffffffll;  // |re| >= 2^14: clamped below
  else if (b >= 0) k = M >> sh;
  else k = -(long long)(((unsigned long long)M + ((1ull << sh) - 1ull)) >> sh);
  k += 309237645312ll;  // 2.25 2^37
  const long long top = (long long)(1ull << (FINISH_KEY_BITS - 1)) - 1;
  return (uint64_t)(k < 0 ? 0 : k > top ? top : k);
}

// c32 = start + delta in binary64, folded into the upper half for the
// descents to finish (status 3), whose Re is their sort key; the others
// keep their end point and sort after them.  Descents that end in the tip
// box keep their start instead (status 4, key TIP_KEY, so that the stable
// sort lists them in index order between the two).  Counts both.
__global__ void k_c32_keys(int64_t count, double box, double2* __restrict__ starts, const float4* __restrict__ pack,
                           uint8_t* __restrict__ status, uint64_t* __restrict__ keys,
                           uint32_t* __restrict__ vals, DevCounters* ctr) {
  // grid-stride over a bounded grid: the counts reach the two counters in a
  // few thousand atomics, not one per warp of the 2^28 descents.  Four
  // elements a round, all loaded before any is stored (the loads of a round
  // are in flight together; a load of starts cannot pass an earlier store
  // to it).
  constexpr int U = 4;
  unsigned long long n3 = 0, n4 = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const uint64_t kx = f64_key(-2.0 + box), ky = f64_key(box);
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i0 < count; i0 += U * stride) {
    float4 q[U];
    double2 c0[U];
    uint8_t st[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * stride;
      if (i < count) {
        q[u] = pack[i];
        c0[u] = starts[i];
        st[u] = status[i];
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + u * stride;
      if (i >= count) break;
      // the binary32 deltas widen on the integer pipe (f64_of_f32: a
      // subnormal delta, far below half an ulp of the start, becomes 0)
      double2 c = make_double2(c0[u].x + f64_of_f32(q[u].x), c0[u].y + f64_of_f32(q[u].y));
      const bool fin = st[u] == 3;
      // Im c < 0 (sign bit set, not -0): fold into the upper half
      const long long by = __double_as_longlong(c.y);
      if (fin && by < 0 && (by << 1) != 0) c.y = __longlong_as_double(by & 0x7fffffffffffffffll);
      uint64_t key = REST_KEY;
      // the tip box, compared on order-preserving integer keys
      if (fin && f64_key(c.x) < kx && f64_key(c.y) < ky) {
        status[i] = 4;  // redone in binary64 from c0
        key = TIP_KEY;
        ++n4;
      } else {
        starts[i] = c;
        if (fin) {
          key = with_scale(finish_key(c.x), q[u].z);
          ++n3;
        }
      }
      keys[i] = key;
      vals[i] = (uint32_t)i;
    }
  }
  warp_add_u64(&ctr->n_c32_fin, n3);
  warp_add_u64(&ctr->n_tip64, n4);
}

// list2 of the descents to redo in binary64: sorted positions n3 .. n3+n4
// (status 4, in index order)
__global__ void k_tip_list(const uint32_t* __restrict__ vals, const unsigned long long* __restrict__ n3,
                           const unsigned long long* __restrict__ n4, uint32_t* __restrict__ list2) {
  const int64_t a = (int64_t)*n3, m = (int64_t)*n4;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x)
    list2[t] = vals[a + t];
}

// The descents redone in binary64 join the list of finished heads
// (list[*nlist ..]) and are counted; k_finish_count then moves *nlist.
// Grid-stride: the list is about 1 % of the descents.
__global__ void k_finish_append(const uint32_t* __restrict__ list2, const unsigned long long* __restrict__ n2,
                                uint32_t* __restrict__ list, const unsigned long long* __restrict__ nlist,
                                int64_t cap, const uint8_t* __restrict__ status, DevCounters* ctr) {
  const int64_t m = (int64_t)*n2, base = (int64_t)*nlist;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned long long nconv = 0, ndiv = 0, nto = 0;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < m && base + t < cap; t += stride) {
    const uint32_t i = list2[t];
    list[base + t] = i;
    const uint8_t st = status[i];
    nconv += st == 0;
    ndiv += st == 1;
    nto += st == 2;
  }
  warp_add_u64(&ctr->n_conv, nconv);
  warp_add_u64(&ctr->n_diverge, ndiv);
  warp_add_u64(&ctr->n_timeout, nto);
}
__global__ void k_finish_count(unsigned long long* nlist, const unsigned long long* n2, int64_t cap) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const unsigned long long t = *nlist + *n2;
    *nlist = t < (unsigned long long)cap ? t : (unsigned long long)cap;
  }
}

// head[p] = 1 for a sorted position p whose end point starts a group;
// link[p] = p - q for a follower of the sorted position q (0 otherwise)
__global__ void k_finish_heads(int64_t count, const uint32_t* __restrict__ vals,
                               const uint64_t* __restrict__ skeys, const double2* __restrict__ c32,
                               const unsigned long long* __restrict__ n3, uint32_t* __restrict__ head,
                               uint8_t* __restrict__ link) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= count) return;
  uint32_t h = 0;
  uint8_t lk = 0;
  // the n3 end points to finish (status 3) sort first: their keys lie below TIP_KEY
  if (p < (int64_t)*n3) {
    const uint32_t i = vals[p];
    h = 1;
    const double2 a = c32[i];
    const float ha = key_scale(skeys[p]);
    const float reach2 = FINISH_SAME2 * ha;  // min(ha, hb) <= ha
    for (int k = 1; k <= FINISH_SCAN && k <= p; ++k) {
      const uint32_t j = vals[p - k];
      const double2 b = c32[j];
      // the differences in binary64, the tests in binary32 (the differences
      // truncated on the integer pipe: never larger, so the scan never stops
      // early)
      const float ex = f32_trunc(a.x - b.x), ey = f32_trunc(a.y - b.y);
      // sorted by Re up to one bucket: every earlier entry lies below
      // b.x + FINISH_BUCKET, so none is within reach once ex - bucket is
      const float eb = ex - (float)FINISH_BUCKET;
      if (eb > 0.f && eb * eb > reach2) break;
      const float sc = fminf(ha, key_scale(skeys[p - k]));
      if (fmaf(ex, ex, ey * ey) <= FINISH_SAME2 * sc) {
        h = 0;
        lk = (uint8_t)k;
        break;
      }
    }
  }
  head[p] = h;
  link[p] = lk;
}

// list[pos[p]] = original index of the head at sorted position p
__global__ void k_finish_list(int64_t count, const uint32_t* __restrict__ head, const uint32_t* __restrict__ pos,
                              const uint32_t* __restrict__ vals, uint32_t* __restrict__ list) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < count && head[p]) list[pos[p]] = vals[p];
}

// Binary64 Newton steps (eq. Newton) from each head's binary32 end point
// until |step| < tol or the next step, predicted, is below tol / 4 (normally
// one step), or the rounding floor.  Persistent, with per-lane refill by warp
// vote (as k_descend): lanes that finished take the next heads of the list
// together once FIN_REFILL wait, so the warp never waits for its slowest
// finish (one to six steps) before starting new ones.
//
// FX: the value in fixed point (mt_fix.cuh; the end points lie near roots, in
// its range), the derivatives in binary32, as without FX, where the value is
// binary64 (the polynomials kept there).  Bound: the integer multiply-add
// pipe (56 %) and issue (70 %); in binary64 that pipe's 3 FMA a step, 16 clocks
// a warp each, with the heads outside the line repeating six steps.  p_24, 4.5 M
// heads: 0.865 -> 0.282 ms, 0.01 of it the binary64 step of the small imaginary
// parts (axis_step) (p_28 15.1 -> 4.65 without it; not taken there, FIN_FX_MAXM).
constexpr int FIN_FB = 28;
constexpr unsigned FIN_REFILL = 6;
template <bool FX>
__global__ void __launch_bounds__(128) k_finish_f64(PolyDev P, const uint32_t* __restrict__ list,
                                                    const unsigned long long* __restrict__ nlist,
                                                    int64_t cap_list, double tol2, int cap, unsigned axis_lo,
                                                    const double2* __restrict__ c32,
                                                    double2* __restrict__ cand,
                                                    uint8_t* __restrict__ status,
                                                    unsigned long long* queue, DevCounters* ctr) {
  const unsigned lane = threadIdx.x & 31;
  const unsigned nl = (unsigned)((int64_t)*nlist < cap_list ? (int64_t)*nlist : cap_list);  // < 2^32
  const float tol2f = f32_trunc(tol2), tol2q = 0.0625f * tol2f;  // tol^2, (tol / 4)^2
  uint32_t at = 0;  // the candidate of this lane's finish
  double zx = 0.0, zy = 0.0;
  long long X = 0, Y = 0;
  float prev2 = 3.0e38f;
  int it = 0, outcome = 0;  // >= 0: no running finish (have: its result waits to be written)
  bool have = false;
  bool drained = false;  // warp-uniform: the list is handed out
  unsigned s64 = 0;
  __shared__ uint32_t axis_buf[FX ? 4 : 1][64];
  uint32_t* abuf = axis_buf[FX ? threadIdx.x >> 5 : 0];
  unsigned na = 0;
  auto axis = [&]() {
    uint32_t i;
    if (axis_pop(abuf, na, i)) cand[i] = axis_step(P.m, P.lcap, cand[i]);
  };
  for (;;) {
    const unsigned wait = __ballot_sync(0xffffffffu, outcome >= 0);
    if (__popc(wait) >= (drained ? 32u : FX ? FIN_REFILL : 1u)) {
      bool near = false;
      if (have && outcome >= 0) {
        if (FX) {
          zx = fx_to_f64<FIN_FB>(X);
          zy = fx_to_f64<FIN_FB>(Y);
          near = outcome == 0 && axis_near(make_double2(zx, zy), axis_lo);
        }
        cand[at] = make_double2(zx, zy);
        status[at] = (uint8_t)outcome;
        have = false;
      }
      if (FX) {
        axis_push(abuf, na, near, at);
        if (na >= 32u) axis();
      }
      if (drained) break;
      unsigned long long b0 = 0;
      if (lane == (unsigned)(__ffs(wait) - 1)) b0 = atomicAdd(queue, (unsigned long long)__popc(wait));
      b0 = __shfl_sync(0xffffffffu, b0, __ffs(wait) - 1);
      if (outcome >= 0) {
        const unsigned long long t = b0 + __popc(wait & lanemask_lt());
        if (t < nl) {
          at = list[t];
          const double2 z = c32[at];
          zx = z.x;
          zy = z.y;
          if (FX) {
            X = fx_from_f64<FIN_FB>(zx);
            Y = fx_from_f64<FIN_FB>(zy);
          }
          it = 0;
          prev2 = 3.0e38f;
          outcome = FX && !(fx_fits<FIN_FB>(zx) && fx_fits<FIN_FB>(zy)) ? 1 : -1;
          have = true;
        }
      }
      if (b0 + __popc(wait) >= nl) drained = true;
    }
    if (outcome < 0) {
      float dr, di, kr, ki, fvx, fvy;
      double vr = 0.0, vi = 0.0;
      bool in = true;
      if (FX) {
        long long Wr, Wi;
        in = fx_value_d32_k<FIN_FB>(P.m, X, Y, Wr, Wi, dr, di, kr, ki);
        fvx = fx_to_f32<FIN_FB>(Wr);
        fvy = fx_to_f32<FIN_FB>(Wi);
      } else {
        orbit_f64_d32_k(P.m, P.lcap, zx, zy, vr, vi, dr, di, kr, ki);
        fvx = f32_trunc(vr);
        fvy = f32_trunc(vi);
      }
      // the quotient in binary32: the derivative is binary32 already, and a
      // step accurate to 1e-7 of itself leaves ~1e-7 q besides the quadratic
      // K q^2 -- far below tol for the q ~ 1e-5 of a descent's scale that
      // the binary32 phase leaves; 64 bits only for the value and z - q
      float qr, qi;
      const bool ok = cdiv_f32s(fvx, fvy, dr, di, qr, qi);
      if (!FX && !ok) {
        double qd, qe;  // a derivative out of binary32's scaled range: binary64
        cdiv_f64(vr, vi, (double)dr, (double)di, qd, qe);
        qr = f32_trunc(qd);
        qi = f32_trunc(qe);
      }
      float fzx, fzy;
      bool finite;
      if (FX) {
        finite = ok && fabsf(qr) < 2.f && fabsf(qi) < 2.f;
        if (finite) {
          X -= fx_from_ff<FIN_FB>(ff{qr, 0.f});
          Y -= fx_from_ff<FIN_FB>(ff{qi, 0.f});
          finite = fx_in<FIN_FB>(X) && fx_in<FIN_FB>(Y);
        }
        fzx = (float)fx_hi(X) * fx_pow2f(-FIN_FB);
        fzy = (float)fx_hi(Y) * fx_pow2f(-FIN_FB);
      } else {
        zx -= f64_of_f32(qr);
        zy -= f64_of_f32(qi);
        fzx = f32_trunc(zx);
        fzy = f32_trunc(zy);
        finite = finite2(zx, zy);
      }
      ++it;
      ++s64;
      const float s2 = fmaf(qr, qr, qi * qi);
      // the next step, predicted: q^2 P''/(2P') (binary32); NaN or inf never accepts
      const float q2r = fmaf(qr, qr, -qi * qi), q2i = 2.f * qr * qi;
      const float pr = fmaf(q2r, kr, -q2i * ki), pi = fmaf(q2r, ki, q2i * kr);
      const float pred2 = fmaf(pr, pr, pi * pi);
      // binary64 rounding floor (16 ulp of the larger of 1 and |z|), in binary32
      const float fl = (1.f + fabsf(fzx) + fabsf(fzy)) * 3.552713678800501e-15f;
      // an orbit that leaves the fixed range (|p_k| >= 4 before the end, about 1 %
      // of the heads: binary32 descents that ended outside the line, status 3
      // with P' beyond binary32) is more steps from any root than the cap allows
      if (!in) outcome = 2;
      else if (!finite || fmaf(fzx, fzx, fzy * fzy) > 1e4f) outcome = 1;
      else if (s2 < tol2f) outcome = 0;
      // quadratic regime (the next step under a quarter of this one) and the
      // next step under tol / 4: c - q is the root to within tol / 4
      else if (pred2 <= tol2q && pred2 <= 0.0625f * s2) outcome = 0;
      else if (s2 >= 0.25f * prev2 && s2 < fl * fl) outcome = 0;  // rounding floor
      else if (it >= cap) outcome = 2;
      prev2 = s2;
    }
  }
  if (FX && na) axis();
  warp_add_u64(&ctr->desc_newton, s64);
  warp_add_u64(&ctr->finish_newton, s64);
}

// Followers take their head's result (following the links back in sorted
// order, each at most FINISH_SCAN positions); descents discarded by the
// binary32 phase (status 1, 2, already counted there) keep their binary32
// end point.  The outcomes of the finished groups are counted here.
__global__ void k_finish_followers(int64_t count, const uint32_t* __restrict__ vals,
                                   const uint32_t* __restrict__ head, const uint8_t* __restrict__ link,
                                   const double2* __restrict__ c32, double2* __restrict__ cand,
                                   uint8_t* __restrict__ status, DevCounters* ctr) {
  unsigned long long nconv = 0, ndiv = 0, nto = 0;
  // sorted positions below n3 hold the end points that were to finish (status 3)
  const int64_t n3 = (int64_t)ctr->n_c32_fin;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < count;
       p += (int64_t)gridDim.x * blockDim.x) {  // grid-stride: few counter atomics
    const uint32_t i = vals[p];
    bool finished = head[p] != 0;
    uint8_t st = finished ? status[i] : (p < n3 ? 3 : 0);  // a head's outcome of the finish
    if (p < n3 && !finished) {
      int64_t q = p - link[p];
      for (int g = 0; g < 4096 && !head[q] && link[q]; ++g) q -= link[q];
      if (head[q]) {
        const uint32_t j = vals[q];
        cand[i] = cand[j];
        st = status[j];
      } else {  // unresolved (never seen): no root from this descent
        cand[i] = c32[i];
        st = 2;
      }
      status[i] = st;
      finished = true;
    } else if (!finished) {
      cand[i] = c32[i];
    }
    if (finished) {
      nconv += st == 0;
      ndiv += st == 1;
      nto += st == 2;
    }
  }
  warp_add_u64(&ctr->n_conv, nconv);
  warp_add_u64(&ctr->n_diverge, ndiv);
  warp_add_u64(&ctr->n_timeout, nto);
}

cudaError_t launch_seed_lift_mixed(const PolyDev& P, double lambda0, int64_t N0, int shrink_steps,
                                   double2* seeds, uint8_t* seed_bad, DevCounters* ctr, cudaStream_t s) {
  if (P.m > MIX_MAXM) return cudaErrorInvalidValue;
  int log2N0 = 0;
  while ((int64_t(1) << log2N0) < N0) ++log2N0;
  const int64_t n = N0 / 2 + 1;
  const int bs = 128;
  const size_t smem = (size_t)P.m * bs * sizeof(float2);
  MT_COUNT_LAUNCH(1);
  k_seed_lift_mixed<<<(unsigned)((n + bs - 1) / bs), bs, smem, s>>>(P, lambda0, N0, log2N0,
                                                                    shrink_steps, seeds, seed_bad, ctr);
  return cudaGetLastError();
}

cudaError_t launch_walk_mixed(const PolyDev& P, double lambda0, int M, int every, int64_t L,
                              int64_t nchunks, int K, const double2* seeds, double2* starts,
                              uint8_t* chunk_fail, DevCounters* ctr, cudaStream_t s, int block, int64_t j0,
                              int64_t nch) {
  if (P.m > MIX_MAXM) return cudaErrorInvalidValue;
  if (nch < 0) nch = nchunks - j0;
  if (nch <= 0) return cudaSuccess;
  const int bs = (block >= 32 && block <= 256 && block % 32 == 0) ? block : 64;
  const size_t smem = (size_t)P.m * bs * sizeof(float2);
  const int64_t grid = (nch + bs - 1) / bs;
  const WalkMixedFn kwalk = walk_mixed_kernel(P);
  MT_COUNT_LAUNCH(1);
  cudaError_t e = ktimer_begin(KS_WALK, s);
  if (e != cudaSuccess) return e;
  kwalk<<<(unsigned)grid, bs, smem, s>>>(P, lambda0, M, every, L, nchunks, K, seeds, starts, chunk_fail, ctr, j0,
                                         nch, j0 * L / every);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return ktimer_end(s);
}

// The anchor buffer: one slot of 32 orbits per warp of the descent's grid
// (at most DM_MAX_WARPS warps).
size_t mixed_anchor_bytes(const PolyDev& P, int64_t count) {
  (void)count;
  const int m1 = P.m > 1 ? P.m - 1 : 1;
  return (size_t)DM_MAX_WARPS * ((size_t)32 * m1 + SLOT_EXTRA) * sizeof(float2) + 256;
}

// One launch of the binary32 descent over starts [0, count), or over the far
// list (list != nullptr with LIST kernels).
static cudaError_t launch_dm(DescMixedFn kern, const PolyDev& P, int K, int gsh, const double2* starts, int64_t count,
                             float2* wbuf, int cap, float4* pack, uint8_t* status, uint32_t* list,
                             unsigned long long* nlist, DevCounters* ctr, cudaStream_t s) {
  const int bs = DM_BS;
  const size_t smem = (size_t)std::max(1, P.m - K) * (bs + 1) * sizeof(float2);
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024 &&  // long orbits: opt in to more than 48 KB
      (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess)
    return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, bs, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int64_t grid = (int64_t)device_sm_count() * per_sm;
  const int64_t need = (count + bs - 1) / bs;
  if (grid > need) grid = need;
  if (grid > DM_MAX_WARPS / (bs / 32)) grid = DM_MAX_WARPS / (bs / 32);
  unsigned* q = (unsigned*)&ctr->queue_head;
  if ((e = cudaMemsetAsync(q, 0, sizeof(*q), s)) != cudaSuccess) return e;
  MT_COUNT_LAUNCH(1);
  if ((e = ktimer_begin(KS_DESC32, s)) != cudaSuccess) return e;
  kern<<<(unsigned)grid, bs, smem, s>>>(P, K, gsh, starts, count, wbuf, cap, pack, status, q, list, nlist, ctr);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return ktimer_end(s);
}

cudaError_t launch_descend_mixed(const PolyDev& P, double2* starts, int64_t count, double tol, int cap, double eps,
                                 double2* cand, uint8_t* status, void* anchors, const FinishScratch& fin,
                                 DevCounters* ctr, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  if (P.m > MIX_MAXM || count > DM_MAX_COUNT) return cudaErrorInvalidValue;
  const int bs = DM_BS;
  cudaError_t e = cudaSuccess;
  float2* wbuf = (float2*)anchors;
  float4* pack = (float4*)cand;  // (delta, scale) until the finish writes the roots
  {
    // s_{l,n} keeps an anchor per start and the whole orbit: its line lies at
    // |s| = 100, and binary32 relative to a neighbour's delta lost tip roots
    // (s_{6,12}: none of 7 levels without, 3 with).
    const bool shared = P.kind == 0 && P.m >= MIX_LONG;
    const int K = shared ? P.m - DM_TAIL : 1;
    const int gsh = shared ? DM_GSH : 0;
    uint32_t* far = fin.pos;  // free until the finish's scan
    unsigned long long* nfar = fin.nheads;
    if ((e = cudaMemsetAsync(nfar, 0, sizeof(*nfar), s)) != cudaSuccess) return e;
    if ((e = launch_dm(desc_mixed_kernel(P), P, K, gsh, starts, count, wbuf, cap, pack, status, far, nfar, ctr, s)) !=
        cudaSuccess)
      return e;
    if (K > 1 && (e = launch_dm(&k_descend_mixed<false, 0, true>, P, 1, 0, starts, count, wbuf, cap, pack, status, far,
                                nfar, ctr, s)) != cudaSuccess)
      return e;
  }
  // binary64 finish, once per group of end points on the same root
  const unsigned nb = (unsigned)((count + bs - 1) / bs);
  unsigned long long* n2 = &ctr->n_tip64;
  if ((e = cudaMemsetAsync(n2, 0, sizeof(*n2), s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(&ctr->n_c32_fin, 0, sizeof(*n2), s)) != cudaSuccess) return e;
  MT_COUNT_LAUNCH(1);
  const unsigned egrid = std::min<unsigned>(nb, (unsigned)device_sm_count() * 16);  // grid-stride kernels
  k_c32_keys<<<egrid, bs, 0, s>>>(count, tip_box(P), starts, pack, status, fin.keys, fin.vals, ctr);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const uint64_t* skeys = nullptr;  // the sorted keys
  {
    bool in_alt = false;
    if ((e = radix_sort_bits(fin.keys, fin.vals, fin.keys_alt, fin.vals_alt, count, fin.radix_tmp, 0,
                             FINISH_KEY_BITS, &in_alt, s)) != cudaSuccess)
      return e;
    // the permutation is read from vals (vals_alt becomes the head list)
    if (in_alt && (e = cudaMemcpyAsync(fin.vals, fin.vals_alt, (size_t)count * sizeof(uint32_t),
                                       cudaMemcpyDeviceToDevice, s)) != cudaSuccess)
      return e;
    skeys = in_alt ? fin.keys_alt : fin.keys;
  }
  MT_COUNT_LAUNCH(1);
  k_finish_heads<<<nb, bs, 0, s>>>(count, fin.vals, skeys, starts, &ctr->n_c32_fin, fin.head, fin.link);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = launch_exclusive_scan(fin.head, fin.pos, count, fin.scan_tmp, fin.nheads, s)) != cudaSuccess) return e;
  MT_COUNT_LAUNCH(1);
  k_finish_list<<<nb, bs, 0, s>>>(count, fin.head, fin.pos, fin.vals, fin.list);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  {
    // persistent: 8 warps per SM keep the binary64 pipe busy, 24 the integer
    // pipes (as k_descend)
    const bool fx = P.fx && P.kind == 0 && !mixed_short(P) && P.m <= FIN_FX_MAXM;
    const auto kfin = fx ? &k_finish_f64<true> : &k_finish_f64<false>;
    int fin_sm = 0;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fin_sm, kfin, bs, 0)) != cudaSuccess) return e;
    if (fin_sm > (fx ? 6 : 2)) fin_sm = fx ? 6 : 2;
    if (fin_sm < 1) fin_sm = 1;
    int64_t fgrid = (int64_t)device_sm_count() * fin_sm;
    if (fgrid > (int64_t)nb) fgrid = (int64_t)nb;
    unsigned long long* q = &ctr->queue_head;
    if ((e = cudaMemsetAsync(q, 0, sizeof(*q), s)) != cudaSuccess) return e;
    MT_COUNT_LAUNCH(1);
    if ((e = ktimer_begin(KS_FINISH, s)) != cudaSuccess) return e;
    kfin<<<(unsigned)fgrid, bs, 0, s>>>(P, fin.list, fin.nheads, count, tol * tol, 6, axis_floor(eps), starts, cand, status, q,
                                     ctr);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = ktimer_end(s)) != cudaSuccess) return e;
  }
  MT_COUNT_LAUNCH(1);
  k_finish_followers<<<egrid, bs, 0, s>>>(count, fin.vals, fin.head, fin.link, starts, cand, status, ctr);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // the tip box: binary64 descents from the starts (list in fin.pos, free
  // once the heads are listed), then counted with the heads
  const unsigned sgrid = (unsigned)device_sm_count() * 4;
  MT_COUNT_LAUNCH(1);
  k_tip_list<<<sgrid, bs, 0, s>>>(fin.vals, &ctr->n_c32_fin, n2, fin.pos);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  PolyDev Pt = P;
  if (mixed_short(P)) Pt.fx = 0;
  if ((e = launch_descend_list(Pt, starts, fin.pos, n2, count, tol, cap, eps, cand, status, ctr, s)) != cudaSuccess)
    return e;
  MT_COUNT_LAUNCH(2);
  k_finish_append<<<sgrid, bs, 0, s>>>(fin.pos, n2, fin.list, fin.nheads, count, status, ctr);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_finish_count<<<1, 32, 0, s>>>(fin.nheads, n2, count);
  return cudaGetLastError();
}

}  // namespace mt
