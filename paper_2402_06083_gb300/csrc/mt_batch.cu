// mt_batch.cu -- many polynomials in one pass: every s_{l,n} with
// l >= 2, n >= 1, l + n <= max_order (eq. polySimple), as the paper's
// misSimpleQuick does one type at a time (Sec. 6.3.1).
//
// GB300 design.  The degrees of the polynomials differ by orders of
// magnitude (2 .. 2^14 for l + n <= 16), so one launch per polynomial would
// leave the GPU mostly idle.  Instead the work of all polynomials is laid
// end to end: seeds of all level lines in one launch, all level-line chunks
// drained by one persistent launch through an atomic chunk queue, all
// Newton descents drained by one persistent launch with per-lane refill
// (k_descend's scheme, each lane looking up the polynomial of the start it
// pops), then one sort by (polynomial, Re) and the segmented root-set,
// type and certificate kernels (SegView).
#include "mt_descent.cuh"
#include "mt_levelline.cuh"

namespace mt {

// largest p with off[p] <= x (off ascending, off[0] = 0)
__device__ __forceinline__ int find_seg(const int64_t* __restrict__ off, int np, int64_t x) {
  int lo = 0, hi = np - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= x) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__global__ void k_seed_lift_batch(const BatchEntry* __restrict__ E, const int64_t* __restrict__ seed_off,
                                  int np, int64_t total, double lambda0, int shrink, double2* seeds,
                                  DevCounters* ctr) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long steps = 0;
  if (g < total) {
    const int p = find_seg(seed_off, np, g);
    const BatchEntry e = E[p];
    seeds[g] = lift_seed(e.P, lambda0, e.N0, e.log2N0, shrink, g - seed_off[p], steps);
  }
  warp_add_u64(&ctr->walk_newton, steps);
  warp_add_u64(&ctr->seed_newton, steps);
}

// persistent: lanes pop level-line chunks of any polynomial from one queue
template <int FB>
__global__ void k_walk_batch(const BatchEntry* __restrict__ E, const int64_t* __restrict__ chunk_off,
                             int np, int64_t total, double lambda0, int M, int every,
                             const double2* __restrict__ seeds, double2* __restrict__ starts,
                             DevCounters* ctr) {
  __shared__ double2 ph[64];
  __shared__ longlong2 phx[64];
  walk_phases<FB>(lambda0, M, ph, phx);
  unsigned long long steps = 0, fails = 0;
  for (;;) {
    const int64_t c = (int64_t)atomicAdd(&ctr->queue_head2, 1ull);
    if (c >= total) break;
    const int p = find_seg(chunk_off, np, c);
    const BatchEntry e = E[p];
    const int64_t j = c - chunk_off[p];
    const double2* sd = seeds + e.seed_off;
    fails += walk_chunk_from<FB, true>(e.P, lambda0, M, every, e.L, e.nchunks, j, sd[j], sd[j + 1], ph, phx,
                                       starts + e.start_off, steps)
                 ? 1
                 : 0;
  }
  warp_add_u64(&ctr->walk_newton, steps);
  warp_add_u64(&ctr->walk_fail, fails);
}

// axis_add (mt_newton.cu) with the polynomial of each entry
static __device__ __noinline__ unsigned axis_add_batch(const BatchEntry* E, const uint16_t* seg, int64_t* buf,
                                                       unsigned n, bool mine, int64_t at, double2* cand,
                                                       unsigned flush) {
  axis_push(buf, n, mine, at);
  if (n >= flush) {
    int64_t i;
    if (axis_pop(buf, n, i)) {
      const PolyDev& P = E[seg[i]].P;
      cand[i] = axis_step(P.m, P.lcap, cand[i]);
    }
  }
  return n;
}

// persistent Newton descents over the starts of all polynomials (k_descend
// with the polynomial looked up per start)
__global__ void __launch_bounds__(128) k_descend_batch(const BatchEntry* __restrict__ E,
                                                       const int64_t* __restrict__ start_off,
                                                       int np, int64_t count, float tol2, unsigned axis_lo,
                                                       const double2* __restrict__ starts,
                                                       double2* __restrict__ cand,
                                                       uint8_t* __restrict__ status,
                                                       uint16_t* __restrict__ seg,
                                                       DevCounters* ctr) {
  const unsigned lane = threadIdx.x & 31;
  int64_t idx = -1;
  Descent d{0, 0, 16.f, 3.0e38f, 0, false, true};
  int m = 1, lcap = -1, cap = 20, outcome = -1;
  unsigned long long steps = 0, orbit = 0, nconv = 0, ndiv = 0, nto = 0;
  bool drained = false;
  __shared__ int64_t axis_buf[4][64];
  int64_t* abuf = axis_buf[threadIdx.x >> 5];
  unsigned na = 0;
  for (;;) {
    // as k_descend: written and refilled together once DESC_REFILL lanes wait
    const unsigned running = __ballot_sync(0xffffffffu, idx >= 0 && idx < count && outcome < 0);
    const unsigned wait = __popc(__ballot_sync(0xffffffffu, idx < 0 || outcome >= 0));
    if (wait >= DESC_REFILL || running == 0u) {
      bool near = false;
      const int64_t at = idx;
      if (outcome >= 0) {
        const double2 z = descent_point(d);
        cand[at] = z;
        near = outcome == 0 && d.fx && axis_near(z, axis_lo);
        status[at] = (uint8_t)outcome;
        nconv += outcome == 0;
        ndiv += outcome == 1;
        nto += outcome == 2;
        outcome = -1;
        idx = -1;
      }
      if (__any_sync(0xffffffffu, near)) na = axis_add_batch(E, seg, abuf, na, near, at, cand, 32u);
      const unsigned need = drained ? 0u : __ballot_sync(0xffffffffu, idx < 0);
      if (need) {
        unsigned long long base = 0;
        if (lane == (unsigned)(__ffs(need) - 1))
          base = atomicAdd(&ctr->queue_head, (unsigned long long)__popc(need));
        base = __shfl_sync(0xffffffffu, base, __ffs(need) - 1);
        drained = (int64_t)(base + __popc(need)) >= count;
        if (idx < 0) {
          idx = (int64_t)(base + __popc(need & lanemask_lt()));
          if (idx < count) {
            const int p = find_seg(start_off, np, idx);
            const BatchEntry e = E[p];
            m = e.P.m;
            lcap = e.P.lcap;
            cap = e.cap;
            seg[idx] = (uint16_t)p;
            descent_start(d, starts[idx], e.P.fx != 0);
          }
        }
      }
      if (drained && idx < 0) idx = count;
    }
    const bool active = idx >= 0 && idx < count && outcome < 0;
    if (!__any_sync(0xffffffffu, active)) {
      if (drained && !__any_sync(0xffffffffu, outcome >= 0)) break;
      continue;
    }
    if (active) {
      outcome = descent_step<true>(m, lcap, d, tol2, cap);
      ++steps;
      orbit += (unsigned)m;
    }
  }
  if (na) axis_add_batch(E, seg, abuf, na, false, 0, cand, 1u);
  warp_add_u64(&ctr->desc_newton, steps);
  warp_add_u64(&ctr->desc_orbit, orbit);
  warp_add_u64(&ctr->n_conv, nconv);
  warp_add_u64(&ctr->n_diverge, ndiv);
  warp_add_u64(&ctr->n_timeout, nto);
}

// (pair id, value) keys for the stable pass that groups candidates by polynomial
__global__ void k_seg_keys(const uint32_t* __restrict__ vals, const uint16_t* __restrict__ seg,
                           const uint8_t* __restrict__ status, int64_t count,
                           uint64_t* __restrict__ keys) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const uint32_t v = vals[i];
  // not-converged candidates sort after every polynomial's roots
  keys[i] = status[v] == 0 ? (uint64_t)seg[v] : 0xffffull;
}

cudaError_t launch_seed_lift_batch(const BatchEntry* E, const int64_t* seed_off, int np,
                                   int64_t total, double lambda0, int shrink, double2* seeds,
                                   DevCounters* ctr, cudaStream_t s) {
  if (total <= 0) return cudaSuccess;
  const int bs = 128;
  MT_COUNT_LAUNCH(1);
  k_seed_lift_batch<<<(unsigned)((total + bs - 1) / bs), bs, 0, s>>>(E, seed_off, np, total, lambda0,
                                                                     shrink, seeds, ctr);
  return cudaGetLastError();
}

cudaError_t launch_walk_batch(const BatchEntry* E, const int64_t* chunk_off, int np, int64_t total,
                              double lambda0, int M, int every, const double2* seeds,
                              double2* starts, DevCounters* ctr, cudaStream_t s) {
  if (total <= 0) return cudaSuccess;
  const int bs = 64;
  int per_sm = 0;
  const int fb = level_fb(lambda0);  // (walk_chunk_from reads each polynomial's fx)
  const auto kern = fb == 28 ? &k_walk_batch<28> : fb == 26 ? &k_walk_batch<26> : &k_walk_batch<0>;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, bs, 0);
  if (e != cudaSuccess) return e;
  int64_t grid = (int64_t)device_sm_count() * (per_sm > 0 ? per_sm : 1);
  const int64_t need = (total + bs - 1) / bs;
  if (grid > need) grid = need;
  MT_COUNT_LAUNCH(1);
  kern<<<(unsigned)grid, bs, 0, s>>>(E, chunk_off, np, total, lambda0, M, every, seeds, starts,
                                             ctr);
  return cudaGetLastError();
}

cudaError_t launch_descend_batch(const BatchEntry* E, const int64_t* start_off, int np,
                                 int64_t count, double tol, double eps, const double2* starts, double2* cand,
                                 uint8_t* status, uint16_t* seg, DevCounters* ctr, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  const int bs = 128;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_descend_batch, bs, 0);
  if (e != cudaSuccess) return e;
  int64_t grid = (int64_t)device_sm_count() * (per_sm > 0 ? per_sm : 1);
  const int64_t need = (count + bs - 1) / bs;
  if (grid > need) grid = need;
  MT_COUNT_LAUNCH(1);
  k_descend_batch<<<(unsigned)grid, bs, 0, s>>>(E, start_off, np, count, tol2_f(tol), axis_floor(eps), starts, cand,
                                                status, seg, ctr);
  return cudaGetLastError();
}

cudaError_t launch_seg_keys(const uint32_t* vals, const uint16_t* seg, const uint8_t* status,
                            int64_t count, uint64_t* keys, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  MT_COUNT_LAUNCH(1);
  k_seg_keys<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(vals, seg, status, count, keys);
  return cudaGetLastError();
}

}  // namespace mt
