// Recompression cores (sm_103a), one CTA per low-rank target:
//  * k_orth -- float factors: orthonormal basis of the sketch Y by pivoted
//              Gram-Schmidt in float-float, truncated at tau (FP64 factors take
//              the plan's Gram, k_pchol and basis stages);
//  * k_core -- core Gram (B^T)^T B^T, its eigen-decomposition by Jacobi, the rank
//              rule sigma_i > eps * sigma_1 (Sec. 4.3 H_eps), and the
//              recomposed factors U = Q W_k, V = B^T W_k.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "acr_device.h"
#include "acr_internal.h"

namespace acr {

namespace cg = cooperative_groups;

namespace {

constexpr int CMAX = 64;   // largest sketch / core dimension
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
  return v;
}

// Targets summed so far and those whose stacked rank exceeds the sketch
// width (sketch_stat[0], [1]); the terms are read by the lanes of one warp.
__device__ __forceinline__ void count_stacked_warp(const TInfo& ti,
                                                   const StackDim* __restrict__ stack,
                                                   float* const* __restrict__ tab,
                                                   const int* const* __restrict__ rtab, int P,
                                                   int p, unsigned long long* sketch_stat) {
  int stacked = 0;
  for (int e = ti.sk_beg + (threadIdx.x & 31); e < ti.sk_end; e += 32) {
    const StackDim sd = stack[e];
    if (sd.g0 >= 0 && !tab[sd.g0 * P + p]) continue;
    if (sd.g1 >= 0 && !tab[sd.g1 * P + p]) continue;
    stacked += dimv(sd.st, sd.rb, sd.ri, rtab, P, p);
  }
  stacked = __reduce_add_sync(FULL, stacked);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(sketch_stat, 1ull);
    if (stacked > ti.p) atomicAdd(sketch_stat + 1, 1ull);
  }
}

// Numbers held as an unevaluated sum hi + lo of two floats (~48 significant
// bits): the float forms' bases, core Grams and rotations run on the FP32 pipe
// instead of this part's narrow FP64 pipe.
struct FF {
  float h, l;
};
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);   // (never contracted into a sum)
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  const float s = p + e;
  return FF{s, e - (s - p)};
}
// a + b: TwoSum of the high parts, low parts added, renormalised
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  const float s = a.h + b.h;
  const float bp = s - a.h;
  float e = (a.h - (s - bp)) + (b.h - bp);
  e += a.l + b.l;
  const float r = s + e;
  return FF{r, e - (r - s)};
}
__device__ __forceinline__ FF ff_neg(FF a) { return FF{-a.h, -a.l}; }
// s += a * b; s is not renormalised
__device__ __forceinline__ void ff_dot(FF& s, FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);   // (never contracted into a sum)
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  const float t = s.h + p, bp = t - s.h;
  s.l += ((s.h - (t - bp)) + (p - bp)) + e;
  s.h = t;
}
// y + a * b
__device__ __forceinline__ FF ff_axpy(FF y, FF a, FF b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  e = fmaf(a.l, b.h, e);
  const float s = y.h + p, bp = s - y.h;
  const float l = ((y.h - (s - bp)) + (p - bp)) + (y.l + e);
  const float r = s + l;
  return FF{r, l - (r - s)};
}
// a / b to ~2^-45 (b normal)
__device__ __forceinline__ FF ff_div(FF a, FF b) {
  const float rb = 1.f / b.h, q = a.h * rb;
  const FF qb = ff_mul(FF{q, 0.f}, b);
  const float d = ff_add(a, ff_neg(qb)).h * rb;
  const float r = q + d;
  return FF{r, d - (r - q)};
}
// x^(-1/2): a Newton step y + y (1 - x y^2) / 2 from the float estimate
__device__ __forceinline__ FF ff_rsqrt(FF x) {
  const float y = rsqrtf(x.h);
  const FF xy2 = ff_mul(x, ff_mul(FF{y, 0.f}, FF{y, 0.f}));
  const FF e = ff_add(FF{1.f, 0.f}, ff_neg(xy2));
  return ff_add(FF{y, 0.f}, ff_mul(FF{y, 0.f}, FF{0.5f * e.h, 0.5f * e.l}));
}

// sums over 2 ... 2 * top lanes
__device__ __forceinline__ float sum_lanes(float a, int top) {
#pragma unroll
  for (int o = top; o > 0; o >>= 1) a += __shfl_xor_sync(FULL, a, o);
  return a;
}
__device__ __forceinline__ FF sum_lanes(FF a, int top) {
#pragma unroll
  for (int o = top; o > 0; o >>= 1)
    a = ff_add(a, FF{__shfl_xor_sync(FULL, a.h, o), __shfl_xor_sync(FULL, a.l, o)});
  return a;
}

// Orthonormal basis Q of range(Y) (m x p, in place) by pivoted modified
// Gram-Schmidt: the column of largest remaining norm is taken and removed from the
// remaining columns, whose norms are then computed afresh; stops when the largest
// remaining norm is at most tau times the largest of Y.
//
// Columns, dots, updates and the norm of the column taken are float-float (the rank
// decision at tau and the basis have to be as good as FP64-accurate Grams with an
// FP64 Cholesky make them; the other columns' norms only order them).  So one
// pass is enough: the basis loses orthogonality by ~2^-45 / tau, at most 3e-8 at
// the smallest tau (1e-6), below the rounding of Q to float, and a remaining norm at
// tau is known to as much of itself (from Grams, whose relative error of 1e-13 is that
// of squares, to 1e-13 / tau^2: 10% at 1e-6).
//
// Bound by the latency of the r dependent steps where few targets are left, else by
// the ~30 operations per remaining entry and step: Y stays in shared memory, 8 lanes
// own a column (CPG columns; the sums of a column take three exchanges), taken columns
// stay where they are, and a step has one barrier.  Sketches of which an SM holds only one
// or none (m = 512 to 2048 at n = 128) are shared by a cluster of OCL CTAs by rows,
// which push their parts of the sums into one another's shared memory: n = 128 setup 368
// ms for the bases (larger ones in global memory: 785; the cluster only beyond one SM's
// 220 KB: 370, and 94 in place of 89 at n = 80; from 54 KB on: 647 and 100).  Beyond the
// cluster's memory they stay in global memory.  n = 64 setup: 30 ms, n = 80: 89 ms
// (a warp per four columns: 41 and 127; plain float columns with a second projection
// per step: 24 and 75, rank decisions off by 1%, orthogonality up to 3e-7; six
// launches with FP64 pivoted Cholesky: 95 ms at n = 64).
constexpr int ONT = 256;

// row length of the staged columns: two neighbours' 8 rows meet no bank conflict
__host__ __device__ constexpr int orth_ld(int m) { return (m + 7) / 16 * 16 + 8; }

constexpr int OCL = 8;   // CTAs of a cluster: the 8 lanes of a column write to one each
enum OrthMode { ORTH_SM, ORTH_CLUSTER, ORTH_GLOBAL };

template <int MODE, int CPG>
__device__ __forceinline__ void orth(const TInfo& ti, int rank, FF tau2,
                                     float* const* __restrict__ tab, int* const* __restrict__ rtab,
                                     int P, int scr_buf, int scr_rbuf,
                                     const StackDim* __restrict__ stack,
                                     unsigned long long* __restrict__ sketch_stat,
                                     double* __restrict__ flops) {
  constexpr int NW = ONT / 32;
  constexpr bool SMEM = MODE != ORTH_GLOBAL, CL = MODE == ORTH_CLUSTER;
  extern __shared__ FF ysm[];
  __shared__ float nrm[2][CMAX];   // squared norms of the remaining columns, by parity of the step
  __shared__ FF bn[CMAX];          // of each basis column: its squared norm, then the reciprocal norm
  __shared__ int piv[CMAX];        // and its place
  __shared__ float mx[NW];
  // the cluster's parts of the sums, written by its CTAs: products with the columns and of
  // the column taken (last); norms; largest entries
  __shared__ FF pdot[CL ? OCL : 1][CL ? CMAX + 1 : 1];
  __shared__ float pnrm[CL ? OCL : 1][CL ? CMAX : 1], pmax[OCL];
  cg::cluster_group cl = cg::this_cluster();
  const int p = blockIdx.y;
  float* scr = tab[scr_buf * P + p];
  int* rs = rtab[scr_rbuf * P + p];
  if (!scr || !rs) return;   // (the whole cluster)
  if constexpr (CL) cl.sync();   // every CTA has started
  // this CTA's rows
  const int mr = CL ? (ti.m + OCL - 1) / OCL : ti.m, r0 = CL ? rank * mr : 0;
  const int m = CL ? max(0, min(mr, ti.m - r0)) : ti.m, pc = ti.p;
  const int64_t gld = ti.m;
  const int ld = SMEM ? orth_ld(mr) : ti.m;
  float* Yg = scr + ti.y_off + r0;
  float* Yl = scr + ti.bt_off;   // low parts beyond shared memory: B^T comes later
  auto get = [&](int i, int c) {
    if constexpr (SMEM) return ysm[i + c * ld];
    else return FF{Yg[i + gld * c], Yl[i + gld * c]};
  };
  auto put = [&](int i, int c, FF v) {
    if constexpr (SMEM) {
      ysm[i + c * ld] = v;
    } else {
      Yg[i + gld * c] = v.h;
      Yl[i + gld * c] = v.l;
    }
  };
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = tid >> 3, l8 = tid & 7;   // this thread's columns c0 + 32 u, rows l8 + 8 k
  // a column's norm (the sum over this CTA's rows, in all 8 lanes) to the next step, in a
  // cluster through every CTA's parts
  auto give_norm = [&](float t, int c, float* next) {
    if (c >= pc) return;
    if constexpr (CL) *cl.map_shared_rank(&pnrm[rank][c], l8) = t;
    else if (l8 == 0) next[c] = t;
  };
  auto take_norms = [&](float* next) {
    if constexpr (CL) {
      cl.sync();
      if (tid < pc) {
        float t = 0.f;
#pragma unroll
        for (int k = 0; k < OCL; ++k) t += pnrm[k][tid];
        next[tid] = t;
      }
    }
  };
  // The largest entry, and the power of two that brings it to [1, 2): sketches whose
  // squares would leave the float range keep all bits (Q does not depend on it).
  float amax = 0.f;
#pragma unroll
  for (int u = 0; u < CPG; ++u) {
    const int c = c0 + 32 * u;
    if (c < pc)
#pragma unroll 4
      for (int i = l8; i < m; i += 8) {
        const float v = Yg[i + gld * c];
        if (SMEM) ysm[i + c * ld].h = v;
        amax = fmaxf(amax, fabsf(v));
      }
  }
  amax = __uint_as_float(__reduce_max_sync(FULL, __float_as_uint(amax)));
  if (lane == 0) mx[warp] = amax;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < NW; ++w) amax = fmaxf(amax, mx[w]);
  if constexpr (CL) {
    if (tid < OCL) *cl.map_shared_rank(&pmax[rank], tid) = amax;
    cl.sync();
#pragma unroll
    for (int k = 0; k < OCL; ++k) amax = fmaxf(amax, pmax[k]);
  }
  const int ex = amax > 0.f && amax <= 3.4e38f ? max(ilogbf(amax), -126) : 0;
  const float up = ldexpf(1.f, -ex / 2), up2 = ldexpf(1.f, -ex - -ex / 2);   // (2^-ex may not fit)
#pragma unroll
  for (int u = 0; u < CPG; ++u) {
    const int c = c0 + 32 * u;
    float t = 0.f;
    if (c < pc)
      for (int i = l8; i < m; i += 8) {
        const float v = (SMEM ? ysm[i + c * ld].h : Yg[i + gld * c]) * up * up2;
        put(i, c, FF{v, 0.f});
        t = fmaf(v, v, t);
      }
    give_norm(sum_lanes(t, 4), c, nrm[0]);
  }
  take_norms(nrm[0]);
  if (sketch_stat && rank == 0 && warp == NW - 1)
    count_stacked_warp(ti, stack, tab, (const int* const*)rtab, P, p, sketch_stat);
  __syncthreads();
  unsigned long long taken = 0ull;
  FF tol{0.f, 0.f};
  int r = 0;
  for (int j = 0; j < pc; ++j) {
    // every warp finds the largest remaining column: bits of the squared norms
    // order like the norms, the low six hold the column (norms that agree to
    // 2^-17 count as equal: the lowest column); NaN norms are passed over
    const float* now = nrm[j & 1];
    unsigned key = 0u;
#pragma unroll
    for (int u = 0; u < CPG; ++u) {
      const int c = lane + 32 * u;
      if (c < pc && now[c] > 0.f) key = max(key, (__float_as_uint(now[c]) & ~63u) | (63u - c));
    }
    key = __reduce_max_sync(FULL, key);
    if (key == 0u) break;
    const int q = 63 - (int)(key & 63u);
    if (now[q] < 0.99f * tol.h) break;
    // its products with the remaining columns and itself
    const unsigned long long gone = taken | 1ull << q;
    FF s[CPG], best{0.f, 0.f};
    bool on[CPG];
#pragma unroll
    for (int u = 0; u < CPG; ++u) {
      s[u] = FF{0.f, 0.f};
      on[u] = c0 + 32 * u < pc && !((gone >> (c0 + 32 * u)) & 1);
    }
    for (int i = lane; i < m; i += 32) ff_dot(best, get(i, q), get(i, q));
#pragma unroll
    for (int u = 0; u < CPG; ++u)
      if (on[u])
#pragma unroll 4
        for (int i = l8; i < m; i += 8) ff_dot(s[u], get(i, c0 + 32 * u), get(i, q));
    best = sum_lanes(best, 16);
#pragma unroll
    for (int u = 0; u < CPG; ++u) s[u] = sum_lanes(s[u], 4);
    if constexpr (CL) {   // the sums over the cluster, by every CTA in the same order
#pragma unroll
      for (int u = 0; u < CPG; ++u)
        if (on[u]) *cl.map_shared_rank(&pdot[rank][c0 + 32 * u], l8) = s[u];
      if (tid < OCL) *cl.map_shared_rank(&pdot[rank][CMAX], tid) = best;
      cl.sync();
      best = FF{0.f, 0.f};
#pragma unroll
      for (int k = 0; k < OCL; ++k) best = ff_add(best, pdot[k][CMAX]);
#pragma unroll
      for (int u = 0; u < CPG; ++u)
        if (on[u]) {
          s[u] = FF{0.f, 0.f};
#pragma unroll
          for (int k = 0; k < OCL; ++k) s[u] = ff_add(s[u], pdot[k][c0 + 32 * u]);
        }
    }
    if (j == 0) tol = ff_mul(tau2, best);
    if (!(best.h > tol.h || (best.h == tol.h && best.l > tol.l))) break;
    taken = gone;
    r = j + 1;
    if (tid == 0) {
      bn[j] = best;
      piv[j] = q;
    }
    // removed from them; their norms (0: taken)
#pragma unroll
    for (int u = 0; u < CPG; ++u) {
      const int c = c0 + 32 * u;
      const FF g = ff_neg(ff_div(s[u], best));
      float t = 0.f;
      if (on[u])
#pragma unroll 4
        for (int i = l8; i < m; i += 8) {
          const FF w = ff_axpy(get(i, c), g, get(i, q));
          put(i, c, w);
          t = fmaf(w.h, w.h, t);
        }
      give_norm(sum_lanes(t, 4), c, nrm[(j + 1) & 1]);
    }
    take_norms(nrm[(j + 1) & 1]);
    __syncthreads();
  }
  if (tid < r) bn[tid] = ff_rsqrt(bn[tid]);
  __syncthreads();
  auto unit = [&](int i, int j) {
    const FF v = get(i, piv[j]), f = bn[j];
    return fmaf(v.h, f.h, fmaf(v.h, f.l, v.l * f.h));
  };
  if (SMEM) {
    for (int j = warp; j < r; j += NW)
      for (int i = lane; i < m; i += 32) Yg[i + gld * j] = unit(i, j);
  } else {   // a thread owns its rows: all of one read before any is written
    for (int i = tid; i < m; i += ONT) {
      float row[CMAX];
      for (int j = 0; j < r; ++j) row[j] = unit(i, j);
      for (int j = 0; j < r; ++j) Yg[i + gld * j] = row[j];
    }
  }
  if (tid == 0 && rank == 0) {
    rs[ti.r_ri] = r;
    if (flops) atomicAdd(flops, 2.0 * ti.m * r * (2.0 * pc - r));
  }
}

template <int MODE, int CPG>
__global__ void __launch_bounds__(ONT, CPG == 1 ? 5 : 3)
    k_orth(const TInfo* __restrict__ tis, const int* __restrict__ order, FF tau2,
           float* const* __restrict__ tab, int* const* __restrict__ rtab, int P, int scr_buf,
           int scr_rbuf, const StackDim* __restrict__ stack,
           unsigned long long* __restrict__ sketch_stat, double* __restrict__ flops) {
  orth<MODE, CPG>(tis[order[blockIdx.x]], 0, tau2, tab, rtab, P, scr_buf, scr_rbuf, stack,
                  sketch_stat, flops);
}
template <int CPG>
__global__ void __cluster_dims__(OCL, 1, 1) __launch_bounds__(ONT, CPG == 1 ? 5 : 3)
    k_orth_cluster(const TInfo* __restrict__ tis, const int* __restrict__ order, FF tau2,
                   float* const* __restrict__ tab, int* const* __restrict__ rtab, int P,
                   int scr_buf, int scr_rbuf, const StackDim* __restrict__ stack,
                   unsigned long long* __restrict__ sketch_stat, double* __restrict__ flops) {
  orth<ORTH_CLUSTER, CPG>(tis[order[blockIdx.x / OCL]], blockIdx.x % OCL, tau2, tab, rtab, P,
                          scr_buf, scr_rbuf, stack, sketch_stat, flops);
}

// ------------------------------------------------------------ Jacobi cores
// The three element types of a core: float (first sweeps), FF and double.
__device__ __forceinline__ float em(float a, float b) { return a * b; }
__device__ __forceinline__ double em(double a, double b) { return a * b; }
__device__ __forceinline__ FF em(FF a, FF b) { return ff_mul(a, b); }
__device__ __forceinline__ float ea(float a, float b) { return a + b; }
__device__ __forceinline__ double ea(double a, double b) { return a + b; }
__device__ __forceinline__ FF ea(FF a, FF b) { return ff_add(a, b); }
__device__ __forceinline__ float en(float a) { return -a; }
__device__ __forceinline__ double en(double a) { return -a; }
__device__ __forceinline__ FF en(FF a) { return ff_neg(a); }
__device__ __forceinline__ float ef(float a) { return a; }              // to float
__device__ __forceinline__ float ef(double a) { return (float)a; }
__device__ __forceinline__ float ef(FF a) { return a.h; }
__device__ __forceinline__ double ed(double a) { return a; }            // to double
__device__ __forceinline__ double ed(FF a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ void es(float& a, float x) { a = x; }        // from float
__device__ __forceinline__ void es(double& a, float x) { a = x; }
__device__ __forceinline__ void es(FF& a, float x) { a = FF{x, 0.f}; }
__device__ __forceinline__ float eshfl(float a, int k) { return __shfl_sync(FULL, a, k); }
__device__ __forceinline__ double eshfl(double a, int k) { return __shfl_sync(FULL, a, k); }
__device__ __forceinline__ FF eshfl(FF a, int k) {
  return FF{__shfl_sync(FULL, a.h, k), __shfl_sync(FULL, a.l, k)};
}
__device__ __forceinline__ double escale(double a, int e) { return ldexp(a, e); }
__device__ __forceinline__ FF escale(FF a, int e) { return FF{ldexpf(a.h, e), ldexpf(a.l, e)}; }

// The root t of least magnitude of q t^2 + d t - q: 1 / (tau + sign(tau) sqrt(1 +
// tau^2)), tau = d / (2 q) (an infinite tau gives 0)
__device__ __forceinline__ float jangle(float d, float q) {
  const float tau = d / (2.f * q);
  return copysignf(1.f / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f))), tau);
}
// The rotation (c, s) that zeroes a_pq of [a_pp a_pq; a_pq a_qq]; an angle that is off leaves
// as much of the entry, which later rotations remove.
// Float (first sweeps): the fast divide, an angle to ~1e-6.
__device__ __forceinline__ void jrot(float app, float aqq, float apq, float& c, float& s) {
  c = 1.f;
  s = 0.f;
  if (apq != 0.f) {
    const float tau = __fdividef(aqq - app, 2.f * apq), at = fabsf(tau), h = fmaf(tau, tau, 1.f);
    // (beyond 1e9 the square root is tau itself; an infinite tau gives the angle 0)
    const float t = copysignf(__fdividef(1.f, at + (at > 1e9f ? at : h * rsqrtf(h))), tau);
    c = rsqrtf(fmaf(t, t, 1.f));
    s = t * c;
  }
}
// Float-float: the angle to float accuracy, its cosine and sine to the pair's, so that the
// rotation is orthogonal to ~1e-14.
__device__ __forceinline__ void jrot(FF app, FF aqq, FF apq, FF& c, FF& s) {
  c = FF{1.f, 0.f};
  s = FF{0.f, 0.f};
  if (apq.h != 0.f) {
    const float t = jangle(ff_add(aqq, ff_neg(app)).h, apq.h), p = __fmul_rn(t, t);
    c = ff_rsqrt(ff_add(FF{1.f, 0.f}, FF{p, fmaf(t, t, -p)}));
    s = ff_mul(FF{t, 0.f}, c);
  }
}
// FP64: the angle by two Newton steps from the float one, whose residuals are FP64 (the
// divisions of the corrections need not be); the cosine likewise.
__device__ __forceinline__ void jrot(double app, double aqq, double apq, double& c, double& s) {
  c = 1.0;
  s = 0.0;
  const double d = aqq - app;
  const float q = (float)apq, df = (float)d;
  if (q != 0.f) {   // (an entry below the float range turns nothing: the largest is near 1)
    const float t0 = jangle(df, q), slope = fmaf(2.f * q, t0, df);
    double t = t0;
#pragma unroll
    for (int k = 0; k < 2; ++k) t -= (double)((float)fma(fma(apq, t, d), t, -apq) / slope);
    const double x = fma(t, t, 1.0);
    double y = (double)rsqrtf((float)x);
    y = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    c = fma(0.5 * y, fma(-x * y, y, 1.0), y);
    s = t * c;
  }
}

constexpr int CNT = 128;

// Cyclic Jacobi of the symmetric r x r matrix A in round-robin order, rotations
// accumulated into V, until the off-diagonal mass is at most conv of the total.
// Every warp computes all rotations of a round in its lanes and hands them
// round by shuffles; a thread rotates 2 x 2 blocks (rows of pair k1, columns of
// pair k2, k1 <= k2, the mirror entry written alongside) into the other copy A2 and
// row pairs of V in place: one barrier per round.  A and A2 trade places with
// every round.  Returns the sweeps done.
template <typename EL>
__device__ int jacobi(EL*& A, EL*& A2, EL* V, int r, int lda, float conv, int most,
                      float (*red)[CNT / 32]) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int nn = (r + 1) & ~1;   // even number of players (an odd r gets a dummy)
  const int np = nn / 2, nblk = np * (np + 1) / 2;
  // work items of a round: the blocks of A, then from a whole warp on the (pair,
  // row) items of V; a thread's items stay its own, the first few's indices
  // in registers (x | y << 8: k1, k2 or pair, row; -1: none)
  const int vbase = (nblk + 31) & ~31, nitem = vbase + np * r;
  constexpr int KEEP = 3;
  auto item = [&](int e) {
    if (e < vbase) {
      if (e >= nblk) return -1;
      int k1 = 0, k2 = e;
      while (k2 >= np - k1) { k2 -= np - k1; ++k1; }
      return k1 | (k1 + k2) << 8;
    }
    if (e >= nitem) return -1;
    const int k = (e - vbase) / r;
    return k | (e - vbase - k * r) << 8;
  };
  int kept[KEEP];
#pragma unroll
  for (int u = 0; u < KEEP; ++u) kept[u] = item(tid + CNT * u);
  // circle method: player 0 fixed, the others rotate
  auto pair_of = [&](int k, int round, int& lo, int& hi) {
    int a = k == 0 ? 0 : k + round, b = nn - 1 - k + round;
    if (a >= nn) a -= nn - 1;
    if (b >= nn) b -= nn - 1;
    lo = min(a, b);
    hi = max(a, b);
  };
  int sweeps = 0;
  for (int sweep = 0; sweep < most && r > 1; ++sweep) {
    // off-diagonal and total mass
    float off = 0.f, tot = 0.f;
    for (int i = tid >> 5; i < r; i += CNT / 32)
      for (int j = lane; j < r; j += 32) {
        const float v = ef(A[i * lda + j]);
        if (i != j) off = fmaf(v, v, off);
        else tot = fmaf(v, v, tot);
      }
    off = warp_sum(off);
    tot = warp_sum(tot);
    if (lane == 0) { red[0][tid >> 5] = off; red[1][tid >> 5] = tot; }
    __syncthreads();
    off = (red[0][0] + red[0][1]) + (red[0][2] + red[0][3]);
    tot = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
    if (off <= conv * (tot + off)) break;
    ++sweeps;
    for (int round = 0; round < nn - 1; ++round) {
      // lane k: the rotation of pair k
      EL rc, rsn;
      es(rc, 1.f);
      es(rsn, 0.f);
      if (lane < np) {
        int lo, hi;
        pair_of(lane, round, lo, hi);
        if (hi < r) jrot(A[lo * lda + lo], A[hi * lda + hi], A[lo * lda + hi], rc, rsn);
      }
      for (int u = 0, e0 = tid & ~31; e0 < nitem; ++u, e0 += CNT) {
        int id = 0;
        if (u < KEEP) {
#pragma unroll
          for (int x = 0; x < KEEP; ++x)
            if (u == x) id = kept[x];
        } else {
          id = item(e0 + lane);
        }
        const bool on = id >= 0;
        if (e0 < vbase) {   // a block: columns first, then rows
          const int k1 = on ? id & 255 : 0, k2 = on ? id >> 8 : 0;
          const EL c1 = eshfl(rc, k1), s1 = eshfl(rsn, k1), c2 = eshfl(rc, k2), s2 = eshfl(rsn, k2);
          if (on) {
            int a1, b1, a2, b2;
            pair_of(k1, round, a1, b1);
            pair_of(k2, round, a2, b2);
            const bool h1 = b1 < r, h2 = b2 < r;
            EL z;
            es(z, 0.f);
            const EL x00 = A[a1 * lda + a2];
            const EL x01 = h2 ? A[a1 * lda + b2] : z;
            const EL x10 = h1 ? A[b1 * lda + a2] : z;
            const EL x11 = (h1 && h2) ? A[b1 * lda + b2] : z;
            const EL y00 = ea(em(c2, x00), en(em(s2, x01))), y01 = ea(em(s2, x00), em(c2, x01));
            const EL y10 = ea(em(c2, x10), en(em(s2, x11))), y11 = ea(em(s2, x10), em(c2, x11));
            const EL z00 = ea(em(c1, y00), en(em(s1, y10))), z01 = ea(em(c1, y01), en(em(s1, y11)));
            const EL z10 = ea(em(s1, y00), em(c1, y10)), z11 = ea(em(s1, y01), em(c1, y11));
            const bool same = k1 == k2;   // a diagonal block stays symmetric
            A2[a1 * lda + a2] = z00;
            if (!same) A2[a2 * lda + a1] = z00;
            if (h2) { A2[a1 * lda + b2] = z01; A2[b2 * lda + a1] = z01; }
            if (h1 && !same) { A2[b1 * lda + a2] = z10; A2[a2 * lda + b1] = z10; }
            if (h1 && h2) {
              A2[b1 * lda + b2] = z11;
              if (!same) A2[b2 * lda + b1] = z11;
            }
          }
        } else {   // V <- V J
          const int k = on ? id & 255 : 0, iv = on ? id >> 8 : 0;
          const EL c = eshfl(rc, k), s = eshfl(rsn, k);
          int a, b;
          pair_of(k, round, a, b);
          if (on && b < r) {
            const EL vx = V[iv * lda + a], vy = V[iv * lda + b];
            V[iv * lda + a] = ea(em(c, vx), en(em(s, vy)));
            V[iv * lda + b] = ea(em(s, vx), em(c, vy));
          }
        }
      }
      __syncthreads();
      EL* t = A;
      A = A2;
      A2 = t;
    }
  }
  return sweeps;
}

// The core of a target (r x r, r the basis size): H = (B^T)^T B^T with
// FP64-accurate sums (float factors: exact products, compensated float-float sums; the
// rank rule resolves singular values only down to the square root of the
// Gram's relative error), scaled by a power of two to a largest diagonal in
// [1/2, 1) (exact: eigenvectors and ratios sigma_i / sigma_1 are unchanged; the
// rotations then stay clear of the ends of the float range, which the Gram's own
// products still have to fit); its eigenvectors; the kept ones W, largest eigenvalue
// first, and the factors U = Q W, V = B^T W straight into the target's leaf.
//
// The eigenvectors: Jacobi sweeps in plain float to an off-diagonal 1e-5 of
// the norm; the float rotations' product made orthonormal (Newton-Schulz, V =
// W + W (I - W^T W) / 2: exact W^T W, the correction small enough for float; twice
// for FP64); H transformed by it in the core's full arithmetic; then sweeps in
// that arithmetic -- float-float to an off-diagonal mass of 1e-16, or of eps^4 / 100 where
// that is less (the rank rule compares eigenvalues down to eps^2), FP64 to 1e-30 --
// which find a nearly diagonal matrix and need one (FP64: two) instead of six
// to eight, at a twelfth of the operations per float sweep (FP64: a 64th).  The
// result is no less accurate than with full arithmetic throughout: FP64, 56 columns, all
// kept: U orthonormal to 6.9e-15 and U V^T to 7.3e-15 of the product (FP64
// sweeps only: 2.7e-14 and 2.5e-14).
//
// Bound by the latency of the ~6 (r - 1) dependent rounds of a core.  Four warps, so that a
// typical core's round (r = 12: 21 blocks and 72 row pairs of V) is one pass over
// the threads.  n = 64 setup: 31 ms (four stages of their own: 90 ms; float-float
// sweeps throughout: 31 ms); n = 32 FP64: 11 ms (Gram, two Jacobi kernels and
// recomposition as launches of their own: 33 ms).
constexpr int CRAW = CNT * 16;   // partial sums of the Gram's tiles
static_assert(sizeof(FF) == sizeof(double), "both element types share the layout");

__host__ __device__ constexpr size_t core_smem(int p) {
  // A; the Gram's staging, then the other A (later W) and V in its place (8-byte
  // entries, rows of up to p + 3); the float rotations' product
  const size_t a = (size_t)p * (p + 4) * 8, g = CRAW * 8;
  return a + (2 * a > g ? 2 * a : g) + (size_t)p * (p + 4) * 4;
}

template <typename T>
__global__ void __launch_bounds__(CNT) k_core(const TInfo* __restrict__ tis, int tbase, double eps,
                                              int kc, int c_role, int maxp,
                                              T* const* __restrict__ tab,
                                              int* const* __restrict__ rtab, int P, int scr_buf,
                                              int scr_rbuf, int* err, double* __restrict__ flops) {
  constexpr bool F64 = sizeof(T) == 8;
  using E = typename std::conditional<F64, double, FF>::type;
  const int p = blockIdx.y;
  const TInfo ti = tis[tbase + blockIdx.x];
  T* scr = tab[scr_buf * P + p];
  int* rs = rtab[scr_rbuf * P + p];
  int* crank = rtab[c_role * P + p];
  if (!scr || !rs || !crank) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int r = rs[ti.r_ri];
  if (r <= 0) {   // an empty basis: rank 0
    if (tid == 0) crank[ti.c_leaf] = 0;
    return;
  }
  extern __shared__ __align__(16) unsigned char csm[];
  const int lda = r | 1;   // odd row length: no bank conflicts down a column
  E* A = reinterpret_cast<E*>(csm);
  const size_t area = (size_t)maxp * (maxp + 4);
  E* A2 = A + area;
  E* V = A2 + area;
  E* raw = A2;   // the Gram is done before the second A and V begin
  float* W = reinterpret_cast<float*>(A2 + max(2 * area, (size_t)CRAW));
  __shared__ float red[2][CNT / 32];
  __shared__ double lam[CMAX];
  __shared__ int ord[CMAX];
  __shared__ int kkeep;

  // ---- Gram of B^T (n x r): thread (tile, slice) owns a 4 x 4 tile of the
  // upper triangle and every S-th row
  const T* B = scr + ti.bt_off;
  const int n = ti.n;
  {
    const int TM = (r + 3) >> 2, ntile = TM * (TM + 1) / 2, mt = 4 * TM;
    // (the CRAW entries staged as values of T; at least 31 rows)
    const int kch = min(256, ((CRAW * 8 / (int)sizeof(T) / mt) - 1) & ~1), ysld = kch + 1;
    T* ys = reinterpret_cast<T*>(raw);
    for (int tb = 0; tb < ntile; tb += CNT) {   // (one pass up to r = 60)
      const int nt = min(CNT, ntile - tb);
      const int S = CNT / nt;
      const int tl = tid / S, slice = tid - tl * S;
      const bool active = tl < nt;
      int a0 = 0, t = tb + (active ? tl : 0);
      while (t >= TM - a0) { t -= TM - a0; ++a0; }
      const int i0 = 4 * a0, j0 = 4 * (a0 + t);
      T s[4][4];
      float c[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) { s[x][y] = T(0); c[x][y] = 0.f; }
      for (int l0 = 0; l0 < n; l0 += kch) {
        const int kk = min(kch, n - l0);
        __syncthreads();
        for (int col = tid >> 5; col < mt; col += CNT / 32)
          for (int l = lane; l < kk; l += 32)
            ys[col * ysld + l] = col < r ? B[(l0 + l) + (int64_t)col * n] : T(0);
        __syncthreads();
        if (active)
          for (int l = slice; l < kk; l += S) {
            T av[4], bv[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              av[x] = ys[(i0 + x) * ysld + l];
              bv[x] = ys[(j0 + x) * ysld + l];
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
              for (int y = 0; y < 4; ++y) {
                if constexpr (F64) s[x][y] = fma(av[x], bv[y], s[x][y]);
                else ff_fma(s[x][y], c[x][y], av[x], bv[y]);
              }
          }
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        E v;
        es(v, 0.f);
        if (active) {
          if constexpr (F64) v = s[e & 3][e >> 2];
          else v = FF{s[e & 3][e >> 2], c[e & 3][e >> 2]};
        }
        raw[e * CNT + tid] = v;
      }
      __syncthreads();
      // the slices' partial sums, in a fixed order
      for (int e = tid; e < nt * 16; e += CNT) {
        const int tq = e >> 4, q = e & 15;
        E h;
        es(h, 0.f);
        for (int sl = 0; sl < S; ++sl) {
          const E x = raw[q * CNT + tq * S + sl];
          if constexpr (F64) {
            h += x;
          } else {
            const float u = h.h + x.h, bp = u - h.h;
            h.l += ((h.h - (u - bp)) + (x.h - bp)) + x.l;
            h.h = u;
          }
        }
        if constexpr (!F64) {
          const float u = h.h + h.l;
          h.l = h.l - (u - h.h);
          h.h = u;
        }
        int tt = tb + tq, a = 0;
        while (tt >= TM - a) { tt -= TM - a; ++a; }
        const int i = 4 * a + (q & 3), j = 4 * (a + tt) + (q >> 2);
        if (i < r && j < r) {
          A[i * lda + j] = h;
          A[j * lda + i] = h;
        }
      }
    }
  }
  __syncthreads();
  // ---- power-of-two scale: the largest diagonal to [1/2, 1)
  int ex = 0;
  {
    double dmax = 0.0;
    for (int i = lane; i < r; i += 32) dmax = fmax(dmax, ed(A[i * lda + i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = fmax(dmax, __shfl_xor_sync(FULL, dmax, o));
    if (dmax > 0.0 && dmax <= 1.0e300) frexp(dmax, &ex);
  }
  __syncthreads();
  float* F0 = reinterpret_cast<float*>(A2);   // float copies for the first sweeps
  float* F1 = F0 + area;
  for (int e = tid; e < r * lda; e += CNT) {
    const int i = e / lda, j = e - i * lda;
    if (j >= r) continue;
    const E v = escale(A[e], -ex);
    A[e] = v;
    F0[e] = ef(v);
    W[e] = i == j ? 1.f : 0.f;
  }
  __syncthreads();

  // ---- eigenvectors
  int sweeps = 0;
  if (r > 1) {
    sweeps = jacobi<float>(F0, F1, W, r, lda, 1e-10f, 10, red);
    __syncthreads();
    // the product of the float rotations, made orthonormal
    float* D = reinterpret_cast<float*>(A2);   // (I - W^T W) / 2
    for (int e = tid; e < r * r; e += CNT) {
      const int i = e / r, j = e - i * r;
      if (F64) {
        double g = 0.0;
        for (int l = 0; l < r; ++l) g = fma((double)W[l * lda + i], (double)W[l * lda + j], g);
        D[i * lda + j] = (float)(0.5 * ((i == j ? 1.0 : 0.0) - g));
      } else {
        float s = i == j ? -1.f : 0.f, c = 0.f;
        for (int l = 0; l < r; ++l) ff_fma(s, c, W[l * lda + i], W[l * lda + j]);
        D[i * lda + j] = -0.5f * (s + c);
      }
    }
    __syncthreads();
    for (int e = tid; e < r * r; e += CNT) {
      const int i = e / r, j = e - i * r;
      float d = 0.f;
      for (int l = 0; l < r; ++l) d = fmaf(W[i * lda + l], D[l * lda + j], d);
      E v, dd;
      es(v, W[i * lda + j]);
      es(dd, d);
      V[i * lda + j] = ea(v, dd);
    }
    __syncthreads();
    if constexpr (F64) {
      for (int e = tid; e < r * r; e += CNT) {
        const int i = e / r, j = e - i * r;
        double g = 0.0;
        for (int l = 0; l < r; ++l) g = fma(V[l * lda + i], V[l * lda + j], g);
        D[i * lda + j] = (float)(0.5 * ((i == j ? 1.0 : 0.0) - g));
      }
      __syncthreads();
      for (int e = tid; e < r * r; e += CNT) {   // (W in place of V: the correction is ~1e-12)
        const int i = e / r, j = e - i * r;
        float d = 0.f;
        for (int l = 0; l < r; ++l) d = fmaf(W[i * lda + l], D[l * lda + j], d);
        V[i * lda + j] += (double)d;
      }
      __syncthreads();
    }
    // A <- V^T (A V)
    for (int e = tid; e < r * r; e += CNT) {
      const int i = e / r, j = e - i * r;
      E t;
      es(t, 0.f);
      for (int l = 0; l < r; ++l) t = ea(t, em(A[i * lda + l], V[l * lda + j]));
      A2[i * lda + j] = t;
    }
    __syncthreads();
    for (int e = tid; e < r * r; e += CNT) {
      const int i = e / r, j = e - i * r;
      if (j < i) continue;
      E t;
      es(t, 0.f);
      for (int l = 0; l < r; ++l) t = ea(t, em(V[l * lda + i], A2[l * lda + j]));
      A[i * lda + j] = t;
      A[j * lda + i] = t;
    }
    __syncthreads();
    const float e2 = (float)(eps * eps);   // (pairs reach ~1e-27)
    const float conv = F64 ? 1e-30f : fminf(1e-16f, fmaxf(1e-24f, 0.01f * e2 * e2));
    sweeps += jacobi<E>(A, A2, V, r, lda, conv, 40, red);
  } else if (tid == 0) {
    es(V[0], 1.f);
  }
  // ---- eigenvalues descending (rank by counting; ties by index), the kept rank
  for (int i = tid; i < r; i += CNT) {
    lam[i] = ed(A[i * lda + i]);
    ord[i] = i;   // (NaN eigenvalues take no place of their own below)
  }
  __syncthreads();
  for (int i = tid; i < r; i += CNT) {
    int pos = 0;
    for (int j = 0; j < r; ++j)
      if (lam[j] > lam[i] || (lam[j] == lam[i] && j < i)) ++pos;
    ord[pos] = i;
  }
  __syncthreads();
  if (tid == 0) {
    const double l1 = lam[ord[0]];
    const double cut = eps * eps * l1;   // sigma_i > eps sigma_1
    int k = 0;
    if (l1 > 0.0)
      for (int j = 0; j < r; ++j) {
        const double lj = lam[ord[j]];
        if (lj > 0.0 && lj > cut) ++k;
        else break;
      }
    if (k > kc) {
      atomicOr(err, ERR_RANKCAP);
      k = kc;
    }
    kkeep = k;
    crank[ti.c_leaf] = k;
    if (flops) atomicAdd(flops, 9.0 * r * r * r * sweeps);
  }
  __syncthreads();
  const int k = kkeep;
  // ---- recomposition: the kept columns W (r x k, rows of whole 4-vectors) in the
  // second A's place
  const int ldw = (k + 3) & ~3;
  T* K = reinterpret_cast<T*>(A2);
  for (int e = tid; e < r * ldw; e += CNT) {
    const int i = e / ldw, j = e - i * ldw;
    T w = T(0);
    if (j < k) {
      const E v = V[i * lda + ord[j]];
      if constexpr (F64) w = v;
      else w = v.h + v.l;
    }
    K[e] = w;
  }
  __syncthreads();
  T* Uo = tab[(3 * c_role + 1) * P + p];
  T* Vo = tab[(3 * c_role + 2) * P + p];
  const int m = ti.m;
  for (int e = tid; e < m + n; e += CNT) {   // a row of U = Q W, then of V = B^T W
    const bool u = e < m;
    const int rows = u ? m : n, i = u ? e : e - m;
    const T* X = (u ? scr + ti.y_off : B) + i;
    T* Z = u ? Uo : Vo;
    if (!Z) continue;
    Z += (u ? ti.u_off : ti.v_off) + i;
    for (int j0 = 0; j0 < k; j0 += 4) {
      T acc[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll 8
      for (int l = 0; l < r; ++l) {
        const T x = X[(int64_t)l * rows];
        const T* w = K + l * ldw + j0;
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] += x * w[q];
      }
      T* z = Z + (int64_t)j0 * rows;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (j0 + q < k) z[q * (int64_t)rows] = acc[q];
    }
  }
}

}  // namespace

void launch_orth(const Plan& pl, double tau, float* const* d_tab, int* const* d_rtab, int P,
                 cudaStream_t st, unsigned long long* d_sketch_stat, double* d_fl) {
  const int nt = (int)pl.torder.size();
  if (nt <= 0 || P <= 0) return;
  // Targets are listed by increasing sketch size; each launch takes those up to
  // the next of these shared-memory sizes (4, 3 and 2 CTAs per SM; one CTA of a cluster
  // of OCL), so that small sketches do not pay for the large ones' occupancy.  Few
  // targets fill no SM twice anyway and need no classes.  Sketches beyond the largest size
  // stay in global memory (L2).
  constexpr int NCLS = 4;
  static const size_t cls[NCLS] = {55296, 74752, 112640, 221184};
  const double t2 = tau * tau;
  const FF tau2{(float)t2, (float)(t2 - (double)(float)t2)};
  auto bytes = [&](int q, int c) {   // per CTA
    const TInfo& ti = pl.targets[pl.torder[q]];
    const int rows = c < NCLS - 1 ? ti.m : (ti.m + OCL - 1) / OCL;
    return (size_t)orth_ld(rows) * ti.p * sizeof(FF);
  };
  const bool few = (int64_t)nt * P <= device_sm_count(), narrow = pl.max_p <= 32;
  int beg = 0;
  for (int c = few ? NCLS - 2 : 0; c <= NCLS && beg < nt; ++c) {
    int end = nt;
    if (c < NCLS)
      for (end = beg; end < nt && bytes(end, c) <= cls[c]; ++end) {}
    if (end > beg) {
      auto kern = c < NCLS - 1    ? (narrow ? k_orth<ORTH_SM, 1> : k_orth<ORTH_SM, 2>)
                  : c == NCLS - 1 ? (narrow ? k_orth_cluster<1> : k_orth_cluster<2>)
                                  : (narrow ? k_orth<ORTH_GLOBAL, 1> : k_orth<ORTH_GLOBAL, 2>);
      size_t smem = 0;   // (padded: not quite in the targets' order)
      for (int q = beg; c < NCLS && q < end; ++q) smem = std::max(smem, bytes(q, c));
      if (smem > 40 * 1024)   // (48 KB without it, the kernel's own arrays included)
        ACR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)cls[c < NCLS - 1 ? NCLS - 2 : NCLS - 1]));
      const int wide = c == NCLS - 1 ? OCL : 1;   // CTAs per target
      for (int t0 = beg; t0 < end; t0 += 65535 / OCL) {
        kern<<<dim3(std::min(65535 / OCL, end - t0) * wide, P), ONT, smem, st>>>(
            (const TInfo*)pl.d_targets, (const int*)pl.d_torder + t0, tau2, d_tab, d_rtab, P,
            3 * pl.nroles, pl.nroles, (const StackDim*)pl.d_stack, d_sketch_stat, d_fl);
        ACR_LAUNCHED(1);
      }
    }
    beg = end;
  }
}

template <typename T>
void launch_core(const Plan& pl, double eps, int kc, int c_role, T* const* d_tab,
                 int* const* d_rtab, int P, int* d_err, cudaStream_t st, double* d_fl) {
  const int nt = (int)pl.targets.size();
  if (nt <= 0 || P <= 0) return;
  const size_t smem = core_smem(pl.max_p);
  if (smem > 40 * 1024)
    ACR_CUDA(cudaFuncSetAttribute(k_core<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)core_smem(CMAX)));
  for (int t0 = 0; t0 < nt; t0 += 65535) {
    const dim3 grid(std::min(65535, nt - t0), P);
    k_core<T><<<grid, CNT, smem, st>>>((const TInfo*)pl.d_targets, t0, eps, kc, c_role, pl.max_p,
                                       d_tab, d_rtab, P, 3 * pl.nroles, pl.nroles, d_err, d_fl);
    ACR_LAUNCHED(1);
  }
}

template void launch_core<double>(const Plan&, double, int, int, double* const*, int* const*, int,
                                  int*, cudaStream_t, double*);
template void launch_core<float>(const Plan&, double, int, int, float* const*, int* const*, int,
                                 int*, cudaStream_t, double*);

}  // namespace acr
