// Recompression cores of float targets (sm_103a), one CTA per low-rank target:
//  * k_orth -- orthonormal basis of the sketch Y: pivoted Gram-Schmidt with
//              re-orthogonalisation, truncated at tau;
//  * k_core -- core Gram (B^T)^T B^T, its Jacobi eigen-decomposition, the rank
//              rule sigma_i > eps * sigma_1 (Sec. 4.3 H_eps), and the
//              recomposed factors U = Q W_k, V = B^T W_k.
// (FP64 factors go through the Gram, k_pchol and k_eig stages of the plan.)
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "acr_device.h"
#include "acr_internal.h"

namespace acr {

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

// Orthonormal basis Q of range(Y) (m x p, in place): the column of largest
// remaining norm is taken, projected once more against the basis so far (the
// second pass that makes Gram-Schmidt orthonormal to rounding), and removed from
// the remaining columns, whose norms are then recomputed; stops when the largest
// remaining norm is at most tau times the largest of Y.  Basis columns are kept
// unscaled with the square of their reciprocal norm, and scaled at the end.
//
// Bound by the latency of the r dependent steps, not by arithmetic or bytes
// (64 x 32 floats per typical target): Y stays in shared memory, a warp owns
// whole columns (CPW of them, their sums and reductions side by side; no barrier
// between a column's dot and its axpy), and a step has three barriers.  It
// replaces six launches of the plan (two compensated Grams, two FP64 pivoted
// Cholesky cores, two basis products: 95 ms of the n = 64 setup; here 25 ms, and
// 30 ms with the columns of a warp one after another and a fourth barrier).
constexpr int ONT = 256;

template <bool SMEM, int CPW>
__global__ void __launch_bounds__(ONT, 6) k_orth(const TInfo* __restrict__ tis,
                                              const int* __restrict__ order, double tau_,
                                              float* const* __restrict__ tab,
                                              int* const* __restrict__ rtab, int P, int scr_buf,
                                              int scr_rbuf, const StackDim* __restrict__ stack,
                                              unsigned long long* __restrict__ sketch_stat,
                                              double* __restrict__ flops) {
  constexpr int NW = ONT / 32;
  extern __shared__ float ysm[];
  __shared__ float nrm[CMAX], rn2[CMAX];
  __shared__ __align__(16) float dot[CMAX];
  __shared__ __align__(16) float part[NW];
  const int p = blockIdx.y;
  const TInfo ti = tis[order[blockIdx.x]];
  float* scr = tab[scr_buf * P + p];
  int* rs = rtab[scr_rbuf * P + p];
  if (!scr || !rs) return;
  const int m = ti.m, pc = ti.p;
  float* Yg = scr + ti.y_off;
  float* Y = SMEM ? ysm : Yg;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  {
    float s[CPW];
#pragma unroll
    for (int u = 0; u < CPW; ++u) s[u] = 0.f;
    for (int i = lane; i < m; i += 32)
#pragma unroll
      for (int u = 0; u < CPW; ++u) {
        const int c = warp + NW * u;
        if (c < pc) {
          const float v = Yg[i + (int64_t)c * m];
          if (SMEM) Y[i + c * m] = v;
          s[u] = fmaf(v, v, s[u]);
        }
      }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int u = 0; u < CPW; ++u) s[u] += __shfl_xor_sync(FULL, s[u], o);
#pragma unroll
    for (int u = 0; u < CPW; ++u)
      if (lane == 0 && warp + NW * u < pc) nrm[warp + NW * u] = s[u];
  }
  if (sketch_stat && warp == NW - 1)
    count_stacked_warp(ti, stack, tab, (const int* const*)rtab, P, p, sketch_stat);
  __syncthreads();
  const float tau2 = (float)(tau_ * tau_);
  float tol = 0.f;
  bool scaled = false;
  int r = 0;
  for (int j = 0; j < pc; ++j) {
    // every warp finds the largest remaining column: bits of the squared norms
    // order like the norms, the low six hold the column (norms that agree to
    // 2^-17 count as equal: the lowest column); NaN norms are passed over
    unsigned ka = 0u, kb = 0u;
    if (j + lane < pc && nrm[j + lane] > 0.f)
      ka = (__float_as_uint(nrm[j + lane]) & ~63u) | (63u - (j + lane));
    if (CPW > 4 && j + lane + 32 < pc && nrm[j + lane + 32] > 0.f)
      kb = (__float_as_uint(nrm[j + lane + 32]) & ~63u) | (63u - (j + lane + 32));
    const unsigned kbest = __reduce_max_sync(FULL, max(ka, kb));
    if (kbest == 0u) break;
    const int q = 63 - (int)(kbest & 63u);
    const float best = nrm[q];
    if (j == 0) {
      // a sketch so small that its squares would lose bits: scaled by a power of
      // two (Q does not depend on it)
      if (best < 0x1p-80f && !scaled) {
        const float f = ldexpf(1.f, -(ilogbf(best) / 2));
        for (int c = warp; c < pc; c += NW) {
          float s = 0.f;
          for (int i = lane; i < m; i += 32) {
            const float v = f * Y[i + (int64_t)c * m];
            Y[i + (int64_t)c * m] = v;
            s = fmaf(v, v, s);
          }
          s = warp_sum(s);
          __syncwarp();
          if (lane == 0) rn2[c] = s;
        }
        __syncthreads();
        if (tid < pc) nrm[tid] = rn2[tid];
        __syncthreads();
        scaled = true;
        j = -1;
        continue;
      }
      tol = tau2 * best;
    }
    if (!(best > tol)) break;
    float* yq = Y + (int64_t)q * m;
    float* yj = Y + (int64_t)j * m;
    // second projection against the basis so far
    if (warp < j) {
      float s[CPW];
#pragma unroll
      for (int u = 0; u < CPW; ++u) s[u] = 0.f;
      for (int i = lane; i < m; i += 32) {
        const float v = yq[i];
#pragma unroll
        for (int u = 0; u < CPW; ++u) {
          const int c = warp + NW * u;
          if (c < j) s[u] = fmaf(Y[i + (int64_t)c * m], v, s[u]);
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < CPW; ++u) s[u] += __shfl_xor_sync(FULL, s[u], o);
#pragma unroll
      for (int u = 0; u < CPW; ++u) {
        const int c = warp + NW * u;
        if (lane == 0 && c < j) dot[c] = s[u] * rn2[c];
      }
    }
    __syncthreads();
    // (the interchange of columns j and q folded in: a thread owns its rows)
    float s2 = 0.f;
    for (int i = tid; i < m; i += ONT) {
      float v = yq[i];
      int c = 0;
      for (; c + 4 <= j; c += 4) {
        const float4 d = *reinterpret_cast<const float4*>(dot + c);
        const float* y = Y + i + (int64_t)c * m;
        const float y0 = y[0], y1 = y[m], y2 = y[2 * (int64_t)m], y3 = y[3 * (int64_t)m];
        v = fmaf(-d.x, y0, v);
        v = fmaf(-d.y, y1, v);
        v = fmaf(-d.z, y2, v);
        v = fmaf(-d.w, y3, v);
      }
      for (; c < j; ++c) v = fmaf(-dot[c], Y[i + (int64_t)c * m], v);
      if (q != j) yq[i] = yj[i];
      yj[i] = v;
      s2 = fmaf(v, v, s2);
    }
    s2 = warp_sum(s2);
    if (lane == 0) part[warp] = s2;
    __syncthreads();
    const float4 p0 = *reinterpret_cast<const float4*>(part);
    const float4 p1 = *reinterpret_cast<const float4*>(part + 4);
    const float nv = ((p0.x + p0.y) + (p0.z + p0.w)) + ((p1.x + p1.y) + (p1.z + p1.w));
    const float rr = nv >= 0x1p-126f ? 1.f / nv : 0.f;
    if (tid == 0) rn2[j] = rr;
    // remove it from the remaining columns (this warp's from c0 on); their norms afresh
    const int c0 = warp + NW * ((j + 1 - warp + NW - 1) / NW);
    if (c0 < pc) {
      float s[CPW], t[CPW];
#pragma unroll
      for (int u = 0; u < CPW; ++u) s[u] = t[u] = 0.f;
      for (int i = lane; i < m; i += 32) {
        const float v = yj[i];
#pragma unroll
        for (int u = 0; u < CPW; ++u)
          if (c0 + NW * u < pc) s[u] = fmaf(v, Y[i + (int64_t)(c0 + NW * u) * m], s[u]);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < CPW; ++u) s[u] += __shfl_xor_sync(FULL, s[u], o);
#pragma unroll
      for (int u = 0; u < CPW; ++u) s[u] *= rr;
      for (int i = lane; i < m; i += 32) {
        const float v = yj[i];
#pragma unroll
        for (int u = 0; u < CPW; ++u)
          if (c0 + NW * u < pc) {
            float* y = Y + i + (int64_t)(c0 + NW * u) * m;
            const float w = fmaf(-s[u], v, *y);
            *y = w;
            t[u] = fmaf(w, w, t[u]);
          }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int u = 0; u < CPW; ++u) t[u] += __shfl_xor_sync(FULL, t[u], o);
#pragma unroll
      for (int u = 0; u < CPW; ++u)
        if (lane == 0 && c0 + NW * u < pc) nrm[c0 + NW * u] = t[u];
    }
    r = j + 1;
    __syncthreads();
  }
  for (int c = warp; c < r; c += NW) {
    const float f = sqrtf(rn2[c]);
    for (int i = lane; i < m; i += 32) Yg[i + (int64_t)c * m] = f * Y[i + (int64_t)c * m];
  }
  if (tid == 0) {
    rs[ti.r_ri] = r;
    if (flops) atomicAdd(flops, (double)m * r * (4.0 * pc));
  }
}

// ------------------------------------------------------------ float-float
// Numbers held as an unevaluated sum hi + lo of two floats (~48 significant
// bits): the core Gram and its Jacobi rotations run on the FP32 pipe instead of
// this part's narrow FP64 pipe.
struct FF {
  float h, l;
};
__device__ __forceinline__ FF ff_mul(FF a, FF b) {
  const float p = a.h * b.h;
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
// (1 + t^2)^(-1/2) to float-float accuracy: one Newton step y + y (1 - x y^2) / 2
// from the float estimate
__device__ __forceinline__ FF ff_rsqrt1p(float t) {
  const float p = t * t;
  const FF x = ff_add(FF{1.f, 0.f}, FF{p, fmaf(t, t, -p)});
  const float y = rsqrtf(x.h);
  const FF xy2 = ff_mul(x, ff_mul(FF{y, 0.f}, FF{y, 0.f}));
  const FF e = ff_add(FF{1.f, 0.f}, ff_neg(xy2));
  return ff_add(FF{y, 0.f}, ff_mul(FF{y, 0.f}, FF{0.5f * e.h, 0.5f * e.l}));
}
// The rotation (c, s) that zeroes a_pq of [a_pp a_pq; a_pq a_qq]: the angle in
// float with the fast divide (an angle off by ~1e-6 leaves ~1e-6 of the entry, which
// later rotations remove), its cosine and sine to float-float accuracy from that angle, so the
// rotation itself is orthogonal to ~1e-14.
__device__ __forceinline__ void ff_rot(FF app, FF aqq, FF apq, FF& c, FF& s) {
  c = FF{1.f, 0.f};
  s = FF{0.f, 0.f};
  if (apq.h != 0.f) {
    const float tau =
        fminf(fmaxf(__fdividef(aqq.h - app.h, 2.f * apq.h), -1e15f), 1e15f);
    const float h = fmaf(tau, tau, 1.f);
    const float t = copysignf(__fdividef(1.f, fabsf(tau) + h * rsqrtf(h)), tau);
    c = ff_rsqrt1p(t);
    s = ff_mul(FF{t, 0.f}, c);
  }
}

// The core H = (B^T)^T B^T of a target (r x r, r the basis size): exact
// products and compensated float-float sums, since the rank rule resolves
// singular values only down to the square root of the Gram's relative error;
// scaled by a power of two to a largest diagonal in [1/2, 1), so that blocks whose
// squares would leave the float range keep the full float-float accuracy (an
// exact scaling: the eigenvectors and the ratios sigma_i / sigma_1 are
// unchanged); cyclic Jacobi in round-robin order, the symmetric half of each
// round's 2 x 2 blocks rotated by one thread each (the mirror entry written
// alongside) together with V; then the kept columns W of V, largest eigenvalue first, and
// the factors U = Q W, V = B^T W straight into the target's leaf.
//
// Bound by the latency of the ~6 (r - 1) dependent rounds of a core, each a
// rotation angle and a handful of float-float operations per thread.  Four warps,
// so that a typical core's round (r = 12: 21 blocks and 72 row pairs of V) is one
// pass over the threads; every warp computes all rotations in its lanes and
// hands them round by shuffles, and a round writes the other copy of A, so
// that it has one barrier.  n = 64 setup: the four stages 90 ms, here 31 ms (36 ms with
// rotations through shared memory and A updated in place).
constexpr int CNT = 128;
constexpr int CRAW = CNT * 16;   // float-float partial sums of the Gram's tiles

__host__ __device__ constexpr size_t core_smem(int p) {
  // A; the Gram's staging, then the other A and V in its place (p x (p + 1)
  // float-float each); W
  const size_t a = (size_t)p * (p + 1) * sizeof(FF), g = CRAW * sizeof(FF);
  return a + (2 * a > g ? 2 * a : g) + (size_t)p * ((p + 3) & ~3) * sizeof(float);
}

__global__ void __launch_bounds__(CNT) k_core(const TInfo* __restrict__ tis, int tbase, double eps,
                                              int kc, int c_role, int maxp,
                                              float* const* __restrict__ tab,
                                              int* const* __restrict__ rtab, int P, int scr_buf,
                                              int scr_rbuf, int* err, double* __restrict__ flops) {
  const int p = blockIdx.y;
  const TInfo ti = tis[tbase + blockIdx.x];
  float* scr = tab[scr_buf * P + p];
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
  FF* A = reinterpret_cast<FF*>(csm);
  FF* A2 = A + (size_t)maxp * (maxp + 1);
  FF* V = A2 + (size_t)maxp * (maxp + 1);
  FF* raw = A2;   // the Gram is done before the second A and V begin
  float* W = reinterpret_cast<float*>(A2 + max(2 * (size_t)maxp * (maxp + 1), (size_t)CRAW));
  __shared__ float red[2][CNT / 32];
  __shared__ float lam[CMAX];
  __shared__ int ord[CMAX];
  __shared__ int kkeep;

  // ---- Gram of B^T (n x r): thread (tile, slice) owns a 4 x 4 tile of the
  // upper triangle and every S-th row
  const float* B = scr + ti.bt_off;
  const int n = ti.n;
  {
    const int TM = (r + 3) >> 2, ntile = TM * (TM + 1) / 2, mt = 4 * TM;
    // (CRAW float-float entries staged as 2 CRAW floats; at least 31 rows)
    const int kch = min(256, ((2 * CRAW / mt) - 1) & ~1), ysld = kch + 1;
    float* ys = reinterpret_cast<float*>(raw);
    for (int tb = 0; tb < ntile; tb += CNT) {   // (one pass up to r = 60)
      const int nt = min(CNT, ntile - tb);
      const int S = CNT / nt;
      const int tl = tid / S, slice = tid - tl * S;
      const bool active = tl < nt;
      int a0 = 0, t = tb + (active ? tl : 0);
      while (t >= TM - a0) { t -= TM - a0; ++a0; }
      const int i0 = 4 * a0, j0 = 4 * (a0 + t);
      float s[4][4], c[4][4];
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) { s[x][y] = 0.f; c[x][y] = 0.f; }
      for (int l0 = 0; l0 < n; l0 += kch) {
        const int kk = min(kch, n - l0);
        __syncthreads();
        for (int col = tid >> 5; col < mt; col += CNT / 32)
          for (int l = lane; l < kk; l += 32)
            ys[col * ysld + l] = col < r ? B[(l0 + l) + (int64_t)col * n] : 0.f;
        __syncthreads();
        if (active)
          for (int l = slice; l < kk; l += S) {
            float av[4], bv[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              av[x] = ys[(i0 + x) * ysld + l];
              bv[x] = ys[(j0 + x) * ysld + l];
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
              for (int y = 0; y < 4; ++y) ff_fma(s[x][y], c[x][y], av[x], bv[y]);
          }
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < 16; ++e)
        raw[e * CNT + tid] = active ? FF{s[e & 3][e >> 2], c[e & 3][e >> 2]} : FF{0.f, 0.f};
      __syncthreads();
      // the slices' partial sums in float-float, in a fixed order
      for (int e = tid; e < nt * 16; e += CNT) {
        const int tq = e >> 4, q = e & 15;
        FF h{0.f, 0.f};
        for (int sl = 0; sl < S; ++sl) {
          const FF x = raw[q * CNT + tq * S + sl];
          const float u = h.h + x.h, bp = u - h.h;
          h.l += ((h.h - (u - bp)) + (x.h - bp)) + x.l;
          h.h = u;
        }
        const float u = h.h + h.l;
        h.l = h.l - (u - h.h);
        h.h = u;
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
  float dmax = 0.f;
  for (int i = 0; i < r; ++i) dmax = fmaxf(dmax, A[i * lda + i].h);
  int ex = 0;
  if (dmax > 0.f && dmax <= 3.0e38f) frexpf(dmax, &ex);
  __syncthreads();
  for (int e = tid; e < r * lda; e += CNT) {
    const int i = e / lda, j = e - i * lda;
    A[e].h = ldexpf(A[e].h, -ex);
    A[e].l = ldexpf(A[e].l, -ex);
    V[e] = FF{i == j ? 1.f : 0.f, 0.f};
  }
  __syncthreads();

  // ---- cyclic Jacobi
  const int nn = (r + 1) & ~1;   // even number of players (an odd r gets a dummy)
  const int np = nn / 2, nblk = np * (np + 1) / 2;
  // work items of a round: the blocks k1 <= k2 of A, then from a whole warp on
  // the (pair, row) items of V; a thread's items stay its own, the first few's
  // indices in registers (x | y << 8: k1, k2 or pair, row; -1: none)
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
  for (int sweep = 0; sweep < 40 && r > 1; ++sweep) {
    // off-diagonal and total mass; converged at 1e-16 (eigenvectors to ~1e-8)
    float off = 0.f, tot = 0.f;
    for (int i = tid >> 5; i < r; i += CNT / 32)
      for (int j = lane; j < r; j += 32) {
        const float v = A[i * lda + j].h;
        if (i != j) off = fmaf(v, v, off);
        else tot = fmaf(v, v, tot);
      }
    off = warp_sum(off);
    tot = warp_sum(tot);
    if (lane == 0) { red[0][tid >> 5] = off; red[1][tid >> 5] = tot; }
    __syncthreads();
    off = (red[0][0] + red[0][1]) + (red[0][2] + red[0][3]);
    tot = (red[1][0] + red[1][1]) + (red[1][2] + red[1][3]);
    if (off <= 1e-16f * (tot + off)) break;
    ++sweeps;
    for (int round = 0; round < nn - 1; ++round) {
      // lane k: the rotation of pair k
      FF rc{1.f, 0.f}, rsn{0.f, 0.f};
      if (lane < np) {
        int lo, hi;
        pair_of(lane, round, lo, hi);
        if (hi < r) ff_rot(A[lo * lda + lo], A[hi * lda + hi], A[lo * lda + hi], rc, rsn);
      }
      auto rot = [&](int k, FF& c, FF& s) {
        c.h = __shfl_sync(FULL, rc.h, k); c.l = __shfl_sync(FULL, rc.l, k);
        s.h = __shfl_sync(FULL, rsn.h, k); s.l = __shfl_sync(FULL, rsn.l, k);
      };
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
        if (e0 < vbase) {
          // A <- J^T A J into the other copy: the 2 x 2 block (rows of pair k1,
          // columns of pair k2) is rotated on its own, columns first, then
          // rows, and mirrored
          const int k1 = on ? id & 255 : 0, k2 = on ? id >> 8 : 0;
          FF c1, s1, c2, s2;
          rot(k1, c1, s1);
          rot(k2, c2, s2);
          if (on) {
            int a1, b1, a2, b2;
            pair_of(k1, round, a1, b1);
            pair_of(k2, round, a2, b2);
            const bool h1 = b1 < r, h2 = b2 < r;
            const FF z{0.f, 0.f};
            const FF x00 = A[a1 * lda + a2];
            const FF x01 = h2 ? A[a1 * lda + b2] : z;
            const FF x10 = h1 ? A[b1 * lda + a2] : z;
            const FF x11 = (h1 && h2) ? A[b1 * lda + b2] : z;
            const FF y00 = ff_add(ff_mul(c2, x00), ff_neg(ff_mul(s2, x01)));
            const FF y01 = ff_add(ff_mul(s2, x00), ff_mul(c2, x01));
            const FF y10 = ff_add(ff_mul(c2, x10), ff_neg(ff_mul(s2, x11)));
            const FF y11 = ff_add(ff_mul(s2, x10), ff_mul(c2, x11));
            const FF z00 = ff_add(ff_mul(c1, y00), ff_neg(ff_mul(s1, y10)));
            const FF z01 = ff_add(ff_mul(c1, y01), ff_neg(ff_mul(s1, y11)));
            const FF z10 = ff_add(ff_mul(s1, y00), ff_mul(c1, y10));
            const FF z11 = ff_add(ff_mul(s1, y01), ff_mul(c1, y11));
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
          FF c, s;
          rot(k, c, s);
          int a, b;
          pair_of(k, round, a, b);
          if (on && b < r) {
            const FF vx = V[iv * lda + a], vy = V[iv * lda + b];
            V[iv * lda + a] = ff_add(ff_mul(c, vx), ff_neg(ff_mul(s, vy)));
            V[iv * lda + b] = ff_add(ff_mul(s, vx), ff_mul(c, vy));
          }
        }
      }
      __syncthreads();
      FF* t = A;
      A = A2;
      A2 = t;
    }
  }
  // ---- eigenvalues descending (rank by counting; ties by index), the kept rank
  for (int i = tid; i < r; i += CNT) lam[i] = A[i * lda + i].h;
  __syncthreads();
  for (int i = tid; i < r; i += CNT) {
    const double li = (double)lam[i] + (double)A[i * lda + i].l;
    int pos = 0;
    for (int j = 0; j < r; ++j) {
      const double lj = (double)lam[j] + (double)A[j * lda + j].l;
      if (lj > li || (lj == li && j < i)) ++pos;
    }
    ord[pos] = i;
  }
  __syncthreads();
  if (tid == 0) {
    const FF f0 = A[ord[0] * lda + ord[0]];
    const double l1 = (double)f0.h + (double)f0.l;
    const double cut = eps * eps * l1;   // sigma_i > eps sigma_1
    int k = 0;
    if (l1 > 0.0)
      for (int j = 0; j < r; ++j) {
        const FF f = A[ord[j] * lda + ord[j]];
        const double lj = (double)f.h + (double)f.l;
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
  // ---- recomposition: W (r x k, row by row, rows of whole float4)
  const int ldw = (k + 3) & ~3;
  for (int e = tid; e < r * ldw; e += CNT) {
    const int i = e / ldw, j = e - i * ldw;
    float w = 0.f;
    if (j < k) {
      const FF v = V[i * lda + ord[j]];
      w = v.h + v.l;
    }
    W[e] = w;
  }
  __syncthreads();
  float* Uo = tab[(3 * c_role + 1) * P + p];
  float* Vo = tab[(3 * c_role + 2) * P + p];
  const int m = ti.m;
  for (int e = tid; e < m + n; e += CNT) {   // a row of U = Q W, then of V = B^T W
    const bool u = e < m;
    const int rows = u ? m : n, i = u ? e : e - m;
    const float* X = (u ? scr + ti.y_off : B) + i;
    float* Z = u ? Uo : Vo;
    if (!Z) continue;
    Z += (u ? ti.u_off : ti.v_off) + i;
    for (int j0 = 0; j0 < k; j0 += 4) {
      float4 acc{0.f, 0.f, 0.f, 0.f};
#pragma unroll 8
      for (int l = 0; l < r; ++l) {
        const float x = X[(int64_t)l * rows];
        const float4 w = *reinterpret_cast<const float4*>(W + l * ldw + j0);
        acc.x = fmaf(x, w.x, acc.x); acc.y = fmaf(x, w.y, acc.y);
        acc.z = fmaf(x, w.z, acc.z); acc.w = fmaf(x, w.w, acc.w);
      }
      float* z = Z + (int64_t)j0 * rows;
      z[0] = acc.x;
      if (j0 + 1 < k) z[rows] = acc.y;
      if (j0 + 2 < k) z[2 * (int64_t)rows] = acc.z;
      if (j0 + 3 < k) z[3 * (int64_t)rows] = acc.w;
    }
  }
}

}  // namespace

void launch_orth(const Plan& pl, double tau, float* const* d_tab, int* const* d_rtab, int P,
                 cudaStream_t st, unsigned long long* d_sketch_stat, double* d_fl) {
  const int nt = (int)pl.torder.size();
  if (nt <= 0 || P <= 0) return;
  // Targets are listed by increasing sketch size; each launch takes those up to
  // the next of these shared-memory sizes (8, 4, 2 and 1 CTA per SM), so that
  // small sketches do not pay for the large ones' occupancy.  Few targets fill
  // no SM twice anyway and go in one launch.  Sketches beyond the largest size
  // stay in global memory (L2).
  static const size_t cls[4] = {28160, 56320, 112640, 225280};
  constexpr int NCLS = 4;
  auto bytes = [&](int q) {
    const TInfo& ti = pl.targets[pl.torder[q]];
    return (size_t)ti.m * ti.p * sizeof(float);
  };
  const bool few = (int64_t)nt * P <= device_sm_count();
  int beg = 0;
  for (int c = few ? NCLS - 1 : 0; c <= NCLS && beg < nt; ++c) {
    int end = nt;
    if (c < NCLS)
      for (end = beg; end < nt && bytes(end) <= cls[c]; ++end) {}
    if (end > beg) {
      auto kern = c < NCLS ? (pl.max_p <= 32 ? k_orth<true, 4> : k_orth<true, 8>)
                           : (pl.max_p <= 32 ? k_orth<false, 4> : k_orth<false, 8>);
      const size_t smem = c < NCLS ? bytes(end - 1) : 0;
      if (smem > 48 * 1024)
        ACR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)cls[NCLS - 1]));
      for (int t0 = beg; t0 < end; t0 += 65535) {
        kern<<<dim3(std::min(65535, end - t0), P), ONT, smem, st>>>(
            (const TInfo*)pl.d_targets, (const int*)pl.d_torder + t0, tau, d_tab, d_rtab, P,
            3 * pl.nroles, pl.nroles, (const StackDim*)pl.d_stack, d_sketch_stat, d_fl);
        ACR_LAUNCHED(1);
      }
    }
    beg = end;
  }
}

void launch_core(const Plan& pl, double eps, int kc, int c_role, float* const* d_tab,
                 int* const* d_rtab, int P, int* d_err, cudaStream_t st, double* d_fl) {
  const int nt = (int)pl.targets.size();
  if (nt <= 0 || P <= 0) return;
  const size_t smem = core_smem(pl.max_p);
  if (smem > 48 * 1024)
    ACR_CUDA(cudaFuncSetAttribute(k_core, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)core_smem(CMAX)));
  for (int t0 = 0; t0 < nt; t0 += 65535) {
    const dim3 grid(std::min(65535, nt - t0), P);
    k_core<<<grid, CNT, smem, st>>>((const TInfo*)pl.d_targets, t0, eps, kc, c_role, pl.max_p,
                                    d_tab, d_rtab, P, 3 * pl.nroles, pl.nroles, d_err, d_fl);
    ACR_LAUNCHED(1);
  }
}

}  // namespace acr
