// Setup kernels of the ACR engine (sm_103a), besides the grouped GEMMs of
// acr_gemm_kernels.cu and the recompression cores of acr_core_kernels.cu:
//  * k_pchol   -- pivoted Cholesky of a sketch Gram (FP64 factors): orthonormal
//                 basis transform of the range finder;
//  * k_leaf_inv_d, k_leaf_inv_f -- Gauss-Jordan inverse with partial pivoting of a dense
//                 diagonal leaf (the leaves of the recursive H-inverse): FP64,
//                 or for float storage float elimination refined to float
//                 accuracy (FP64 when refinement cannot get there);
//  * k_hscale  -- exact diagonal scalings diag(r) X diag(c) (first CR level,
//                 where the plane couplings are diagonal);
//  * k_plane_dense / k_plane_lr -- H-format of a 7-point plane block.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <type_traits>

#include <cstdint>

#include "acr_device.h"
#include "acr_internal.h"

namespace acr {

namespace cg = cooperative_groups;

namespace {

// ---------------------------------------------------------------- cores
constexpr int CMAX = 64;   // largest sketch / core dimension

// Pivoted Cholesky of G (pd x pd): G = P L L^T P^T, stop when the largest
// remaining diagonal <= tau^2 * max diag(G) (truncating pass).  Writes
// T (p x r, ld p) with Q = Y T orthonormal, and r.
//
// The truncating pass also counts the target (sketch_stat[0]) and, when the
// stacked rank of its summed terms exceeds the sketch width p, the range
// finder's inexact case (sketch_stat[1]).
template <typename T>
__device__ void count_stacked(const TInfo& ti, const StackDim* __restrict__ stack,
                              T* const* __restrict__ tab, const int* const* __restrict__ rtab,
                              int P, int p, unsigned long long* sketch_stat) {
  int64_t stacked = 0;
  for (int e = ti.sk_beg; e < ti.sk_end; ++e) {
    const StackDim sd = stack[e];
    if (sd.g0 >= 0 && !tab[sd.g0 * P + p]) continue;
    if (sd.g1 >= 0 && !tab[sd.g1 * P + p]) continue;
    stacked += dimv(sd.st, sd.rb, sd.ri, rtab, P, p);
  }
  atomicAdd(sketch_stat, 1ull);
  if (stacked > ti.p) atomicAdd(sketch_stat + 1, 1ull);
}

constexpr int PCHOL_WARP_MAX = 32;   // Grams up to this size: one warp each
constexpr int PW = 4;                // warps (targets) per CTA of k_pchol_warp
constexpr size_t PCHOL_WARP_SMEM =
    PW * (2 * 32 * 33 * sizeof(double) + 2 * 32 * sizeof(double) + 32 * sizeof(int));

// The same pivoted Cholesky for Grams up to 32 x 32, one warp per target,
// four targets per CTA, warp barriers only: lane i owns row i of the pivot
// search, of each new factor column and (for the inverse) column i.
template <typename T>
__global__ void __launch_bounds__(32 * PW) k_pchol_warp(
    const TInfo* __restrict__ tis, int tbase, int tend, bool truncate, double tau,
    T* const* __restrict__ tab, int* const* __restrict__ rtab, int P, int scr_buf, int scr_rbuf,
    const StackDim* __restrict__ stack, unsigned long long* __restrict__ sketch_stat,
    double* __restrict__ flops) {
  constexpr int M = PCHOL_WARP_MAX;
  const int p = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = tbase + blockIdx.x * PW + warp;
  if (t >= tend) return;
  const TInfo ti = tis[t];
  T* scr = tab[scr_buf * P + p];
  int* rs = rtab[scr_rbuf * P + p];
  if (!scr || !rs) return;
  const int ld = ti.p;
  const int pd = truncate ? ti.p : rs[ti.r_ri];
  if (pd > M) return;   // k_pchol takes it
  if (truncate && sketch_stat && lane == 0) count_stacked(ti, stack, tab, rtab, P, p, sketch_stat);
  extern __shared__ double dsm[];
  double* base = dsm + (size_t)warp * (2 * 32 * 33 + 2 * 32 + 16);
  double (*L)[M + 1] = reinterpret_cast<double (*)[M + 1]>(base);
  double (*F)[M + 1] = reinterpret_cast<double (*)[M + 1]>(base + 32 * 33);
  double* d = base + 2 * 32 * 33;
  double* colbuf = d + 32;
  int* piv = reinterpret_cast<int*>(colbuf + 32);
  const double* G = reinterpret_cast<const double*>(scr + ti.g_off);   // FP64 Gram
  T* Tm = scr + ti.t_off;
  for (int e = lane; e < pd * pd; e += 32) {
    const int i = e % pd, j = e / pd;
    L[i][j] = G[i + (int64_t)j * ld];
  }
  for (int e = lane; e < M * (M + 1); e += 32) (&F[0][0])[e] = 0.0;
  __syncwarp();
  double dm = 0.0;
  if (lane < pd) {
    d[lane] = L[lane][lane];
    piv[lane] = lane;
    dm = d[lane];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
  __syncwarp();
  const double tol = truncate ? tau * tau * dm : 1e-30 * dm;
  int r = 0;
  for (int j = 0; j < pd; ++j) {
    // largest remaining diagonal among pivoted positions j..pd-1
    double best = -1.0;
    int bi = -1;
    if (lane >= j && lane < pd) { best = d[piv[lane]]; bi = lane; }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (oi >= 0 && (bi < 0 || ov > best || (ov == best && oi < bi))) { best = ov; bi = oi; }
    }
    if (bi < 0 || !(best > tol) || !(best > 0.0)) {
      if (!truncate) r = pd;
      break;
    }
    const int q = bi;
    const double ljj = sqrt(best);
    __syncwarp();
    if (lane == 0) { const int tt = piv[j]; piv[j] = piv[q]; piv[q] = tt; }
    __syncwarp();
    const double rjj = 1.0 / ljj;   // one division per column (FP64 division is slow here)
    if (lane >= j && lane < pd) {
      const int i = lane;
      const int src = (i == j) ? q : (i == q ? j : i);
      double sum = L[piv[i]][piv[j]];
      for (int l = 0; l < j; ++l) sum -= F[src][l] * F[q][l];
      colbuf[i] = (i == j) ? ljj : sum * rjj;
    }
    __syncwarp();
    if (q != j && lane < j) {
      const double tt = F[j][lane]; F[j][lane] = F[q][lane]; F[q][lane] = tt;
    }
    if (lane >= j && lane < pd) {
      F[lane][j] = colbuf[lane];
      if (lane > j) d[piv[lane]] -= colbuf[lane] * colbuf[lane];
    }
    __syncwarp();
    if (lane == 0) d[piv[j]] = 0.0;
    __syncwarp();
    r = j + 1;
  }
  __syncwarp();
  // inverse of the r x r lower factor, column c by lane c, into L (the
  // diagonal's reciprocals taken once, by lane i for row i)
  if (lane < r) d[lane] = (F[lane][lane] != 0.0) ? 1.0 / F[lane][lane] : 0.0;
  __syncwarp();
  if (lane < r) {
    const int c = lane;
    for (int i = 0; i < r; ++i) {
      double sacc = (i == c) ? 1.0 : 0.0;
      for (int l = c; l < i; ++l) sacc -= F[i][l] * L[l][c];
      L[i][c] = (i >= c) ? sacc * d[i] : 0.0;
    }
  }
  __syncwarp();
  for (int e = lane; e < pd * r; e += 32) {
    const int i = e % pd, c = e / pd;
    Tm[i + (int64_t)c * ld] = (T)0;
  }
  __syncwarp();
  for (int e = lane; e < r * r; e += 32) {
    const int j = e % r, c = e / r;
    Tm[piv[j] + (int64_t)c * ld] = (T)(j <= c ? L[c][j] : 0.0);
  }
  if (lane == 0) {
    rs[ti.r_ri] = r;
    if (flops) atomicAdd(flops, (double)pd * r * r - 2.0 * r * r * r / 3.0 + (double)r * r * r / 3.0);
  }
}

template <typename T>
__global__ void __launch_bounds__(NT) k_pchol(const TInfo* __restrict__ tis, int tbase, bool truncate,
                                              double tau, T* const* __restrict__ tab,
                                              int* const* __restrict__ rtab, int P, int scr_buf,
                                              int scr_rbuf, const StackDim* __restrict__ stack,
                                              unsigned long long* __restrict__ sketch_stat,
                                              double* __restrict__ flops) {
  const int p = blockIdx.y;
  const TInfo ti = tis[tbase + blockIdx.x];
  T* scr = tab[scr_buf * P + p];
  int* rs = rtab[scr_rbuf * P + p];
  if (!scr || !rs) return;
  const int ld = ti.p;
  const int pd = truncate ? ti.p : rs[ti.r_ri];
  if (pd <= PCHOL_WARP_MAX) return;   // k_pchol_warp's cores
  if (truncate && sketch_stat && threadIdx.x == 0) count_stacked(ti, stack, tab, rtab, P, p, sketch_stat);
  extern __shared__ double dsm[];
  double (*L)[CMAX + 1] = reinterpret_cast<double (*)[CMAX + 1]>(dsm);
  double (*F)[CMAX + 1] = reinterpret_cast<double (*)[CMAX + 1]>(dsm + CMAX * (CMAX + 1));
  __shared__ double d[CMAX];
  __shared__ double colbuf[CMAX];
  __shared__ int piv[CMAX];
  __shared__ double sv[NT];
  const double* G = reinterpret_cast<const double*>(scr + ti.g_off);   // FP64 Gram
  T* Tm = scr + ti.t_off;
  for (int e = threadIdx.x; e < pd * pd; e += NT) {
    int i = e % pd, j = e / pd;
    L[i][j] = (double)G[i + (int64_t)j * ld];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < pd; i += NT) { d[i] = L[i][i]; piv[i] = i; }
  __syncthreads();
  // scale reference: largest diagonal
  double dm = 0;
  for (int i = threadIdx.x; i < pd; i += NT) dm = fmax(dm, d[i]);
  sv[threadIdx.x] = dm;
  __syncthreads();
  for (int s = NT / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) sv[threadIdx.x] = fmax(sv[threadIdx.x], sv[threadIdx.x + s]);
    __syncthreads();
  }
  const double dmax = sv[0];
  __syncthreads();
  const double tol = truncate ? tau * tau * dmax : 1e-30 * dmax;
  int r = 0;
  // F: lower factor in pivoted order
  for (int e = threadIdx.x; e < CMAX * (CMAX + 1); e += NT) (&F[0][0])[e] = 0.0;
  __syncthreads();
  __shared__ int s_q, s_stop;
  __shared__ double s_ljj;
  for (int j = 0; j < pd; ++j) {
    if (threadIdx.x < 32) {
      // largest remaining diagonal among pivoted positions j..pd-1
      double best = -1.0;
      int bi = -1;
      for (int i = j + (threadIdx.x & 31); i < pd; i += 32) {
        const double v = d[piv[i]];
        if (v > best) { best = v; bi = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (oi >= 0 && (bi < 0 || ov > best || (ov == best && oi < bi))) { best = ov; bi = oi; }
      }
      if (threadIdx.x == 0) {
        const bool stop = bi < 0 || !(best > tol) || !(best > 0.0);
        s_stop = stop ? 1 : 0;
        if (!stop) {
          const int t = piv[j]; piv[j] = piv[bi]; piv[bi] = t;
          s_q = bi;
          s_ljj = sqrt(best);
        }
      }
    }
    __syncthreads();
    if (s_stop) {
      // truncating pass: the rest of range(Y) is below tau; re-orthogonalising
      // pass: keep the dimension, the remaining directions get zero columns
      if (!truncate) r = pd;
      break;
    }
    const int q = s_q;
    const double ljj = s_ljj;
    // the rows of the partial factor follow the pivot interchange; then column j
    for (int i = j + threadIdx.x; i < pd; i += NT) {
      // row i of the pivoted factor (before this step's swap, row q held what is now row j)
      const int src = (i == j) ? q : (i == q ? j : i);
      double sum = L[piv[i]][piv[j]];
      for (int l = 0; l < j; ++l) sum -= F[src][l] * F[q][l];
      colbuf[i] = (i == j) ? ljj : sum / ljj;
    }
    __syncthreads();
    // the row swap touches columns < j only; column j is written alongside
    if (q != j)
      for (int l = threadIdx.x; l < j; l += NT) {
        const double t = F[j][l]; F[j][l] = F[q][l]; F[q][l] = t;
      }
    for (int i = j + threadIdx.x; i < pd; i += NT) {
      F[i][j] = colbuf[i];
      if (i > j) d[piv[i]] -= colbuf[i] * colbuf[i];
    }
    if (threadIdx.x == 0) d[piv[j]] = 0.0;
    __syncthreads();
    r = j + 1;
  }
  // inverse of the r x r lower factor (columns with zero diagonal give zero)
  // Linv stored in L (reuse): solve F Linv = I column by column (thread per column)
  __syncthreads();
  for (int c = threadIdx.x; c < r; c += NT) {
    for (int i = 0; i < r; ++i) {
      double s = (i == c) ? 1.0 : 0.0;
      for (int l = c; l < i; ++l) s -= F[i][l] * L[l][c];
      L[i][c] = (F[i][i] != 0.0 && i >= c) ? s / F[i][i] : 0.0;
    }
  }
  __syncthreads();
  // T (ld, rows pd): T[piv[j]][c] = Linv[c][j]  (Linv^T), other rows 0
  for (int e = threadIdx.x; e < pd * r; e += NT) {
    int i = e % pd, c = e / pd;
    Tm[i + (int64_t)c * ld] = (T)0;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < r * r; e += NT) {
    int j = e % r, c = e / r;
    Tm[piv[j] + (int64_t)c * ld] = (T)(j <= c ? L[c][j] : 0.0);
  }
  if (threadIdx.x == 0) {
    rs[ti.r_ri] = r;
    if (flops) atomicAdd(flops, (double)pd * r * r - 2.0 * r * r * r / 3.0 + (double)r * r * r / 3.0);
  }
}

// Largest |a| over the block (every thread passes its own candidate).
template <int TH>
__device__ __forceinline__ double block_absmax(double v, double* red8) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red8[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = red8[0];
  for (int w = 1; w < TH / 32; ++w) r = fmax(r, red8[w]);
  __syncthreads();
  return r;
}

// Breakdown bound on the growth max|A| * max|A^-1| of a dense leaf inverse
// (a lower bound on the condition number over n^2).  The leaf is read from
// its storage precision, whose rounding u perturbs it by ~u relatively, so
// the inverse keeps about -log10(growth * u) correct digits: the bound is
// 1e10 for FP64 storage (6 digits kept) and 1e6 for float storage (about
// one digit).  This is how an indefinite plane (Sec. 8) whose leaf nearly
// meets an eigenvalue is caught, not only an exactly zero pivot.
template <typename T>
__host__ __device__ constexpr double leaf_growth_max() { return sizeof(T) == 8 ? 1e10 : 1e6; }

// In-place Gauss-Jordan inverse with partial pivoting, FP64, n <= 64.
// Per elimination step warp 0 finds the pivot with shuffles, takes the one
// reciprocal of the step and publishes the scaled pivot row, the displaced
// row and the multipliers; then every entry is updated with the row
// interchange folded in -- two barriers per step.  Thread t owns row t % 64
// and columns t / 64 + 4 m.  The interchanges become one column permutation
// of the result, applied when it is stored.
// TH threads: thread t owns row t % 64 and columns t / 64 + (TH / 64) m.
template <typename T, int TH>
__device__ void leaf_inv_fp64(T* __restrict__ Ap, int n, double (*A)[CMAX + 1], int* err,
                              double* __restrict__ flops) {
  static_assert(TH % 64 == 0 && TH <= 1024 && CMAX == 64, "64 x 64 leaves, whole rows of threads");
  constexpr int CS = TH / 64;
  __shared__ double rowk[CMAX], colk[CMAX], krow[CMAX];
  __shared__ int piv[CMAX];
  __shared__ int cmap[CMAX];
  __shared__ int s_q, s_bad;
  __shared__ double s_pinv;
  __shared__ double red8[TH / 32];
  const int ti = threadIdx.x & 63, tj = threadIdx.x >> 6;
  double amax = 0.0;
  for (int j = tj; j < n; j += CS)
    if (ti < n) {
      A[ti][j] = (double)Ap[ti + (int64_t)j * n];
      amax = fmax(amax, fabs(A[ti][j]));
    }
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  amax = block_absmax<TH>(amax, red8);
  for (int k = 0; k < n; ++k) {
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      double best = -1.0;
      int q = -1;
      for (int i = k + lane; i < n; i += 32) {
        const double v = fabs(A[i][k]);
        if (v > best) { best = v; q = i; }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const double ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int oi = __shfl_xor_sync(0xffffffffu, q, o);
        if (oi >= 0 && (q < 0 || ov > best || (ov == best && oi < q))) { best = ov; q = oi; }
      }
      // every lane holds the same winner
      if (q < 0 || !(best > 0.0)) {
        if (lane == 0) s_bad = 1;
      } else {
        const double pinv = 1.0 / A[q][k];
        for (int j = lane; j < n; j += 32) {
          rowk[j] = (j == k) ? pinv : A[q][j] * pinv;   // new row k
          krow[j] = A[k][j];                             // old row k (moves to row q)
          colk[j] = (j == k) ? 0.0 : (j == q ? A[k][k] : A[j][k]);   // multipliers after the swap
        }
        if (lane == 0) { s_q = q; s_pinv = pinv; piv[k] = q; }
      }
    }
    __syncthreads();
    if (s_bad) break;
    const int q = s_q;
    const double pinv = s_pinv;
    if (ti < n) {
      const double f = colk[ti];
      for (int j = tj; j < n; j += CS) {
        if (ti == k) {
          A[ti][j] = rowk[j];
        } else {
          const double old = (ti == q) ? krow[j] : A[ti][j];
          A[ti][j] = (j == k) ? -f * pinv : old - f * rowk[j];
        }
      }
    }
    __syncthreads();
  }
  if (s_bad) {
    if (threadIdx.x == 0) atomicOr(err, ERR_PIVOT);
    return;
  }
  // pivot growth of the computed inverse (a NaN or Inf entry fails too)
  double xmax = 0.0;
  for (int j = tj; j < n; j += CS)
    if (ti < n) {
      const double v = fabs(A[ti][j]);
      xmax = (v <= 1.7976931348623157e308) ? fmax(xmax, v) : INFINITY;   // NaN, Inf -> Inf
    }
  xmax = block_absmax<TH>(xmax, red8);
  if (!(amax * xmax <= leaf_growth_max<T>())) {
    if (threadIdx.x == 0) atomicOr(err, ERR_GROWTH);
    return;
  }
  if (threadIdx.x == 0) {
    // the interchanges, undone last first as column swaps, compose into one
    // permutation: stored column c comes from working column pi(c)
    int pi_[CMAX];
    for (int c = 0; c < n; ++c) pi_[c] = c;
    for (int k = n - 1; k >= 0; --k) {
      const int q = piv[k];
      const int t = pi_[k]; pi_[k] = pi_[q]; pi_[q] = t;
    }
    for (int c = 0; c < n; ++c) cmap[pi_[c]] = c;
  }
  __syncthreads();
  for (int j = tj; j < n; j += CS)
    if (ti < n) Ap[ti + (int64_t)cmap[j] * n] = (T)A[ti][j];
  if (flops && threadIdx.x == 0) atomicAdd(flops, 2.0 * n * n * n);
}

template <int TH>
__device__ __forceinline__ float block_absmaxf(float v, float* red8) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) red8[threadIdx.x >> 5] = v;
  __syncthreads();
  float r = red8[0];
  for (int w = 1; w < TH / 32; ++w) r = fmaxf(r, red8[w]);
  __syncthreads();
  return r;
}

// Leaf inverse of float storage without the FP64 pipe (a small fraction of
// the FP32 one on this part): Gauss-Jordan with partial pivoting in float
// gives X0 with relative error ~ cond * 6e-8; mixed-precision iterative
// refinement X <- X + X0 R, R = I - A X, with the residual formed from exact
// products and compensated sums (float-float, ff_fma), then contracts the error
// by ~ |I - X0 A| per step until the correction is below two units in the last
// place of the largest entry: the result is the inverse to float rounding, as
// the FP64 elimination rounded to float gives.
// When it cannot get there (a float pivot of zero, a non-finite entry, a
// correction that does not at least halve, no convergence in eight steps) the
// leaf is inverted by the FP64 elimination instead (the shared buffers
// reused), so the pivot and growth diagnostics are those of the FP64 form.
//
// At most n / 2 leaves are inverted at a time, one per plane, and every other
// launch of the plane waits for them: latency is all that counts.  A cluster of
// LCL CTAs takes one leaf.  Every CTA eliminates the whole leaf (cheaper than
// an exchange per step): panels of 8 columns in one warp's registers, whose
// 8 dependent steps (pivot search by one warp-wide maximum, 8 shuffles, 16
// multiply-adds per lane) need no barrier, then one rank-8 update of the other
// columns by all warps.  The refinement's 2 x 64^3 products per step, which would
// fill one SM for 10 us, are split by columns over the cluster; the outcomes are
// pushed to every CTA before the one cluster barrier.  64 x 64 leaf, 1 to
// 32 planes: 27 to 35 us (one CTA with two barriers per elimination step:
// 141 to 145 us; the whole leaf in one warp's registers, 64 columns per step: 50 us).
constexpr int LCL = 8;                 // CTAs per leaf; columns of the inverse per CTA
constexpr int LTH = 256;               // threads: 2 entries of the CTA's 64 x 8 each
constexpr int LPW = 8;                 // panel width

// In-place Gauss-Jordan inverse of X (64 x 64, rows and columns from n on zero) by the CTA, rows
// never moved: pivot row piv[k] of step k keeps its place, so that the result's
// row piv[k] belongs to unknown k and its column k to equation piv[k].  False if
// a pivot column is zero (to within 64 subnormal units).
__device__ __forceinline__ bool leaf_gj(float (*X)[CMAX + 1], int n, float (*xq)[CMAX], int* piv,
                                        int* step, int* s_ok) {
  const int tid = threadIdx.x, lane = tid & 31;
  constexpr int NC = CMAX / (LTH / 64);   // columns of a thread's row in the update
  const int i = tid & 63, c0 = (tid >> 6) * NC;
  unsigned used = 0;                   // warp 0: bit 0 row lane, bit 1 row lane + 32
  if (tid == 0) *s_ok = 1;
  if (tid < CMAX) step[tid] = -1;      // the step whose pivot a row was
  __syncthreads();
  for (int kb = 0; kb < n; kb += LPW) {
    const int kw = min(LPW, n - kb);
    if (tid < 32) {
      float x0[LPW], x1[LPW], s0 = 1.f, s1 = 1.f;
#pragma unroll
      for (int c = 0; c < LPW; ++c) { x0[c] = X[lane][kb + c]; x1[c] = X[lane + 32][kb + c]; }
#pragma unroll
      for (int t = 0; t < LPW; ++t) {
        if (t < kw) {
          // the largest remaining |entry| of column kb + t, its row in the six low
          // bits (entries that agree to 2^-17 count as equal: the lowest row)
          const unsigned b0 = (used & 1u) ? 0u : ((__float_as_uint(fabsf(x0[t])) & ~63u) | (63u - lane));
          const unsigned b1 = (used & 2u) ? 0u : ((__float_as_uint(fabsf(x1[t])) & ~63u) | (31u - lane));
          const unsigned best = __reduce_max_sync(0xffffffffu, max(b0, b1));
          const int q = 63 - (int)(best & 63u);
          if ((best & ~63u) == 0u && lane == 0) *s_ok = 0;
          const bool hi = q >= 32;
          float v[LPW];
#pragma unroll
          for (int c = 0; c < LPW; ++c) v[c] = __shfl_sync(0xffffffffu, hi ? x1[c] : x0[c], q & 31);
          // (the pivot row is scaled when the panel is done: until then its entries,
          // the multipliers it is updated with included, are 1 / s times their value)
          const float pinv = 1.f / v[t];
          const bool p0 = lane == q, p1 = lane + 32 == q;
          used |= (p0 ? 1u : 0u) | (p1 ? 2u : 0u);
          const float f0 = p0 ? 0.f : x0[t] * pinv, f1 = p1 ? 0.f : x1[t] * pinv;
          s0 = p0 ? pinv : s0;
          s1 = p1 ? pinv : s1;
#pragma unroll
          for (int c = 0; c < LPW; ++c)
            if (c != t) {
              x0[c] = fmaf(-f0, v[c], x0[c]);
              x1[c] = fmaf(-f1, v[c], x1[c]);
            }
          x0[t] = p0 ? 1.f : -f0;
          x1[t] = p1 ? 1.f : -f1;
          if (lane == 0) { piv[kb + t] = q; step[q] = kb + t; }
        }
      }
#pragma unroll
      for (int c = 0; c < LPW; ++c)
        if (c < kw) { X[lane][kb + c] = x0[c] * s0; X[lane + 32][kb + c] = x1[c] * s1; }
    }
    __syncthreads();
    if (!*s_ok) return false;
    // the pivot rows' old entries, then X[i][j] <- (i not a pivot row) X[i][j] +
    // sum_t X[i][kb + t] xq[t][j] for the columns outside the panel
    float pr[LPW], y[NC];
    const bool pivot = step[i] >= kb;
#pragma unroll
    for (int t = 0; t < LPW; ++t) pr[t] = t < kw ? X[i][kb + t] : 0.f;
#pragma unroll
    for (int u = 0; u < NC; ++u) y[u] = pivot ? 0.f : X[i][c0 + u];
    for (int e = tid; e < LPW * CMAX; e += LTH)
      xq[e >> 6][e & 63] = (e >> 6) < kw ? X[piv[kb + (e >> 6)]][e & 63] : 0.f;
    __syncthreads();
#pragma unroll
    for (int t = 0; t < LPW; ++t)
#pragma unroll
      for (int u = 0; u < NC; u += 4) {
        const float4 v = *reinterpret_cast<const float4*>(&xq[t][c0 + u]);
        y[u] = fmaf(pr[t], v.x, y[u]);
        y[u + 1] = fmaf(pr[t], v.y, y[u + 1]);
        y[u + 2] = fmaf(pr[t], v.z, y[u + 2]);
        y[u + 3] = fmaf(pr[t], v.w, y[u + 3]);
      }
#pragma unroll
    for (int u = 0; u < NC; ++u)
      if (c0 + u < kb || c0 + u >= kb + LPW) X[i][c0 + u] = y[u];
    __syncthreads();
  }
  return true;
}

__global__ void __cluster_dims__(LCL, 1, 1) __launch_bounds__(LTH)
    k_leaf_inv_f(float* const* __restrict__ dense, int64_t off, int n, int* err,
                 double* __restrict__ flops, unsigned long long* __restrict__ fallbacks) {
  static_assert(CMAX == 64 && LCL * 8 == CMAX && LTH == 4 * CMAX, "64 x 64 leaves");
  float* Ap = dense[blockIdx.x / LCL];
  if (!Ap) return;   // the whole cluster
  Ap += off;
  cg::cluster_group cl = cg::this_cluster();
  cl.barrier_arrive();   // (this CTA has started: the others may write its s_state)
  const int rank = (int)cl.block_rank();
  // A and X0 together hold the FP64 fallback's matrix
  __shared__ __align__(16) float lsm[2 * CMAX * (CMAX + 1)];
  float (*A)[CMAX + 1] = reinterpret_cast<float (*)[CMAX + 1]>(lsm);
  float (*X0)[CMAX + 1] = reinterpret_cast<float (*)[CMAX + 1]>(lsm + CMAX * (CMAX + 1));
  __shared__ __align__(16) float Xc[CMAX][8], Rc[CMAX][8];
  float (*xq)[CMAX] = reinterpret_cast<float (*)[CMAX]>(&Rc[0][0]);   // elimination only
  __shared__ int piv[CMAX], step[CMAX];
  __shared__ int s_ok;
  __shared__ float red8[LTH / 32];
  __shared__ float s_state[LCL][2];   // per column group: 1 if it needs the fallback; largest entry
  const int tid = threadIdx.x;
  const int i = tid & 63, jl = 2 * (tid >> 6), j0 = 8 * rank + jl;
  float amax = 0.f;
  {
    float v[CMAX / 4];
#pragma unroll
    for (int q = 0; q < CMAX / 4; ++q) {
      const int j = (tid >> 6) + 4 * q;
      v[q] = (i < n && j < n) ? Ap[i + (int64_t)j * n] : 0.f;
    }
#pragma unroll
    for (int q = 0; q < CMAX / 4; ++q) {
      A[i][(tid >> 6) + 4 * q] = v[q];
      X0[i][(tid >> 6) + 4 * q] = v[q];
      amax = fmaxf(amax, fabsf(v[q]));
    }
  }
  amax = block_absmaxf<LTH>(amax, red8);
  // 1. the float elimination; its result in natural order
  bool fallback = !leaf_gj(X0, n, xq, piv, step, &s_ok), done = false;
  int steps = 0;
  float x[2] = {0.f, 0.f};
  float xmax = 0.f;
  if (!fallback) {
    float v[CMAX / 4];
    const int row = step[i];
#pragma unroll
    for (int q = 0; q < CMAX / 4; ++q) v[q] = X0[i][(tid >> 6) + 4 * q];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < CMAX / 4; ++q) {
      const int j = (tid >> 6) + 4 * q;
      if (i < n && j < n) X0[row][piv[j]] = v[q];
      const float w = fabsf(v[q]);
      if (i < n && j < n) xmax = (w <= 3.0e38f) ? fmaxf(xmax, w) : INFINITY;
    }
    xmax = block_absmaxf<LTH>(xmax, red8);
    if (!(xmax <= 3.0e38f)) fallback = true;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      x[q] = (i < n && j0 + q < n) ? X0[i][j0 + q] : 0.f;
      Xc[i][jl + q] = x[q];
    }
    __syncthreads();
  }
  // 2. refinement of this CTA's columns (rows and columns beyond n are zero)
  float dprev = INFINITY;
  for (int it = 0; it < 8 && !done && !fallback; ++it) {
    ++steps;
    float sh[2] = {0.f, 0.f}, sl[2] = {0.f, 0.f};
#pragma unroll 4
    for (int l = 0; l < n; ++l) {
      const float a = A[i][l];
      const float2 v = *reinterpret_cast<const float2*>(&Xc[l][jl]);
      ff_fma(sh[0], sl[0], a, v.x);
      ff_fma(sh[1], sl[1], a, v.y);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
      Rc[i][jl + q] = (i < n && j0 + q < n) ? ((i == j0 + q ? 1.f : 0.f) - sh[q]) - sl[q] : 0.f;
    __syncthreads();
    float d[2] = {0.f, 0.f};
#pragma unroll 8
    for (int l = 0; l < n; ++l) {
      const float a = X0[i][l];
      const float2 v = *reinterpret_cast<const float2*>(&Rc[l][jl]);
      d[0] = fmaf(a, v.x, d[0]);
      d[1] = fmaf(a, v.y, d[1]);
    }
    float dmax = 0.f;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      dmax = (fabsf(d[q]) <= 3.0e38f) ? fmaxf(dmax, fabsf(d[q])) : INFINITY;
      x[q] += d[q];
      Xc[i][jl + q] = x[q];
    }
    dmax = block_absmaxf<LTH>(dmax, red8);
    if (!(dmax <= 3.0e38f)) fallback = true;                  // non-finite
    else if (dmax <= 2.4e-7f * xmax) done = true;
    else if (dmax > 0.5f * dprev) fallback = true;            // not contracting
    dprev = dmax;
  }
  if (!done) fallback = true;
  xmax = 0.f;
#pragma unroll
  for (int q = 0; q < 2; ++q) xmax = (fabsf(x[q]) <= 3.0e38f) ? fmaxf(xmax, fabsf(x[q])) : INFINITY;
  xmax = block_absmaxf<LTH>(xmax, red8);
  cl.barrier_wait();
  if (tid < LCL) {   // to every CTA of the cluster
    float* st = cl.map_shared_rank(&s_state[rank][0], tid);
    st[0] = fallback ? 1.f : 0.f;
    st[1] = xmax;
  }
  cl.sync();   // every CTA has read the leaf and knows all columns' outcome
  fallback = false;
  for (int c = 0; c < LCL; ++c) {
    fallback = fallback || s_state[c][0] != 0.f || !(s_state[c][1] <= 3.0e38f);
    xmax = fmaxf(xmax, s_state[c][1]);
  }
  if (!fallback) {
    if (!((double)amax * (double)xmax <= leaf_growth_max<float>())) {
      if (rank == 0 && tid == 0) atomicOr(err, ERR_GROWTH);
      return;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
      if (i < n && j0 + q < n) Ap[i + (int64_t)(j0 + q) * n] = x[q];
    if (flops && rank == 0 && tid == 0) atomicAdd(flops, 2.0 * n * n * n * (1 + 2 * steps));
    return;
  }
  // 3. FP64 elimination of the stored leaf (untouched so far)
  if (rank != 0) return;
  if (fallbacks && tid == 0) atomicAdd(fallbacks, 1ull);
  leaf_inv_fp64<float, LTH>(Ap, n, reinterpret_cast<double (*)[CMAX + 1]>(lsm), err, flops);
}

// Leaf inverse of FP64 storage: the same elimination (rows never moved, panels of 8
// columns) in FP64.  The 64^3 multiply-adds alone take one SM's FP64 pipe 63 us
// (two lanes per clock), so a cluster of LCL CTAs shares a leaf by columns: the
// owner of a panel eliminates it in one warp's registers and pushes it to every CTA, and
// after one cluster barrier each updates its own 8 columns.  64 x 64 leaf: 123 us
// against 219 us in one CTA.
__global__ void __cluster_dims__(LCL, 1, 1) __launch_bounds__(128)
    k_leaf_inv_d(double* const* __restrict__ dense, int64_t off, int n, int* err,
                 double* __restrict__ flops) {
  constexpr int TH = 128;
  double* Ap = dense[blockIdx.x / LCL];
  if (!Ap) return;   // the whole cluster
  Ap += off;
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank();
  __shared__ double X[CMAX][LPW + 1];            // this CTA's columns
  __shared__ double Pn[2][CMAX][LPW + 1];        // the panel, by parity
  __shared__ double xq[LPW][LPW];                // the pivot rows' old entries of X
  __shared__ int piv[CMAX], step[CMAX];          // row of each step's pivot; step of each row
  __shared__ int s_ok[2];
  __shared__ double s_max[LCL][2];               // per CTA: largest entry of A, of the inverse
  __shared__ double red8[TH / 32];
  const int tid = threadIdx.x, lane = tid & 31;
  const int i = tid & 63, jh = 4 * (tid >> 6), c0 = LPW * rank;
  // No CTA writes into another's shared memory before that one has started and has set
  // its own step[]: the arrival follows that, and the wait hides behind the loads.
  if (tid < CMAX) step[tid] = -1;
  cl.barrier_arrive();
  double amax = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = c0 + jh + q;
    const double v = (i < n && j < n) ? Ap[i + (int64_t)j * n] : 0.0;
    X[i][jh + q] = v;
    amax = fmax(amax, fabs(v));
  }
  amax = block_absmax<TH>(amax, red8);
  cl.barrier_wait();
  unsigned used = 0;   // warp 0: rows lane, lane + 32 that have been pivots
  int buf = 0;
  for (int kb = 0; kb < n; kb += LPW, buf ^= 1) {
    const int kw = min(LPW, n - kb);
    if (rank == kb / LPW) {
      if (tid < 32) {
        // (rows that were pivots of earlier panels)
        used = (step[lane] >= 0 ? 1u : 0u) | (step[lane + 32] >= 0 ? 2u : 0u);
        double x0[LPW], x1[LPW];
        int pv[LPW], ok = 1;
#pragma unroll
        for (int c = 0; c < LPW; ++c) { x0[c] = X[lane][c]; x1[c] = X[lane + 32][c]; }
#pragma unroll
        for (int t = 0; t < LPW; ++t) {
          pv[t] = -1;
          if (t < kw) {
            // the largest remaining |entry| by its upper bits (entries that agree to
            // 2^-14 count as equal: the lowest row)
            const unsigned h0 = (unsigned)__double2hiint(fabs(x0[t]));
            const unsigned h1 = (unsigned)__double2hiint(fabs(x1[t]));
            const unsigned b0 = (used & 1u) ? 0u : ((h0 & ~63u) | (63u - lane));
            const unsigned b1 = (used & 2u) ? 0u : ((h1 & ~63u) | (31u - lane));
            const unsigned best = __reduce_max_sync(0xffffffffu, max(b0, b1));
            const int q = 63 - (int)(best & 63u);
            if ((best & ~63u) == 0u) ok = 0;
            const bool hi = q >= 32;
            double v[LPW];
#pragma unroll
            for (int c = 0; c < LPW; ++c) v[c] = __shfl_sync(0xffffffffu, hi ? x1[c] : x0[c], q & 31);
            const double pinv = 1.0 / v[t];
            const bool p0 = lane == q, p1 = lane + 32 == q;
            used |= (p0 ? 1u : 0u) | (p1 ? 2u : 0u);
            pv[t] = q;
            const double f0 = x0[t], f1 = x1[t];
#pragma unroll
            for (int c = 0; c < LPW; ++c) {
              const double w = c == t ? pinv : v[c] * pinv;
              x0[c] = p0 ? w : (c == t ? -f0 * pinv : fma(-f0, w, x0[c]));
              x1[c] = p1 ? w : (c == t ? -f1 * pinv : fma(-f1, w, x1[c]));
            }
          }
        }
#pragma unroll
        for (int c = 0; c < LPW; ++c) {
          X[lane][c] = x0[c];
          X[lane + 32][c] = x1[c];
          Pn[buf][lane][c] = x0[c];
          Pn[buf][lane + 32][c] = x1[c];
        }
        if (lane < LCL) {   // pivots and outcome to every CTA
          int* dp = cl.map_shared_rank(piv, lane);
          int* ds = cl.map_shared_rank(step, lane);
          int* dk = cl.map_shared_rank(s_ok, lane);
#pragma unroll
          for (int t = 0; t < LPW; ++t)
            if (pv[t] >= 0) {
              dp[kb + t] = pv[t];
              ds[pv[t]] = kb + t;
            }
          dk[buf] = ok;
        }
      }
      __syncthreads();
      for (int c = 0; c < LCL; ++c) {
        if (c == rank) continue;
        double* d = cl.map_shared_rank(&Pn[buf][0][0], c);
        for (int e = tid; e < CMAX * (LPW + 1); e += TH) d[e] = (&Pn[buf][0][0])[e];
      }
    }
    cl.sync();   // the panel is everywhere; everyone is done with the one before
    if (!s_ok[buf]) {
      if (rank == 0 && tid == 0) atomicOr(err, ERR_PIVOT);
      cl.sync();
      return;
    }
    if (rank != kb / LPW) {
      if (tid < LPW * LPW)
        xq[tid >> 3][tid & 7] = (tid >> 3) < kw ? X[piv[kb + (tid >> 3)]][tid & 7] : 0.0;
      __syncthreads();
      const int st = step[i];
      const bool pivot = st >= kb && st < kb + LPW;
      double y[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) y[q] = pivot ? 0.0 : X[i][jh + q];
#pragma unroll
      for (int t = 0; t < LPW; ++t) {
        const double pr = t < kw ? Pn[buf][i][t] : 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q) y[q] = fma(pr, xq[t][jh + q], y[q]);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) X[i][jh + q] = y[q];
    }
    __syncthreads();
  }
  // pivot growth of the computed inverse (a NaN or Inf entry fails too)
  double xmax = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (i < n && c0 + jh + q < n) {
      const double v = fabs(X[i][jh + q]);
      xmax = (v <= 1.7976931348623157e308) ? fmax(xmax, v) : INFINITY;
    }
  xmax = block_absmax<TH>(xmax, red8);
  if (tid < LCL) {
    double* d = cl.map_shared_rank(&s_max[rank][0], tid);
    d[0] = amax;
    d[1] = xmax;
  }
  cl.sync();
  for (int c = 0; c < LCL; ++c) {
    amax = fmax(amax, s_max[c][0]);
    xmax = fmax(xmax, s_max[c][1]);
  }
  if (!(amax * xmax <= leaf_growth_max<double>())) {
    if (rank == 0 && tid == 0) atomicOr(err, ERR_GROWTH);
    return;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = c0 + jh + q;
    if (i < n && c < n) Ap[step[i] + (int64_t)piv[c] * n] = X[i][jh + q];
  }
  if (flops && rank == 0 && tid == 0) atomicAdd(flops, 2.0 * n * n * n);
}

// out = sgn * diag(r) X diag(c): dense part
template <typename T>
__global__ void k_hscale_dense(T* const* __restrict__ od, T* const* __restrict__ xd,
                               const double* const* __restrict__ rsc,
                               const double* const* __restrict__ csc,
                               const int* __restrict__ dinfo, int lsz, double sgn) {
  const int d = blockIdx.x, p = blockIdx.y;
  T* o = od[p];
  const T* x = xd[p];
  const double* r = rsc[p];
  const double* c = csc[p];
  if (!o || !x) return;
  const int t0 = dinfo[2 * d], s0 = dinfo[2 * d + 1];
  const int64_t off = (int64_t)d * lsz * lsz;
  for (int e = threadIdx.x; e < lsz * lsz; e += blockDim.x) {
    int i = e % lsz, j = e / lsz;
    o[off + e] = (T)(sgn * r[t0 + i] * (double)x[off + e] * c[s0 + j]);
  }
}

template <typename T>
__global__ void k_hscale_lr(T* const* __restrict__ oU, T* const* __restrict__ oV,
                            int* const* __restrict__ orank, T* const* __restrict__ xU,
                            T* const* __restrict__ xV, const int* const* __restrict__ xrank,
                            const double* const* __restrict__ rsc,
                            const double* const* __restrict__ csc, const int* __restrict__ linfo,
                            const int64_t* __restrict__ row0, const int64_t* __restrict__ col0,
                            int kc, double sgn) {
  const int l = blockIdx.x, p = blockIdx.y;
  if (!oU[p] || !xU[p]) return;
  const int k = xrank[p][l];
  const int m = linfo[4 * l], n = linfo[4 * l + 1], t0 = linfo[4 * l + 2], s0 = linfo[4 * l + 3];
  const double* r = rsc[p];
  const double* c = csc[p];
  T* u = oU[p] + row0[l] * kc;
  T* v = oV[p] + col0[l] * kc;
  const T* xu = xU[p] + row0[l] * kc;
  const T* xv = xV[p] + col0[l] * kc;
  for (int e = threadIdx.x; e < m * k; e += blockDim.x) {
    int i = e % m;
    u[e] = (T)(sgn * r[t0 + i] * (double)xu[e]);
  }
  for (int e = threadIdx.x; e < n * k; e += blockDim.x) {
    int j = e % n;
    v[e] = (T)(c[s0 + j] * (double)xv[e]);
  }
  if (threadIdx.x == 0) orank[p][l] = k;
}

// D_k dense leaves from the stencil: leaf rows/cols in cluster order.
template <typename T>
__global__ void k_plane_dense(const double* __restrict__ coef, int n, const int* __restrict__ planes,
                              T* const* __restrict__ dense, const int* __restrict__ perm,
                              const int* __restrict__ dinfo, int lsz) {
  const int d = blockIdx.x, pi = blockIdx.y;
  T* o = dense[pi];
  if (!o) return;
  const int64_t N = (int64_t)n * n * n;
  const int64_t base = (int64_t)planes[pi] * n * n;
  const int t0 = dinfo[2 * d], s0 = dinfo[2 * d + 1];
  o += (int64_t)d * lsz * lsz;
  for (int e = threadIdx.x; e < lsz * lsz; e += blockDim.x) {
    int i = e % lsz, j = e / lsz;
    int a = perm[t0 + i], b = perm[s0 + j];
    int ax = a % n;
    double v = 0.0;
    if (a == b) v = coef[0 * N + base + a];
    else if (b == a - 1 && ax > 0) v = coef[1 * N + base + a];
    else if (b == a + 1 && ax < n - 1) v = coef[2 * N + base + a];
    else if (b == a - n) v = coef[3 * N + base + a];
    else if (b == a + n) v = coef[4 * N + base + a];
    o[e] = (T)v;
  }
}

// exact sparse low-rank factors of admissible blocks of D_k: one rank-one
// term per stencil coupling (row i, col j, direction d)
template <typename T>
__global__ void k_plane_lr(const double* __restrict__ coef, int n, const int* __restrict__ planes,
                           T* const* __restrict__ U, T* const* __restrict__ V,
                           int* const* __restrict__ rank, const int* __restrict__ perm,
                           const int* __restrict__ cpl, const int* __restrict__ cptr,
                           const int* __restrict__ linfo, const int64_t* __restrict__ row0,
                           const int64_t* __restrict__ col0, int kc) {
  const int l = blockIdx.x, pi = blockIdx.y;
  if (!U[pi]) return;
  const int64_t N = (int64_t)n * n * n;
  const int64_t base = (int64_t)planes[pi] * n * n;
  const int m = linfo[4 * l], nn = linfo[4 * l + 1], t0 = linfo[4 * l + 2];
  const int c0 = cptr[l], c1 = cptr[l + 1];
  const int k = c1 - c0;
  T* u = U[pi] + row0[l] * kc;
  T* v = V[pi] + col0[l] * kc;
  for (int e = threadIdx.x; e < m * k; e += blockDim.x) u[e] = (T)0;
  for (int e = threadIdx.x; e < nn * k; e += blockDim.x) v[e] = (T)0;
  __syncthreads();
  for (int q = threadIdx.x; q < k; q += blockDim.x) {
    int i = cpl[3 * (c0 + q)], j = cpl[3 * (c0 + q) + 1], dir = cpl[3 * (c0 + q) + 2];
    int a = perm[t0 + i];
    u[i + (int64_t)q * m] = (T)coef[(int64_t)dir * N + base + a];
    v[j + (int64_t)q * nn] = (T)1;
  }
  if (threadIdx.x == 0) rank[pi][l] = k;
}

}  // namespace


template <typename T>
void launch_pchol(const Plan& pl, int tbeg, int tend, bool truncate, double tau, T* const* d_tab,
                  int* const* d_rtab, int P, cudaStream_t st, unsigned long long* d_sketch_stat,
                  double* d_fl) {
  int nt = tend - tbeg;
  if (nt <= 0 || P <= 0) return;
  const size_t smem = 2 * CMAX * (CMAX + 1) * sizeof(double);
  ACR_CUDA(cudaFuncSetAttribute(k_pchol<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  ACR_CUDA(cudaFuncSetAttribute(k_pchol_warp<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)PCHOL_WARP_SMEM));
  for (int t0 = 0; t0 < nt; t0 += 65535 * PW) {
    const int cnt = std::min(65535 * PW, nt - t0);
    dim3 grid((cnt + PW - 1) / PW, P);
    k_pchol_warp<T><<<grid, 32 * PW, PCHOL_WARP_SMEM, st>>>(
        (const TInfo*)pl.d_targets, tbeg + t0, tbeg + t0 + cnt, truncate, tau, d_tab, d_rtab, P,
        3 * pl.nroles, pl.nroles, (const StackDim*)pl.d_stack, d_sketch_stat, d_fl);
    ACR_LAUNCHED(1);
  }
  // Grams wider than a warp's (none when every sketch is at most 32 wide:
  // the second pass's basis is never wider than its sketch)
  if (pl.max_p <= PCHOL_WARP_MAX) return;
  for (int t0 = 0; t0 < nt; t0 += 65535) {
    dim3 grid(std::min(65535, nt - t0), P);
    k_pchol<T><<<grid, NT, smem, st>>>((const TInfo*)pl.d_targets, tbeg + t0, truncate, tau, d_tab,
                                    d_rtab, P, 3 * pl.nroles, pl.nroles,
                                    (const StackDim*)pl.d_stack, d_sketch_stat, d_fl);
    ACR_LAUNCHED(1);
  }
}

template <typename T>
void launch_leaf_inv(T* const* d_dense, int64_t off, int lsz, int P, int* d_err, cudaStream_t st,
                     double* d_fl, unsigned long long* d_fallbacks) {
  if (P <= 0) return;
  if constexpr (std::is_same<T, float>::value) {
    k_leaf_inv_f<<<P * LCL, LTH, 0, st>>>(d_dense, off, lsz, d_err, d_fl, d_fallbacks);
  } else {
    k_leaf_inv_d<<<P * LCL, 128, 0, st>>>(d_dense, off, lsz, d_err, d_fl);
  }
  ACR_LAUNCHED(1);
}

template <typename T>
void launch_hscale(const StructDev& sd, T* const* out_dense, T* const* out_U, T* const* out_V,
                   int* const* out_rank, T* const* x_dense, T* const* x_U, T* const* x_V,
                   const int* const* x_rank, const double* const* rowscale,
                   const double* const* colscale, double sgn, int kc, int P, cudaStream_t st) {
  if (P <= 0) return;
  if (sd.nd > 0)
    k_hscale_dense<T><<<dim3(sd.nd, P), 256, 0, st>>>(out_dense, x_dense, rowscale, colscale,
                                                      sd.dinfo, sd.lsz, sgn);
  if (sd.nl > 0)
    k_hscale_lr<T><<<dim3(sd.nl, P), 256, 0, st>>>(out_U, out_V, out_rank, x_U, x_V, x_rank,
                                                   rowscale, colscale, sd.linfo, sd.row0,
                                                   sd.col0, kc, sgn);
  ACR_LAUNCHED((sd.nd > 0) + (sd.nl > 0));
}

template <typename T>
void launch_plane_to_h(const StructDev& sd, const double* coef, int n, const int* d_planes, int P,
                       T* const* dense, T* const* U, T* const* V, int* const* rank, int kc,
                       cudaStream_t st) {
  if (P <= 0) return;
  if (sd.nd > 0)
    k_plane_dense<T><<<dim3(sd.nd, P), 256, 0, st>>>(coef, n, d_planes, dense, sd.perm, sd.dinfo,
                                                     sd.lsz);
  if (sd.nl > 0)
    k_plane_lr<T><<<dim3(sd.nl, P), 256, 0, st>>>(coef, n, d_planes, U, V, rank, sd.perm, sd.cpl,
                                                  sd.cptr, sd.linfo, sd.row0, sd.col0, kc);
  ACR_LAUNCHED((sd.nd > 0) + (sd.nl > 0));
}

template void launch_pchol<double>(const Plan&, int, int, bool, double, double* const*,
                                   int* const*, int, cudaStream_t, unsigned long long*, double*);
#define ACR_INST(T)                                                                              \
  template void launch_leaf_inv<T>(T* const*, int64_t, int, int, int*, cudaStream_t, double*,     \
                                   unsigned long long*);                                         \
  template void launch_hscale<T>(const StructDev&, T* const*, T* const*, T* const*, int* const*, \
                                 T* const*, T* const*, T* const*, const int* const*,             \
                                 const double* const*, const double* const*, double, int, int,   \
                                 cudaStream_t);                                                  \
  template void launch_plane_to_h<T>(const StructDev&, const double*, int, const int*, int,      \
                                     T* const*, T* const*, T* const*, int* const*, int,          \
                                     cudaStream_t);

ACR_INST(double)
ACR_INST(float)

}  // namespace acr
