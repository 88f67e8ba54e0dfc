// The preconditioner apply for 32 right-hand sides at once (float and bfloat16
// factors): the batched H-matrix-vector product (Sec. 4.1 substitution, "solely
// based on H-matrix-vector multiplications") as an H-matrix x matrix product, each
// stored factor entry read once for all 32 vectors.  Three launches per product:
//  * k_proj32 : the FP64 vectors' chunk as floats (once, for every product that
//               meets it), and per low-rank leaf the partial V_l^T X over each
//               leaf-size chunk of its columns (transposed: U_l^T X);
//  * k_tsum32 : the partial projections of a leaf (FP64) summed, as floats;
//  * k_rows32 : per row chunk c, Y[c] = beta Y[c] + alpha (sum of dense leaves
//               times X + sum of U_l[rows of c] TV_l).
// Products and sums are float over runs of at most 8 products, which enter
// compensated float pairs, at every leaf size.
//
// The products are 64 x K x 32 with K of a few hundred to a thousand: CUDA-core
// work of 32 multiply-adds per loaded entry, bound by issue slots (2.6 of 4 per clock, FMA
// pipe 48%: the compensated additions take nearly as many as the products) and shared
// memory at half its rate (two 16-byte vectors per 16 products; 8 x 4 outputs per thread
// with the contraction split over two halves of the CTA read less but held 128 registers
// and were slower: 104 against 90 us with sums of 64).  A tcgen05 form (split TF32, M = 128 with hi and lo rows stacked) spent its
// time staging -- both operands through registers for the split, in core-matrix
// order, the vectors converted from FP64 again for every chunk that reads them --
// and took 236 us per launch on average for the n = 64 Helmholtz recipe (4096
// x 32 per plane, up to 32 planes), its projections 94 us.  32 vectors at n = 64: 4.5 ms
// per apply against 8.4 ms.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "acr_device.h"
#include "acr_internal.h"

namespace acr {

namespace {

constexpr int R = 32;                            // right-hand sides per pass
constexpr int MAXLQ = 256;                       // low-rank leaves per chunk
// Products in a float sum.  The rounding an apply adds (the relative defect of its
// linearity, random vectors) is 0.72e-7 to 0.76e-7 with 8 at 25- to 64-point leaves, where
// the groups of 8 right-hand sides have 0.66e-7 to 0.94e-7; with 16 it is 1.0e-7, with 64
// 2.0e-7 (the tensor form had 2.7e-7).  Per apply at n = 64: 4.5 ms (64: 3.8 ms);
// n = 48: 2.9 ms against 10.4 ms in groups of 8, n = 80: 8.7 ms against 34 ms.
constexpr int RUN = 8;
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ float ldf(float v) { return v; }
__device__ __forceinline__ float ldf(__nv_bfloat16 v) { return __bfloat162float(v); }

// s + c += v, compensated (TwoSum)
__device__ __forceinline__ void pair_add(float& s, float& c, float v) {
  const float t = s + v, bp = t - s;
  c += (s - (t - bp)) + (v - bp);
  s = t;
}

// cum[0 .. nq] = exclusive sums of cum[1 .. nq] (a CTA's leaves; one warp)
__device__ __forceinline__ void warp_cumulate(int* cum, int nq) {
  const int lane = threadIdx.x & 31;
  int base = 0;
  if (lane == 0) cum[0] = 0;
  for (int q0 = 0; q0 < nq; q0 += 32) {
    int v = q0 + lane < nq ? cum[q0 + lane + 1] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(FULL, v, o);
      if (lane >= o) v += u;
    }
    if (q0 + lane < nq) cum[q0 + lane + 1] = base + v;
    base += __shfl_sync(FULL, v, 31);
  }
}
// the q with cum[q] <= t < cum[q + 1]
__device__ __forceinline__ int find_q(const int* cum, int nq, int t) {
  int lo = 0, hi = nq;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (cum[mid] <= t) lo = mid;
    else hi = mid;
  }
  return lo;
}

// A warp takes 8 columns of the chunk's low-rank leaves at a time (of one leaf or
// several): 64 rows of them pass through its shared slice, and lane rr
// accumulates the 8 products with right-hand side rr.
template <typename T>
__global__ void __launch_bounds__(256) k_proj32(MatvecDev mv, T* const* __restrict__ U,
                                                T* const* __restrict__ V,
                                                const int* const* __restrict__ rank,
                                                const double* const* __restrict__ x,
                                                double* __restrict__ tv, float* __restrict__ xf,
                                                bool trans, int64_t vs) {
  chain_begin();
  __shared__ float xs[64][R + 1];
  __shared__ __align__(16) float zs[8][64][8];
  __shared__ int64_t s_off[MAXLQ];
  __shared__ int s_ld[MAXLQ], s_seg[MAXLQ], s_cum[MAXLQ + 1];
  const int c = blockIdx.x, p = blockIdx.y;
  const T* Fb = trans ? U[p] : V[p];
  const double* xp = x[p];
  if (!Fb || !xp) return;
  const int lsz = mv.lsz, kc = mv.kc, tid = threadIdx.x;
  const int* ptr = trans ? mv.l_ptr : mv.lt_ptr;
  const int* lf = trans ? mv.l_leaf : mv.lt_leaf;
  const int* lo = trans ? mv.l_rowoff : mv.lt_coloff;
  const int* sptr = trans ? mv.segt_ptr : mv.seg_ptr;
  const int nseg = trans ? mv.nsegt : mv.nseg;
  const int q0 = ptr[c], nq = min(ptr[c + 1] - q0, MAXLQ);
  for (int e = tid; e < R * lsz; e += 256) {
    const int rr = e / lsz, i = e - rr * lsz;
    xs[i][rr] = (float)xp[rr * vs + (int64_t)c * lsz + i];
  }
  for (int q = tid; q < nq; q += 256) {
    const int l = lf[q0 + q];
    s_cum[q + 1] = rank[p][l];
    s_ld[q] = trans ? mv.lr_m[l] : mv.lr_n[l];
    s_off[q] = (trans ? mv.lr_row0[l] : mv.lr_col0[l]) * kc + lo[q0 + q];
    s_seg[q] = sptr[l] + lo[q0 + q] / lsz;
  }
  __syncthreads();
  if (tid < 32) warp_cumulate(s_cum, nq);
  float* xo = xf + ((int64_t)p * mv.nchunks + c) * lsz * R;
  for (int e = tid; e < R * lsz; e += 256) xo[e] = xs[e >> 5][e & 31];
  __syncthreads();
  const int warp = tid >> 5, lane = tid & 31;
  const int total = nq > 0 ? s_cum[nq] : 0;
  float (*z)[8] = zs[warp];
  for (int t0 = 8 * warp; t0 < total; t0 += 64) {
    // lane c < 8: column t0 + c
    const T* col = nullptr;
    int64_t out = 0;
    if (lane < 8 && t0 + lane < total) {
      const int q = find_q(s_cum, nq, t0 + lane), j = t0 + lane - s_cum[q];
      col = Fb + s_off[q] + (int64_t)j * s_ld[q];
      out = ((int64_t)p * nseg + s_seg[q]) * kc + j;
    }
    float v0[8], v1[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const T* ck = reinterpret_cast<const T*>(
          __shfl_sync(FULL, reinterpret_cast<unsigned long long>(col), k));
      v0[k] = (ck && lane < lsz) ? ldf(ck[lane]) : 0.f;
      v1[k] = (ck && lane + 32 < lsz) ? ldf(ck[lane + 32]) : 0.f;
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 8; k += 4) {
      *reinterpret_cast<float4*>(&z[lane][k]) = make_float4(v0[k], v0[k + 1], v0[k + 2], v0[k + 3]);
      *reinterpret_cast<float4*>(&z[lane + 32][k]) = make_float4(v1[k], v1[k + 1], v1[k + 2], v1[k + 3]);
    }
    __syncwarp();
    float s[8], cc[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) { s[k] = 0.f; cc[k] = 0.f; }
    for (int h = 0; h < lsz; h += RUN) {
      float a[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) a[k] = 0.f;
      const int rows = min(RUN, lsz - h);
#pragma unroll 8
      for (int i = 0; i < rows; ++i) {
        const float4 p0 = *reinterpret_cast<const float4*>(&z[h + i][0]);
        const float4 p1 = *reinterpret_cast<const float4*>(&z[h + i][4]);
        const float w = xs[h + i][lane];
        a[0] = fmaf(p0.x, w, a[0]); a[1] = fmaf(p0.y, w, a[1]);
        a[2] = fmaf(p0.z, w, a[2]); a[3] = fmaf(p0.w, w, a[3]);
        a[4] = fmaf(p1.x, w, a[4]); a[5] = fmaf(p1.y, w, a[5]);
        a[6] = fmaf(p1.z, w, a[6]); a[7] = fmaf(p1.w, w, a[7]);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) pair_add(s[k], cc[k], a[k]);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int64_t o = __shfl_sync(FULL, out, k);
      if (t0 + k < total) tv[o * R + lane] = (double)s[k] + (double)cc[k];
    }
  }
}

// One CTA per low-rank leaf: its segments' partial projections summed in order, 8
// columns at a time (16 lanes per column, two right-hand sides each).
__global__ void __launch_bounds__(128) k_tsum32(MatvecDev mv, const void* const* __restrict__ U,
                                                const int* const* __restrict__ rank,
                                                const double* const* __restrict__ x,
                                                const double* __restrict__ tv,
                                                float* __restrict__ tf, bool trans) {
  chain_begin();
  const int p = blockIdx.y, l = blockIdx.x, lane = threadIdx.x & 15;
  if (!U[p] || !x[p]) return;
  const int* sptr = trans ? mv.segt_ptr : mv.seg_ptr;
  const int nseg = trans ? mv.nsegt : mv.nseg;
  const int k = rank[p][l], s0 = sptr[l], s1 = sptr[l + 1];
  for (int j = threadIdx.x >> 4; j < k; j += 8) {
    double s[2] = {0.0, 0.0};
    const double2* src =
        reinterpret_cast<const double2*>(tv + (((int64_t)p * nseg + s0) * mv.kc + j) * R) + lane;
    const int64_t step = (int64_t)mv.kc * R / 2;
#pragma unroll 4
    for (int sg = s0; sg < s1; ++sg, src += step) {
      const double2 v = *src;
      s[0] += v.x;
      s[1] += v.y;
    }
    reinterpret_cast<float2*>(tf + (((int64_t)p * mv.nl + l) * mv.kc + j) * R)[lane] =
        make_float2((float)s[0], (float)s[1]);
  }
}

// 128 threads, 4 x 4 outputs each of the chunk's 64 x 32: chunks of up to 64
// contraction rows (a dense leaf, or the low-rank leaves' columns end to end) staged in
// shared memory, both operands read as 16-byte vectors; every chunk's float sums
// enter compensated pairs.
constexpr int WT = 128, ALD = 68, BLD = 36;

template <typename T>
__global__ void __launch_bounds__(WT, 4)
    k_rows32(MatvecDev mv, T* const* __restrict__ D, T* const* __restrict__ U,
             T* const* __restrict__ V, const int* const* __restrict__ rank,
             const double* const* __restrict__ x, double* const* __restrict__ y, double alpha,
             double beta, const float* __restrict__ xf, const float* __restrict__ tf, bool trans,
             int64_t vs) {
  chain_begin();
  __shared__ __align__(16) float As[64 * ALD];
  __shared__ __align__(16) float Bs[64 * BLD];
  __shared__ int64_t s_off[MAXLQ];
  __shared__ int s_ld[MAXLQ], s_leaf[MAXLQ], s_cum[MAXLQ + 1];
  __shared__ const T* ra[64];
  __shared__ const float* rb[64];
  const int c = blockIdx.x, p = blockIdx.y;
  double* yp = y[p];
  if (!yp) return;
  const bool have = D[p] != nullptr && x[p] != nullptr;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, lsz = mv.lsz, kc = mv.kc;
  const int* dptr = trans ? mv.dt_ptr : mv.d_ptr;
  const int* dleaf = trans ? mv.dt_leaf : mv.d_leaf;
  const int* dcol = trans ? mv.dt_row : mv.d_col;
  const int* lptr = trans ? mv.lt_ptr : mv.l_ptr;
  const int* lleaf = trans ? mv.lt_leaf : mv.l_leaf;
  const int d0 = dptr[c], nd = have ? dptr[c + 1] - d0 : 0;
  const int l0 = lptr[c], nlc = have ? min(lptr[c + 1] - l0, MAXLQ) : 0;
  for (int q = tid; q < nlc; q += WT) {
    const int l = lleaf[l0 + q];
    s_leaf[q] = l;
    s_cum[q + 1] = rank[p][l];
    s_ld[q] = trans ? mv.lr_n[l] : mv.lr_m[l];
    s_off[q] = trans ? mv.lr_col0[l] * kc + mv.lt_coloff[l0 + q]
                     : mv.lr_row0[l] * kc + mv.l_rowoff[l0 + q];
  }
  __syncthreads();
  if (warp == 0) warp_cumulate(s_cum, nlc);
  const int ty = tid >> 3, tx = tid & 7;
  float hi[4][4], lo[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) { hi[a][b] = 0.f; lo[a][b] = 0.f; }
  auto multiply = [&](int kf) {
    __syncthreads();
    for (int k0 = 0; k0 < kf; k0 += RUN) {
      float acc[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = 0.f;
      auto product = [&](int k) {
        const float4 a4 = *reinterpret_cast<const float4*>(As + k * ALD + 4 * ty);
        const float4 b4 = *reinterpret_cast<const float4*>(Bs + k * BLD + 4 * tx);
        const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
      };
      if (k0 + RUN <= kf) {
#pragma unroll
        for (int k = 0; k < RUN; ++k) product(k0 + k);
      } else {
        for (int k = k0; k < kf; ++k) product(k);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) pair_add(hi[u][v], lo[u][v], acc[u][v]);
    }
    __syncthreads();
  };
  const T* Dp = D[p];
  const float* xb = xf + (int64_t)p * mv.nchunks * lsz * R;
  for (int q = 0; q < nd; ++q) {
    const T* blk = Dp + (int64_t)dleaf[d0 + q] * lsz * lsz;
    const float* xq = xb + (int64_t)dcol[d0 + q] * R;
    float4 b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + WT * u;
      b[u] = (e >> 3) < lsz ? *reinterpret_cast<const float4*>(xq + 4 * e)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T a[16];
      if (!trans) {   // lanes along the rows
        const int i = tid & 63;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int l = (tid >> 6) + 2 * (16 * h + u);
          a[u] = (i < lsz && l < lsz) ? blk[i + l * lsz] : T(0.f);
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) As[((tid >> 6) + 2 * (16 * h + u)) * ALD + i] = ldf(a[u]);
      } else {        // 8 contraction rows x 4 output rows per warp and load
        const int l = 8 * (warp + 4 * h) + (lane >> 2);
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int i = 4 * u + (lane & 3);
          a[u] = (i < lsz && l < lsz) ? blk[l + i * lsz] : T(0.f);
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) As[l * ALD + 4 * u + (lane & 3)] = ldf(a[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + WT * u;
      *reinterpret_cast<float4*>(Bs + (e >> 3) * BLD + 4 * (e & 7)) = b[u];
    }
    multiply(lsz);
  }
  const int ktot = nlc > 0 ? s_cum[nlc] : 0;
  const T* Fp = trans ? V[p] : U[p];
  for (int c0 = 0; c0 < ktot; c0 += 64) {
    const int kf = min(64, ktot - c0);
    if (tid < kf) {
      const int q = find_q(s_cum, nlc, c0 + tid), j = c0 + tid - s_cum[q];
      ra[tid] = Fp + s_off[q] + (int64_t)j * s_ld[q];
      rb[tid] = tf + (((int64_t)p * mv.nl + s_leaf[q]) * kc + j) * R;
    }
    __syncthreads();
    float4 b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + WT * u;
      b[u] = (e >> 3) < kf ? *reinterpret_cast<const float4*>(rb[e >> 3] + 4 * (e & 7))
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int i = tid & 63;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      T a[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) {
        const int l = (tid >> 6) + 2 * (16 * h + u);
        a[u] = (i < lsz && l < kf) ? ra[l][i] : T(0.f);
      }
#pragma unroll
      for (int u = 0; u < 16; ++u) As[((tid >> 6) + 2 * (16 * h + u)) * ALD + i] = ldf(a[u]);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int e = tid + WT * u;
      *reinterpret_cast<float4*>(Bs + (e >> 3) * BLD + 4 * (e & 7)) = b[u];
    }
    multiply(kf);
  }
  // through shared memory, so that rows go out contiguously, 16 right-hand sides at a time
  double* out = reinterpret_cast<double*>(As);   // [right-hand side][row]
  for (int g = 0; g < 2; ++g) {
    __syncthreads();
    if ((tx >> 2) == g)
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int u = 0; u < 4; ++u)
          out[(4 * (tx & 3) + v) * 64 + 4 * ty + u] = (double)hi[u][v] + (double)lo[u][v];
    __syncthreads();
    for (int e = tid; e < 16 * 64; e += WT) {
      const int rr = 16 * g + (e >> 6), i = e & 63;
      if (i >= lsz) continue;
      double* yc = yp + (int64_t)rr * vs + (int64_t)c * lsz + i;
      const double old = (beta != 0.0) ? beta * *yc : 0.0;
      *yc = old + (have ? alpha * out[e] : 0.0);
    }
  }
}

}  // namespace

size_t wide_scratch_floats(const MatvecDev& mv, int P) {
  return (size_t)P * ((size_t)mv.nchunks * mv.lsz * R + (size_t)std::max(mv.nl, 1) * mv.kc * R);
}

template <typename T>
void launch_hmatvec_wide(const MatvecDev& mv, T* const* dense, T* const* U, T* const* V,
                         const int* const* rank, const double* const* x, double* const* y,
                         double alpha, double beta, bool trans, double* tv, float* work, int P,
                         int64_t vs, cudaStream_t st) {
  if (P <= 0) return;
  float* xf = work;
  float* tf = work + (size_t)P * mv.nchunks * mv.lsz * R;
  launch_chain(k_proj32<T>, dim3(mv.nchunks, P), 256, 0, st, mv, U, V, rank, x, tv, xf, trans, vs);
  if (mv.nl > 0)
    launch_chain(k_tsum32, dim3(mv.nl, P), 128, 0, st, mv, (const void* const*)(trans ? U : V),
                 rank, x, tv, tf, trans);
  launch_chain(k_rows32<T>, dim3(mv.nchunks, P), WT, 0, st, mv, dense, U, V, rank, x, y, alpha,
               beta, xf, tf, trans, vs);
  ACR_LAUNCHED(mv.nl > 0 ? 3 : 2);
}

template void launch_hmatvec_wide<float>(const MatvecDev&, float* const*, float* const*,
                                         float* const*, const int* const*, const double* const*,
                                         double* const*, double, double, bool, double*, float*,
                                         int, int64_t, cudaStream_t);
template void launch_hmatvec_wide<__nv_bfloat16>(const MatvecDev&, __nv_bfloat16* const*,
                                                 __nv_bfloat16* const*, __nv_bfloat16* const*,
                                                 const int* const*, const double* const*,
                                                 double* const*, double, double, bool, double*,
                                                 float*, int, int64_t, cudaStream_t);

}  // namespace acr
