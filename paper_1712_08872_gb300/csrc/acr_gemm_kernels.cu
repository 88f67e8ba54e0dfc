// Grouped small GEMMs of the setup plans (sm_103a, CUDA cores):
//  * k_gcat      -- one CTA per group, items K-concatenated in shared staging
//                   (the default of every stage that is no inner product);
//  * k_gbundle   -- factor stages: one CTA per bundle of groups that share
//                   their A operands;
//  * k_ggemm     -- an earlier staged form, one of the autotuner's shapes;
//  * k_gwarp     -- one warp per group (row panels of up to 64 rows);
//  * k_gdot, k_gdot_warp -- inner-product stages (both operands contiguous
//                   along the contraction);
//  * launch_ggemm -- the stage dispatcher (kernel shape per stage tag).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "acr_device.h"
#include "acr_internal.h"

namespace acr {

namespace {

constexpr int TILE = 64;

constexpr int STAGE_BYTES = 36864;   // shared staging of one K-chunk (A and B panels)

// One CTA computes the (m x n) output tile of one group for one plane:
//   C = beta C + sum_items coef * op(A)[rows] op(B)
// Items are concatenated along K in a shared staging buffer (each item's
// coefficient folded into its A panel, rows outside the item zero), so a
// group of many thin items costs one barrier pair per full chunk.  Large
// tiles (m, n > 32) use 4x4 register blocking over 64x64; smaller tiles
// spread their outputs over the threads and split each chunk's K across the
// spare threads, reducing the partial sums in shared memory at the end.
// SB: shared staging bytes of one K-chunk; MINB: CTAs per SM the register
// budget is sized for (the autotuned shape: larger chunks vs more CTAs)
template <typename T, typename Acc, int SB, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_ggemm(const GGroup* __restrict__ groups,
                                              const GItem* __restrict__ items,
                                              T* const* __restrict__ tab,
                                              const int* const* __restrict__ rtab, int P,
                                              int gbase, const double* __restrict__ coefs,
                                              double* __restrict__ flops) {
  const int p = blockIdx.y;
  const GGroup G = groups[gbase + blockIdx.x];
  long long fl = 0;   // counted flops (integer: FP64 is a slow pipe here)
  T* C = tab[G.cbuf * P + p];
  if (!C) return;
  const int m = dimv(G.m_st, G.m_rb, G.m_ri, rtab, P, p);
  const int n = dimv(G.n_st, G.n_rb, G.n_ri, rtab, P, p);
  if (m <= 0 || n <= 0) return;
  C += G.coff;
  constexpr int SE = SB / sizeof(Acc);
  __shared__ __align__(16) unsigned char stage_raw[SB];
  __shared__ Acc red[NT];
  Acc* sm = reinterpret_cast<Acc*>(stage_raw);
  const Acc beta = G.beta >= 0 ? (Acc)coefs[G.beta] : Acc(0);
  const bool blocked = (m > 32 && n > 32);
  // tall thin tiles (16 < m <= 64, 8 < n <= 32): 4 x NB micro-tiles on 16 x 16
  // threads over the whole K range (rows ty + 16 a, columns tx + 16 b,
  // accumulator a * 2 + b: compile-time indices keep them in registers)
  const int thinNB = (!blocked && m > 16 && n > 8 && n <= 32) ? (n > 16 ? 2 : 1) : 0;
  const bool thin = thinNB > 0;
  const int lda_s = (blocked || thin) ? TILE + 1 : m + 1;
  const int ldb_s = blocked ? TILE + 1 : (thin ? 16 * thinNB + 1 : n + 1);
  const int KC = SE / (lda_s + ldb_s);
  Acc* As = sm;                 // As[kk * lda_s + i]
  Acc* Bs = sm + KC * lda_s;    // Bs[kk * ldb_s + j]

  // thread roles
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;   // blocked
  const int nout = m * n;
  int OL = 1;
  while (OL < nout && OL < NT) OL <<= 1;
  const int S = (blocked || thin) ? 1 : NT / OL;
  const int lane = threadIdx.x % OL, slice = threadIdx.x / OL;
  const int Q = (nout + OL - 1) / OL;
  Acc acc[16];
#pragma unroll
  for (int q = 0; q < 16; ++q) acc[q] = Acc(0);

  auto thin_loop = [&](auto nbc, int kfill) {
    constexpr int NB = decltype(nbc)::value;
    for (int kk = 0; kk < kfill; ++kk) {
      Acc av[4], bv[NB];
#pragma unroll
      for (int a = 0; a < 4; ++a) av[a] = As[kk * lda_s + ty + 16 * a];
#pragma unroll
      for (int b = 0; b < NB; ++b) bv[b] = Bs[kk * ldb_s + tx + 16 * b];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[a * 2 + b] += av[a] * bv[b];
    }
  };
  auto compute = [&](int kfill) {
    __syncthreads();
    if (thin) {
      if (thinNB == 2) thin_loop(std::integral_constant<int, 2>(), kfill);
      else thin_loop(std::integral_constant<int, 1>(), kfill);
    } else if (blocked) {
      for (int kk = 0; kk < kfill; ++kk) {
        Acc av[4], bv[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) av[a] = As[kk * lda_s + ty + 16 * a];
#pragma unroll
        for (int b = 0; b < 4; ++b) bv[b] = Bs[kk * ldb_s + tx + 16 * b];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[a * 4 + b] += av[a] * bv[b];
      }
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q >= Q) break;
        const int o = lane + q * OL;
        if (o >= nout) break;
        const Acc* ap = As + (o % m);
        const Acc* bp = Bs + (o / m);
        Acc s0 = Acc(0), s1 = Acc(0), s2 = Acc(0), s3 = Acc(0);
        int kk = slice;
        for (; kk + 3 * S < kfill; kk += 4 * S) {
          s0 += ap[kk * lda_s] * bp[kk * ldb_s];
          s1 += ap[(kk + S) * lda_s] * bp[(kk + S) * ldb_s];
          s2 += ap[(kk + 2 * S) * lda_s] * bp[(kk + 2 * S) * ldb_s];
          s3 += ap[(kk + 3 * S) * lda_s] * bp[(kk + 3 * S) * ldb_s];
        }
        for (; kk < kfill; kk += S) s0 += ap[kk * lda_s] * bp[kk * ldb_s];
        acc[q] += (s0 + s1) + (s2 + s3);
      }
    }
    __syncthreads();
  };

  // items in batches of 32, each resolved by one thread of warp 0 (the
  // chains of dependent loads of a batch in flight at once) into a shared
  // table that the whole CTA then walks
  struct ItemR {
    const T* A;
    const T* B;
    int k, rows, aflags, bflags, lda, ldb, row_off, seed, omega_row0;
    Acc cf;
  };
  __shared__ ItemR sit[32];
  int kfill = 0;
  for (int base = G.ib; base < G.ie; base += 32) {
    const int cnt = min(32, G.ie - base);
    __syncthreads();   // the previous batch's table is read by every thread
    if (threadIdx.x < cnt) {
      const GItem J = items[base + threadIdx.x];
      ItemR R{};
      bool ok = !(J.guard0 >= 0 && !tab[J.guard0 * P + p]) &&
                !(J.guard1 >= 0 && !tab[J.guard1 * P + p]);
      if (ok && J.abuf >= 0) { R.A = tab[J.abuf * P + p]; ok = R.A != nullptr; if (ok) R.A += J.aoff; }
      if (ok && J.bbuf >= 0) { R.B = tab[J.bbuf * P + p]; ok = R.B != nullptr; if (ok) R.B += J.boff; }
      if (ok) {
        R.k = dimv(J.k_st, J.k_rb, J.k_ri, rtab, P, p);
        R.rows = dimv(J.r_st, J.r_rb, J.r_ri, rtab, P, p);
        R.cf = (Acc)coefs[J.coef];
      }
      R.aflags = J.aflags; R.bflags = J.bflags; R.lda = J.lda; R.ldb = J.ldb;
      R.row_off = J.row_off; R.seed = J.seed; R.omega_row0 = J.omega_row0;
      sit[threadIdx.x] = R;
    }
    __syncthreads();
    for (int qi = 0; qi < cnt; ++qi) {
      const ItemR I = sit[qi];
      const int k = I.k, rows = I.rows;
      if (k <= 0 || rows <= 0) continue;
      const T* A = I.A;
      const T* B = I.B;
      const Acc cf = I.cf;
      const int r0 = I.row_off;
      if ((I.aflags & FL_IDENT) || (I.bflags & FL_IDENT)) {
        // C(r0+i, j) += cf * B(i, j)  or  cf * A(i, j): straight into the accumulators
        fl += (long long)rows * n;
        const bool ai = I.aflags & FL_IDENT;
        if (thin) {
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const int i = ty + 16 * a - r0;
            if (i < 0 || i >= rows) continue;
#pragma unroll
            for (int b = 0; b < 2; ++b) {
              const int j = tx + 16 * b;
              if (b < thinNB && j < n)
                acc[a * 2 + b] += cf * (ai ? (Acc)B[i + (int64_t)j * I.ldb] : (Acc)A[i + (int64_t)j * I.lda]);
            }
          }
        } else if (blocked) {
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const int i = ty + 16 * a - r0;
            if (i < 0 || i >= rows) continue;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              const int j = tx + 16 * b;
              if (j < n)
                acc[a * 4 + b] += cf * (ai ? (Acc)B[i + (int64_t)j * I.ldb] : (Acc)A[i + (int64_t)j * I.lda]);
            }
          }
        } else if (slice == 0) {
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            if (q >= Q) break;
            const int o = lane + q * OL;
            if (o >= nout) break;
            const int i = o % m - r0, j = o / m;
            if (i < 0 || i >= rows) continue;
            acc[q] += cf * (ai ? (Acc)B[i + (int64_t)j * I.ldb] : (Acc)A[i + (int64_t)j * I.lda]);
          }
        }
        continue;
      }
      fl += 2LL * rows * n * k;
      const bool at = I.aflags & FL_T, bt = I.bflags & FL_T, bo = I.bflags & FL_OMEGA;
      const bool full = (r0 == 0 && rows >= m);
      // a whole 64 x 64 dense leaf (contiguous, 16-byte aligned): staged with
      // vector loads and shift indexing once it fits the chunk entirely
      const bool blockA = (rows == 64 && r0 == 0 && k == 64 && I.lda == 64 && KC >= 64 &&
                           (reinterpret_cast<uintptr_t>(A) & 15) == 0);
      const bool blockB = (!bo && !bt && n == 64 && k == 64 && I.ldb == 64 && KC >= 64 &&
                           (reinterpret_cast<uintptr_t>(B) & 15) == 0);
      if ((blockA || blockB) && kfill + 64 > KC) {
        compute(kfill);
        kfill = 0;
      }
      for (int k0 = 0; k0 < k;) {
        const int t = min(k - k0, KC - kfill);
        // A panel -> As[(kfill + kk) * lda_s + r0 + i], zero elsewhere in those columns
        if (blockA && t == 64) {
          constexpr int V = 16 / sizeof(T);
          for (int e0 = threadIdx.x * V; e0 < 4096; e0 += NT * V) {
            T v[V];
            *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(A + e0);
#pragma unroll
            for (int q = 0; q < V; ++q) {
              const int e = e0 + q;
              // column-major block: e = i + 64 l  (A)  or  e = l + 64 i  (A^T)
              const int i = at ? (e >> 6) : (e & 63), kk = at ? (e & 63) : (e >> 6);
              As[(kfill + kk) * lda_s + i] = cf * (Acc)v[q];
            }
          }
        } else {
        if (!full)
          for (int e = threadIdx.x; e < t * m; e += NT) {
            const int kk = e / m, i = e - kk * m;
            if (i < r0 || i >= r0 + rows) As[(kfill + kk) * lda_s + i] = Acc(0);
          }
        if (at) {
          for (int e = threadIdx.x; e < rows * t; e += NT) {
            const int i = e / t, kk = e - i * t;
            As[(kfill + kk) * lda_s + r0 + i] = cf * (Acc)A[(k0 + kk) + (int64_t)i * I.lda];
          }
        } else {
          for (int e = threadIdx.x; e < rows * t; e += NT) {
            const int kk = e / rows, i = e - kk * rows;
            As[(kfill + kk) * lda_s + r0 + i] = cf * (Acc)A[i + (int64_t)(k0 + kk) * I.lda];
          }
        }
        }
        // B panel -> Bs[(kfill + kk) * ldb_s + j]
        if (blockB && t == 64) {
          constexpr int V = 16 / sizeof(T);
          for (int e0 = threadIdx.x * V; e0 < 4096; e0 += NT * V) {
            T v[V];
            *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(B + e0);
#pragma unroll
            for (int q = 0; q < V; ++q) {
              const int e = e0 + q;   // e = l + 64 j
              Bs[(kfill + (e & 63)) * ldb_s + (e >> 6)] = (Acc)v[q];
            }
          }
        } else if (bo) {
          for (int e = threadIdx.x; e < t * n; e += NT) {
            const int kk = e / n, j = e - kk * n;
            Bs[(kfill + kk) * ldb_s + j] =
                (Acc)omega((uint32_t)I.seed, (uint32_t)(I.omega_row0 + k0 + kk), (uint32_t)j);
          }
        } else if (bt) {
          for (int e = threadIdx.x; e < t * n; e += NT) {
            const int kk = e / n, j = e - kk * n;
            Bs[(kfill + kk) * ldb_s + j] = (Acc)B[j + (int64_t)(k0 + kk) * I.ldb];
          }
        } else {
          for (int e = threadIdx.x; e < t * n; e += NT) {
            const int j = e / t, kk = e - j * t;
            Bs[(kfill + kk) * ldb_s + j] = (Acc)B[(k0 + kk) + (int64_t)j * I.ldb];
          }
        }
        kfill += t;
        k0 += t;
        if (kfill == KC) {
          compute(kfill);
          kfill = 0;
        }
      }
    }
  }
  if (kfill > 0) compute(kfill);

  if (thin) {
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int i = ty + 16 * a;
      if (i >= m) continue;
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const int j = tx + 16 * b;
        if (b >= thinNB || j >= n) continue;
        T* c = C + i + (int64_t)j * G.ldc;
        Acc v = acc[a * 2 + b];
        if (G.beta >= 0) v += beta * (Acc)(*c);
        *c = (T)v;
      }
    }
  } else if (blocked) {
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const int i = ty + 16 * a;
      if (i >= m) continue;
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const int j = tx + 16 * b;
        if (j >= n) continue;
        T* c = C + i + (int64_t)j * G.ldc;
        Acc v = acc[a * 4 + b];
        if (G.beta >= 0) v += beta * (Acc)(*c);
        *c = (T)v;
      }
    }
  } else {
    if (S > 1) {   // Q == 1: one output per lane, reduce the K slices
      red[threadIdx.x] = acc[0];
      __syncthreads();
      if (slice == 0) {
        Acc s2 = Acc(0);
        for (int t2 = 0; t2 < S; ++t2) s2 += red[lane + t2 * OL];
        acc[0] = s2;
      }
    }
    if (slice == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (q >= Q) break;
        const int o = lane + q * OL;
        if (o >= nout) break;
        T* c = C + (o % m) + (int64_t)(o / m) * G.ldc;
        Acc v = acc[q];
        if (G.beta >= 0) v += beta * (Acc)(*c);
        *c = (T)v;
      }
    }
  }
  if (flops && threadIdx.x == 0 && fl > 0) atomicAdd(flops, (double)fl);
}

// Grouped products with outputs of up to 64 x 64 (every stage that is no inner
// product), one CTA per group.  A group's items of dynamic rank (a few columns
// each) are laid end to end along the inner dimension and cut into chunks of KC
// rows whatever their own ranks are; a chunk's rows get their operand
// addresses first (one thread per row), so that all of its loads are in flight
// together -- a group of thirty rank-3 items costs two round trips to L2, not
// thirty.  Its items with a dense leaf (inner dimension = leaf size) are chunks of
// their own, addressed without a table.  Operands are staged without integer
// divisions: those contiguous along the output with lanes along it, the
// others (A transposed, B plain) as 8 x 4 patches per warp, whose loads fill
// whole 32-byte sectors and whose stores meet no bank conflict.  4 x 4 register
// tiles read both operands as 16-byte vectors (3 shared wavefronts per 16
// multiply-adds); outputs with fewer than 256 tiles split the chunk's rows over
// the spare threads, whose partial sums are added in a fixed order at the end.
//
// Bound by the latency of its chunks (three CTAs per SM, ~4 us per dense item at one
// CTA), not by the FMA pipe: dense sums of the n = 64 convection-diffusion setup
// 47 ms against 62 ms in k_ggemm, n = 80 (50-point leaves, which k_ggemm stages
// with a division per entry) 110 against 172 ms, sketch products 91 against 140 ms.
constexpr int CI = 64;         // items resolved at a time
constexpr int CLD = TILE + 4;  // row length of the staged A: 16-byte rows, 8 x 4 patches conflict-free

template <typename T>
struct __align__(16) CatOp {   // one operand of a chunk row
  const T* x;                  // A: first entry, contiguous; B: first entry
  int info;                    // A: first output row | rows << 8; B: stride of the columns
  float cf;                    // A: coefficient (+-1)
};

// 16-byte vectors of shared operands
__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
  const float4 x = *reinterpret_cast<const float4*>(p);
  v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
  const double2 x = *reinterpret_cast<const double2*>(p), y = *reinterpret_cast<const double2*>(p + 2);
  v[0] = x.x; v[1] = x.y; v[2] = y.x; v[3] = y.y;
}

template <typename T>
__host__ __device__ constexpr int cat_bytes() { return 64 * 2 * CLD * (int)sizeof(T); }   // 64 rows of both operands

template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 3 : 2)
    k_gcat(const GGroup* __restrict__ groups, const GItem* __restrict__ items,
           T* const* __restrict__ tab, const int* const* __restrict__ rtab, int P, int gbase,
           const double* __restrict__ coefs, double* __restrict__ flops) {
  const int p = blockIdx.y;
  const GGroup G = groups[gbase + blockIdx.x];
  T* C = tab[G.cbuf * P + p];
  if (!C) return;
  const int m = dimv(G.m_st, G.m_rb, G.m_ri, rtab, P, p);
  const int nall = dimv(G.n_st, G.n_rb, G.n_ri, rtab, P, p);
  // this CTA's columns j0 ... j0 + n - 1 of the group's output
  const int nc = ((nall + 4 * (int)gridDim.z - 1) / (4 * (int)gridDim.z)) * 4;
  const int j0 = blockIdx.z * nc, n = min(nc, nall - j0);
  if (m <= 0 || n <= 0) return;
  C += G.coff + (int64_t)j0 * G.ldc;
  extern __shared__ __align__(16) unsigned char cat_raw[];
  struct ItemR {
    const T* A;
    const T* B;
    int rows, flags, lda, ldb, row_off, seed, omega_row0, k;
    float cf;
  };
  __shared__ ItemR sit[CI];
  __shared__ int koff[CI + 1];      // first row of each item in the batch
  __shared__ int xlist[CI], s_cnt[4];   // dense items from the front, identity items from the back
  __shared__ CatOp<T> ra[128], rb[128];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int MT = (m + 3) >> 2, N4 = (n + 3) >> 2, tiles = MT * N4;
  const int ldb_s = 4 * N4 + 4;
  const int KC = min(128, (cat_bytes<T>() / (int)sizeof(T) / (CLD + ldb_s)) & ~7);
  T* As = reinterpret_cast<T*>(cat_raw);      // As[kk * CLD + i]
  T* Bs = As + KC * CLD;                      // Bs[kk * ldb_s + j]
  const int S = NT / tiles;                   // row slices (tiles <= 256)
  const int slice = tid / tiles, tile = tid - slice * tiles;
  const int ty = tile / N4, tx = tile - ty * N4;
  const bool active = slice < S;
  T acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
  auto compute = [&](int kf) {
    __syncthreads();
    if (active) {
#pragma unroll 4
      for (int kk = slice; kk < kf; kk += S) {
        T a[4], b[4];
        ld4(As + kk * CLD + 4 * ty, a);
        ld4(Bs + kk * ldb_s + 4 * tx, b);
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) acc[x][y] += a[x] * b[y];
      }
    }
    __syncthreads();
  };

  for (int base = G.ib; base < G.ie; base += CI) {
    const int cnt = min(CI, G.ie - base);
    __syncthreads();   // the previous batch is done with the tables
    if (tid < CI) {
      ItemR R{};
      bool dyn = false;
      if (tid < cnt) {
        const GItem J = items[base + tid];
        bool ok = !(J.guard0 >= 0 && !tab[J.guard0 * P + p]) &&
                  !(J.guard1 >= 0 && !tab[J.guard1 * P + p]);
        if (ok && J.abuf >= 0) { R.A = tab[J.abuf * P + p]; ok = R.A != nullptr; if (ok) R.A += J.aoff; }
        if (ok && J.bbuf >= 0) { R.B = tab[J.bbuf * P + p]; ok = R.B != nullptr; if (ok) R.B += J.boff; }
        if (ok) {
          R.k = dimv(J.k_st, J.k_rb, J.k_ri, rtab, P, p);
          R.rows = dimv(J.r_st, J.r_rb, J.r_ri, rtab, P, p);
          R.cf = (float)coefs[J.coef];
          if (R.k <= 0 || R.rows <= 0) R.k = R.rows = 0;
        }
        // A transposed (1); B contiguous along the columns (2), sketch rows (8); identity A (16), B (32)
        R.flags = ((J.aflags & FL_T) ? 1 : 0) | ((J.bflags & FL_T) ? 2 : 0) |
                  ((J.bflags & FL_OMEGA) ? 8 : 0) | ((J.aflags & FL_IDENT) ? 16 : 0) |
                  ((J.bflags & FL_IDENT) ? 32 : 0);
        dyn = J.k_rb >= 0;
        R.lda = J.lda; R.ldb = J.ldb;
        R.row_off = J.row_off; R.seed = J.seed; R.omega_row0 = J.omega_row0;
        if (flops && R.k > 0) {
          const double w = (R.flags & 48) ? (double)R.rows * n : 2.0 * R.rows * n * R.k;
          atomicAdd(flops, w);
        }
      }
      sit[tid] = R;
      const bool ident = R.k > 0 && (R.flags & 48), dense = R.k > 0 && !dyn && !ident;
      int inc = (R.k > 0 && dyn) ? R.k : 0;   // inclusive scan over the warp's items
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      koff[tid + 1] = inc;
      const unsigned md = __ballot_sync(0xffffffffu, dense), mi = __ballot_sync(0xffffffffu, ident);
      if (lane == 0) { s_cnt[warp] = __popc(md); s_cnt[2 + warp] = __popc(mi); }
      asm volatile("bar.sync 1, 64;" ::: "memory");   // the two resolving warps
      if (tid >= 32) koff[tid + 1] = inc + koff[32];
      if (tid == 0) koff[0] = 0;
      const unsigned below = (1u << lane) - 1u;
      if (dense) xlist[(warp ? s_cnt[0] : 0) + __popc(md & below)] = tid;
      if (ident) xlist[CI - 1 - (warp ? s_cnt[2] : 0) - __popc(mi & below)] = tid;
    }
    __syncthreads();
    const int ktot = koff[CI], ndense = s_cnt[0] + s_cnt[1], nident = s_cnt[2] + s_cnt[3];
    if (active && slice == 0)
      for (int q = 0; q < nident; ++q) {
        // C(r0 + i, j) += cf * B(i, j)  or  cf * A(i, j)
        const ItemR& I = sit[xlist[CI - 1 - q]];
        const bool ai = I.flags & 16, bt = I.flags & 2;
        const int64_t si = ai && bt ? I.ldb : 1, sj = ai ? (bt ? 1 : I.ldb) : I.lda;
        const T* X = ai ? I.B : I.A;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const int i = 4 * ty + a - I.row_off;
          if (i < 0 || i >= I.rows) continue;
#pragma unroll
          for (int b = 0; b < 4; ++b)
            if (4 * tx + b < n) acc[a][b] += (T)I.cf * X[i * si + (j0 + 4 * tx + b) * sj];
        }
      }
    // ---- the dynamic-rank items
    for (int c0 = 0; c0 < ktot; c0 += KC) {
      const int kf = min(KC, ktot - c0);
      if (tid < kf) {   // each row's operands
        const int r = c0 + tid;
        int lo = 0, hi = CI;            // the item with koff[lo] <= r < koff[lo + 1]
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (koff[mid] <= r) lo = mid;
          else hi = mid;
        }
        const ItemR& I = sit[lo];
        const int l = r - koff[lo];
        ra[tid] = CatOp<T>{I.A + (int64_t)l * I.lda, I.row_off | I.rows << 8, I.cf};
        rb[tid] = (I.flags & 2) ? CatOp<T>{I.B + (int64_t)l * I.ldb + j0, 1, 0.f}
                                : CatOp<T>{I.B + l + (int64_t)j0 * I.ldb, I.ldb, 0.f};
      }
      __syncthreads();
      {
        const int i = tid & 63;
        constexpr int U = 8;
        for (int k0 = tid >> 6; k0 < kf; k0 += 4 * U) {
          T v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            v[u] = T(0);
            if (k0 + 4 * u < kf) {
              const CatOp<T> D = ra[k0 + 4 * u];
              const int ii = i - (D.info & 255);
              if (ii >= 0 && ii < (D.info >> 8)) v[u] = (T)D.cf * D.x[ii];
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (k0 + 4 * u < kf) As[(k0 + 4 * u) * CLD + i] = v[u];
        }
      }
      {
        const int jw = N4 <= 1 ? 4 : N4 <= 2 ? 8 : N4 <= 4 ? 16 : N4 <= 8 ? 32 : 64;
        const int j = tid & (jw - 1), ks = NT / jw;
        constexpr int U = 4;
        for (int k0 = tid / jw; k0 < kf; k0 += ks * U) {
          T v[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            v[u] = T(0);
            if (k0 + ks * u < kf && j < n) {
              const CatOp<T> D = rb[k0 + ks * u];
              v[u] = D.x[(int64_t)j * D.info];
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (k0 + ks * u < kf && j < 4 * N4) Bs[(k0 + ks * u) * ldb_s + j] = v[u];
        }
      }
      compute(kf);
    }
    // ---- the items with a dense leaf: all of a thread's loads in flight, the
    // next item's (float) while the tiles of the one before are multiplied
    const int lk = 8 * warp + (lane >> 2);   // row of the 8 x 4 patches
    constexpr bool AHEAD = sizeof(T) == 4;
    T va[16], vb[16];
    auto load = [&](int q) {
      const ItemR& I = sit[xlist[q]];
      const int k = I.k, rows = I.rows, r0 = I.row_off, flags = I.flags;
      if (flags & 1) {
        const T* A = I.A + lk;
        const int64_t ld = I.lda;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int ii = 4 * u + (lane & 3) - r0;
          va[u] = (lk < k && ii >= 0 && ii < rows) ? A[ii * ld] : T(0);
        }
      } else {
        const int ii = (tid & 63) - r0;
        const T* A = I.A + ii;
        const int64_t ld = I.lda;
        const bool in = ii >= 0 && ii < rows;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int l = (tid >> 6) + 4 * u;
          va[u] = (in && l < k) ? A[l * ld] : T(0);
        }
      }
      if (!(flags & 10)) {
        const T* B = I.B + lk;
        const int64_t ld = I.ldb;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int j = 4 * u + (lane & 3);
          vb[u] = (u < N4 && lk < k && j < n) ? B[(j0 + j) * ld] : T(0);
        }
      }
    };
    if (AHEAD && ndense > 0) load(0);
    for (int q = 0; q < ndense; ++q) {
      if (!AHEAD) load(q);
      const ItemR& I = sit[xlist[q]];
      const int k = I.k, flags = I.flags;
      const T cf = (T)I.cf;
      if (flags & 1) {
#pragma unroll
        for (int u = 0; u < 16; ++u) As[lk * CLD + 4 * u + (lane & 3)] = cf * va[u];
      } else {
#pragma unroll
        for (int u = 0; u < 16; ++u) As[((tid >> 6) + 4 * u) * CLD + (tid & 63)] = cf * va[u];
      }
      if (!(flags & 10)) {
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (u < N4) Bs[lk * ldb_s + 4 * u + (lane & 3)] = vb[u];
      } else {
        for (int e = warp; e < k; e += NT / 32)
          for (int j = lane; j < n; j += 32)
            Bs[e * ldb_s + j] = (flags & 8) ? (T)omega((uint32_t)I.seed, (uint32_t)(I.omega_row0 + e),
                                                       (uint32_t)(j0 + j))
                                            : I.B[j0 + j + (int64_t)e * I.ldb];
      }
      if (AHEAD && q + 1 < ndense) load(q + 1);
      compute(k);
    }
  }
  // the slices' sums, laid out by columns: element (i, j) of slice s at
  // red[s * R + j * 4 MT + i]; stored with lanes along the rows
  T* red = reinterpret_cast<T*>(cat_raw);
  const int R = 16 * tiles, m4 = 4 * MT;
  const T beta = G.beta >= 0 ? (T)coefs[G.beta] : T(0);
  __syncthreads();
  if (active)
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
      for (int a = 0; a < 4; ++a) red[slice * R + (4 * tx + b) * m4 + 4 * ty + a] = acc[a][b];
  __syncthreads();
  for (int jb = warp; jb < n; jb += 4 * (NT / 32)) {
    T old[4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h, j = jb + u * (NT / 32);
        old[u][h] = (G.beta >= 0 && i < m && j < n) ? C[i + (int64_t)j * G.ldc] : T(0);
      }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h, j = jb + u * (NT / 32);
        if (i >= m || j >= n) continue;
        T v = red[j * m4 + i];
        for (int s = 1; s < S; ++s) v += red[s * R + j * m4 + i];
        C[i + (int64_t)j * G.ldc] = G.beta >= 0 ? v + beta * old[u][h] : v;
      }
  }
}

// The factor products of a bundle: groups whose items read the same A operands
// (the leaves of one block B(r, s), or A(t, r)) against the factors of different
// low-rank blocks.  The groups' columns stand side by side, up to 64 at a time, so
// that every dense leaf is staged once for all of them: alone, a group of rank
// 3 does 6 flops per entry of the 64 x 64 leaf it loads and the stage is
// bound by L2; a bundle of 16 does about 100 (n = 64 setup: 45 ms against 88 ms with
// one CTA per group and 71 ms with one warp per group; n = 80: 127 against 342 and
// 181 ms).  Tiles, chunks and staging as in
// k_gcat (A plain or transposed, B plain, C overwritten).
constexpr int BI = 32;         // items resolved at a time

template <typename T>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 3 : 2)
    k_gbundle(const int* __restrict__ bundles, const GGroup* __restrict__ groups,
              const GItem* __restrict__ items, T* const* __restrict__ tab,
              const int* const* __restrict__ rtab, int P, const double* __restrict__ coefs,
              double* __restrict__ flops) {
  const int p = blockIdx.y;
  const int gb = bundles[2 * blockIdx.x], ng = bundles[2 * blockIdx.x + 1] - gb;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ __align__(16) unsigned char cat_raw[];
  struct ItemA {
    const T* A;
    int k, rows, flags, lda, row_off;
    float cf;
  };
  __shared__ ItemA sit[BI];
  __shared__ const T* bp[BI][BUNDLE_MAX];   // B operand of (item, group)
  __shared__ int bld[BI][BUNDLE_MAX];
  __shared__ T* cp[BUNDLE_MAX];             // output of each group
  __shared__ int cld[BUNDLE_MAX], noff[BUNDLE_MAX + 1], ib[BUNDLE_MAX];
  __shared__ int koff[BI + 1], xlist[BI], s_nd;
  __shared__ short colg[TILE], coll[TILE];  // group and own column of each output column
  __shared__ CatOp<T> ra[128];
  __shared__ int2 rb[128];                  // item and row of each chunk row
  const GGroup G0 = groups[gb];
  const int m = dimv(G0.m_st, G0.m_rb, G0.m_ri, rtab, P, p);
  if (tid < 32) {
    int n = 0;
    if (lane < ng) {
      const GGroup G = groups[gb + lane];
      T* C = tab[G.cbuf * P + p];
      n = C ? max(0, dimv(G.n_st, G.n_rb, G.n_ri, rtab, P, p)) : 0;
      cp[lane] = C ? C + G.coff : nullptr;
      cld[lane] = G.ldc;
      ib[lane] = G.ib;
    }
    int inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane < ng) noff[lane + 1] = inc;
    if (lane == 0) noff[0] = 0;
  }
  __syncthreads();
  const int nall = noff[ng], nitems = G0.ie - G0.ib;
  if (m <= 0 || nall <= 0) return;
  const int MT = (m + 3) >> 2;
  for (int j0 = 0; j0 < nall; j0 += TILE) {
    const int n = min(TILE, nall - j0);
    const int N4 = (n + 3) >> 2, tiles = MT * N4, ldb_s = 4 * N4 + 4;
    const int KC = min(128, (cat_bytes<T>() / (int)sizeof(T) / (CLD + ldb_s)) & ~7);
    T* As = reinterpret_cast<T*>(cat_raw);
    T* Bs = As + KC * CLD;
    const int S = NT / tiles;
    const int slice = tid / tiles, tile = tid - slice * tiles;
    const int ty = tile / N4, tx = tile - ty * N4;
    const bool active = slice < S;
    T acc[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] = T(0);
    auto compute = [&](int kf) {
      __syncthreads();
      if (active) {
#pragma unroll 4
        for (int kk = slice; kk < kf; kk += S) {
          T a[4], b[4];
          ld4(As + kk * CLD + 4 * ty, a);
          ld4(Bs + kk * ldb_s + 4 * tx, b);
#pragma unroll
          for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) acc[x][y] += a[x] * b[y];
        }
      }
      __syncthreads();
    };
    if (tid < TILE) {
      int g = 0;
      if (tid < n)
        while (noff[g + 1] <= j0 + tid) ++g;
      colg[tid] = (short)g;
      coll[tid] = (short)(j0 + tid - noff[g]);
    }
    for (int base = 0; base < nitems; base += BI) {
      const int cnt = min(BI, nitems - base);
      __syncthreads();
      if (tid < 32) {
        ItemA R{};
        bool dyn = false;
        if (lane < cnt) {
          const GItem J = items[G0.ib + base + lane];
          R.A = tab[J.abuf * P + p];
          if (R.A) {
            R.A += J.aoff;
            R.k = dimv(J.k_st, J.k_rb, J.k_ri, rtab, P, p);
            R.rows = dimv(J.r_st, J.r_rb, J.r_ri, rtab, P, p);
            R.cf = (float)coefs[J.coef];
            if (R.k <= 0 || R.rows <= 0) R.k = R.rows = 0;
          }
          R.flags = (J.aflags & FL_T) ? 1 : 0;
          R.lda = J.lda; R.row_off = J.row_off;
          dyn = J.k_rb >= 0;
          if (flops && R.k > 0) atomicAdd(flops, 2.0 * R.rows * n * R.k);
        }
        sit[lane] = R;
        const bool dense = R.k > 0 && !dyn;
        int inc = (R.k > 0 && dyn) ? R.k : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += v;
        }
        koff[lane + 1] = inc;
        if (lane == 0) koff[0] = 0;
        const unsigned md = __ballot_sync(0xffffffffu, dense);
        if (dense) xlist[__popc(md & ((1u << lane) - 1u))] = lane;
        if (lane == 0) s_nd = __popc(md);
      } else {
        for (int e = tid - 32; e < cnt * ng; e += NT - 32) {
          const int q = e / ng, g = e - q * ng;
          const GItem& J = items[ib[g] + base + q];
          const T* B = tab[J.bbuf * P + p];
          bp[q][g] = B ? B + J.boff : nullptr;
          bld[q][g] = J.ldb;
        }
      }
      __syncthreads();
      const int ktot = koff[BI], ndense = s_nd;
      // ---- the dynamic-rank items
      for (int c0 = 0; c0 < ktot; c0 += KC) {
        const int kf = min(KC, ktot - c0);
        if (tid < kf) {
          const int r = c0 + tid;
          int lo = 0, hi = BI;
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (koff[mid] <= r) lo = mid;
            else hi = mid;
          }
          const ItemA& I = sit[lo];
          const int l = r - koff[lo];
          ra[tid] = CatOp<T>{I.A + (int64_t)l * I.lda, I.row_off | I.rows << 8, I.cf};
          rb[tid] = make_int2(lo, l);
        }
        __syncthreads();
        {
          const int i = tid & 63;
          constexpr int U = 8;
          for (int k0 = tid >> 6; k0 < kf; k0 += 4 * U) {
            T v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              v[u] = T(0);
              if (k0 + 4 * u < kf) {
                const CatOp<T> D = ra[k0 + 4 * u];
                const int ii = i - (D.info & 255);
                if (ii >= 0 && ii < (D.info >> 8)) v[u] = (T)D.cf * D.x[ii];
              }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
              if (k0 + 4 * u < kf) As[(k0 + 4 * u) * CLD + i] = v[u];
          }
        }
        {   // lanes along the rows, which are contiguous within an item
          constexpr int U = 4;
          const int kk = tid & 127;
          const int2 r = rb[kk < kf ? kk : 0];
          for (int jb = tid >> 7; jb < 4 * N4; jb += 2 * U) {
            T v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const int j = jb + 2 * u;
              v[u] = T(0);
              if (kk < kf && j < n) {
                const int g = colg[j];
                const T* B = bp[r.x][g];
                if (B) v[u] = B[r.y + (int64_t)coll[j] * bld[r.x][g]];
              }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
              if (kk < kf && jb + 2 * u < 4 * N4) Bs[kk * ldb_s + jb + 2 * u] = v[u];
          }
        }
        compute(kf);
      }
      // ---- the dense leaves
      const int lk = 8 * warp + (lane >> 2);   // row of the 8 x 4 patches
      T va[16], vb[16];
      auto load = [&](int x) {
        const int q = xlist[x];
        const ItemA& I = sit[q];
        const int k = I.k, rows = I.rows, r0 = I.row_off;
        if (I.flags & 1) {
          const T* A = I.A + lk;
          const int64_t ld = I.lda;
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int ii = 4 * u + (lane & 3) - r0;
            va[u] = (lk < k && ii >= 0 && ii < rows) ? A[ii * ld] : T(0);
          }
        } else {
          const int ii = (tid & 63) - r0;
          const T* A = I.A + ii;
          const int64_t ld = I.lda;
          const bool in = ii >= 0 && ii < rows;
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const int l = (tid >> 6) + 4 * u;
            va[u] = (in && l < k) ? A[l * ld] : T(0);
          }
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int j = 4 * u + (lane & 3);
          vb[u] = T(0);
          if (u < N4 && lk < k && j < n) {
            const int g = colg[j];
            const T* B = bp[q][g];
            if (B) vb[u] = B[lk + (int64_t)coll[j] * bld[q][g]];
          }
        }
      };
      if (ndense > 0) load(0);
      for (int x = 0; x < ndense; ++x) {
        const ItemA& I = sit[xlist[x]];
        const int k = I.k;
        const T cf = (T)I.cf;
        if (I.flags & 1) {
#pragma unroll
          for (int u = 0; u < 16; ++u) As[lk * CLD + 4 * u + (lane & 3)] = cf * va[u];
        } else {
#pragma unroll
          for (int u = 0; u < 16; ++u) As[((tid >> 6) + 4 * u) * CLD + (tid & 63)] = cf * va[u];
        }
#pragma unroll
        for (int u = 0; u < 16; ++u)
          if (u < N4) Bs[lk * ldb_s + 4 * u + (lane & 3)] = vb[u];
        if (x + 1 < ndense) load(x + 1);
        compute(k);
      }
    }
    T* red = reinterpret_cast<T*>(cat_raw);
    const int R = 16 * tiles, m4 = 4 * MT;
    __syncthreads();
    if (active)
#pragma unroll
      for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) red[slice * R + (4 * tx + b) * m4 + 4 * ty + a] = acc[a][b];
    __syncthreads();
    for (int j = warp; j < n; j += NT / 32) {
      const int g = colg[j];
      T* C = cp[g] + (int64_t)coll[j] * cld[g];
      for (int i = lane; i < m; i += 32) {
        T v = red[j * m4 + i];
        for (int s = 1; s < S; ++s) v += red[s * R + j * m4 + i];
        C[i] = v;
      }
    }
    __syncthreads();
  }
}

// Warp-per-group form of k_ggemm for float operands and row panels
// (m <= 64 output rows): one warp owns one group's m x n output, lane l
// rows l and l + 32, NB columns at a time (more columns: further passes over
// the items).  Per item, a K-chunk of B (times the item's coefficient) is
// staged in the warp's own shared slice; A is read straight from global
// memory, four K-steps of loads in flight, each lane its two rows.  No
// block-wide barrier: a CTA's 8 warps run 8 independent groups, so the
// many tiny groups of the factor, sketch and basis stages (64 x r outputs,
// r of a few units, K of a few units to 64) cost a warp's worth of latency
// each instead of a whole CTA's staging round trip.
template <int NB>
__device__ __forceinline__ void gwarp_panel(const GGroup& G, const GItem* __restrict__ items,
                                            float* const* __restrict__ tab,
                                            const int* const* __restrict__ rtab, int P, int p,
                                            int m, int n, float* C,
                                            const double* __restrict__ coefs, float* Bs,
                                            long long& fl) {
  constexpr int KCH = 32, LDB = NB + 4;
  const int lane = threadIdx.x & 31;
  const float beta = G.beta >= 0 ? (float)coefs[G.beta] : 0.f;
  for (int j0 = 0; j0 < n; j0 += NB) {
    const int nb = min(NB, n - j0);
    float acc0[NB], acc1[NB];
#pragma unroll
    for (int j = 0; j < NB; ++j) { acc0[j] = 0.f; acc1[j] = 0.f; }
    for (int base = G.ib; base < G.ie; base += 32) {
      // lane q resolves item base + q: every item's chain of dependent loads
      // (descriptor, operand pointers, ranks, coefficient) in flight at once
      const float* rA = nullptr;
      const float* rB = nullptr;
      int rk = 0, rrows = 0, rflags = 0, rr0 = 0, rlda = 0, rldb = 0, rseed = 0, rorow = 0;
      float rcf = 0.f;
      if (base + lane < G.ie) {
        const GItem I = items[base + lane];
        bool ok = !(I.guard0 >= 0 && !tab[I.guard0 * P + p]) &&
                  !(I.guard1 >= 0 && !tab[I.guard1 * P + p]);
        if (ok && I.abuf >= 0) { rA = tab[I.abuf * P + p]; ok = rA != nullptr; if (ok) rA += I.aoff; }
        if (ok && I.bbuf >= 0) { rB = tab[I.bbuf * P + p]; ok = rB != nullptr; if (ok) rB += I.boff; }
        if (ok) {
          rk = dimv(I.k_st, I.k_rb, I.k_ri, rtab, P, p);
          rrows = dimv(I.r_st, I.r_rb, I.r_ri, rtab, P, p);
          rcf = (float)coefs[I.coef];
          rflags = ((I.aflags & FL_IDENT) ? 1 : 0) | ((I.bflags & FL_IDENT) ? 2 : 0) |
                   ((I.aflags & FL_T) ? 4 : 0) | ((I.bflags & FL_T) ? 8 : 0) |
                   ((I.bflags & FL_OMEGA) ? 16 : 0);
          rr0 = I.row_off; rlda = I.lda; rldb = I.ldb; rseed = I.seed; rorow = I.omega_row0;
        } else {
          rk = 0;
        }
      }
      const int cnt = min(32, G.ie - base);
      for (int q = 0; q < cnt; ++q) {
        const int k = __shfl_sync(0xffffffffu, rk, q);
        const int rows = __shfl_sync(0xffffffffu, rrows, q);
        if (k <= 0 || rows <= 0) continue;
        const float* A = reinterpret_cast<const float*>(
            __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(rA), q));
        const float* B = reinterpret_cast<const float*>(
            __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(rB), q));
        const float cf = __shfl_sync(0xffffffffu, rcf, q);
        const int flags = __shfl_sync(0xffffffffu, rflags, q);
        const int row_off = __shfl_sync(0xffffffffu, rr0, q);
        const int lda = __shfl_sync(0xffffffffu, rlda, q);
        const int ldb = __shfl_sync(0xffffffffu, rldb, q);
        const int seed = __shfl_sync(0xffffffffu, rseed, q);
        const int orow0 = __shfl_sync(0xffffffffu, rorow, q);
        const int i0 = lane - row_off, i1 = lane + 32 - row_off;
        const bool v0 = i0 >= 0 && i0 < rows, v1 = i1 >= 0 && i1 < rows;
        if (flags & 3) {
          // C(row_off + i, j) += cf * B(i, j)  or  cf * A(i, j)
          fl += (long long)rows * nb;
          const float* src = (flags & 1) ? B : A;
          const int ld = (flags & 1) ? ldb : lda;
#pragma unroll
          for (int j = 0; j < NB; ++j) {
            if (j < nb) {
              if (v0) acc0[j] += cf * src[i0 + (int64_t)(j0 + j) * ld];
              if (v1) acc1[j] += cf * src[i1 + (int64_t)(j0 + j) * ld];
            }
          }
          continue;
        }
        fl += 2LL * rows * nb * k;
        const bool at = flags & 4, bt = flags & 8, bo = flags & 16;
        // A(i, l): A[i + l lda] (plain) or A[l + i lda] (transposed)
        const int astep = at ? 1 : lda;
        const float* a0 = A + (v0 ? (at ? (int64_t)i0 * lda : i0) : 0);
        const float* a1 = A + (v1 ? (at ? (int64_t)i1 * lda : i1) : 0);
        for (int k0 = 0; k0 < k; k0 += KCH) {
          const int kt = min(KCH, k - k0);
          __syncwarp();
          for (int e = lane; e < kt * NB; e += 32) {
            const int kk = e / NB, j = e % NB;
            float v = 0.f;
            if (j < nb) {
              const int l = k0 + kk, jj = j0 + j;
              v = bo ? omega((uint32_t)seed, (uint32_t)(orow0 + l), (uint32_t)jj)
                     : (bt ? B[jj + (int64_t)l * ldb] : B[l + (int64_t)jj * ldb]);
            }
            Bs[kk * LDB + j] = cf * v;
          }
          __syncwarp();
          // A pointers at this chunk (offsets within a 64-row leaf panel
          // stay far inside 32 bits: K-chunks of at most 32 columns)
          const float* p0 = a0 + (int64_t)k0 * astep;
          const float* p1 = a1 + (int64_t)k0 * astep;
          // K-steps of A loads in flight (fewer for wide panels: registers)
          constexpr int UK = NB >= 32 ? 2 : 4;
          int kk = 0;
          for (; kk + UK <= kt; kk += UK) {
            float x0[UK], x1[UK];
#pragma unroll
            for (int u = 0; u < UK; ++u) {
              x0[u] = v0 ? p0[(kk + u) * astep] : 0.f;
              x1[u] = v1 ? p1[(kk + u) * astep] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < UK; ++u) {
#pragma unroll
              for (int q = 0; q < NB / 4; ++q) {
                const float4 b = *reinterpret_cast<const float4*>(Bs + (kk + u) * LDB + 4 * q);
                acc0[4 * q] += x0[u] * b.x; acc0[4 * q + 1] += x0[u] * b.y;
                acc0[4 * q + 2] += x0[u] * b.z; acc0[4 * q + 3] += x0[u] * b.w;
                acc1[4 * q] += x1[u] * b.x; acc1[4 * q + 1] += x1[u] * b.y;
                acc1[4 * q + 2] += x1[u] * b.z; acc1[4 * q + 3] += x1[u] * b.w;
              }
            }
          }
          for (; kk < kt; ++kk) {
            const float y0 = v0 ? p0[kk * astep] : 0.f;
            const float y1 = v1 ? p1[kk * astep] : 0.f;
#pragma unroll
            for (int q = 0; q < NB / 4; ++q) {
              const float4 b = *reinterpret_cast<const float4*>(Bs + kk * LDB + 4 * q);
              acc0[4 * q] += y0 * b.x; acc0[4 * q + 1] += y0 * b.y;
              acc0[4 * q + 2] += y0 * b.z; acc0[4 * q + 3] += y0 * b.w;
              acc1[4 * q] += y1 * b.x; acc1[4 * q + 1] += y1 * b.y;
              acc1[4 * q + 2] += y1 * b.z; acc1[4 * q + 3] += y1 * b.w;
            }
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      if (j >= nb) continue;
      if (lane < m) {
        float* c = C + lane + (int64_t)(j0 + j) * G.ldc;
        *c = acc0[j] + (G.beta >= 0 ? beta * *c : 0.f);
      }
      if (lane + 32 < m) {
        float* c = C + lane + 32 + (int64_t)(j0 + j) * G.ldc;
        *c = acc1[j] + (G.beta >= 0 ? beta * *c : 0.f);
      }
    }
  }
}

// NB output columns per pass: 8 (80 registers, 3 CTAs per SM) or 32 (one
// pass for the sketch width, 2 CTAs per SM)
template <int NB, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_gwarp(const GGroup* __restrict__ groups,
                                                    const GItem* __restrict__ items,
                                                    float* const* __restrict__ tab,
                                                    const int* const* __restrict__ rtab, int P,
                                                    int gbeg, int gend,
                                                    const double* __restrict__ coefs,
                                                    double* __restrict__ flops, int* err) {
  __shared__ __align__(16) float bsm[NT / 32][32 * (NB + 4)];   // KCH x (NB + 4) per warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = gbeg + blockIdx.x * (NT / 32) + warp;
  const int p = blockIdx.y;
  if (g >= gend) return;
  const GGroup G = groups[g];
  float* C = tab[G.cbuf * P + p];
  if (!C) return;
  const int m = dimv(G.m_st, G.m_rb, G.m_ri, rtab, P, p);
  const int n = dimv(G.n_st, G.n_rb, G.n_ri, rtab, P, p);
  if (m <= 0 || n <= 0) return;
  if (m > 64) {   // row panels only (the host launches this form for leaf-row stages)
    if (lane == 0) atomicOr(err, ERR_SHAPE);
    return;
  }
  C += G.coff;
  long long fl = 0;
  gwarp_panel<NB>(G, items, tab, rtab, P, p, m, n, C, coefs, bsm[warp], fl);
  if (flops && lane == 0 && fl > 0) atomicAdd(flops, (double)fl);
}

// Stages whose items read A transposed and B untransposed (or the sketch
// hash), so both operands are contiguous along the contraction: U^T V,
// Z^T Omega, X^T Q and the Grams.  Each warp owns a 4x4 output sub-tile and
// a slice of K; lanes stride K with coalesced loads straight into registers;
// the 16 sums are reduced with shuffles (and across K-slices through shared
// memory in a fixed order).  No staging, no integer division per element.
template <typename T, typename Acc>
__global__ void __launch_bounds__(NT) k_gdot(const GGroup* __restrict__ groups,
                                             const GItem* __restrict__ items,
                                             T* const* __restrict__ tab,
                                             const int* const* __restrict__ rtab, int P, int gbase,
                                             const double* __restrict__ coefs,
                                             double* __restrict__ flops) {
  const int p = blockIdx.y;
  const GGroup G = groups[gbase + blockIdx.x];
  T* C = tab[G.cbuf * P + p];
  if (!C) return;
  const int m = dimv(G.m_st, G.m_rb, G.m_ri, rtab, P, p);
  const int n = dimv(G.n_st, G.n_rb, G.n_ri, rtab, P, p);
  if (m <= 0 || n <= 0) return;
  C += G.coff;
  const Acc beta = G.beta >= 0 ? (Acc)coefs[G.beta] : Acc(0);
  const int TM = (m + 3) >> 2, TN = (n + 3) >> 2, ntile = TM * TN;
  const int KS = ntile >= 8 ? 1 : 8 / ntile;
  const int units = ntile * KS;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ Acc red[8 * 16];
  if (flops && threadIdx.x == 0) {
    double fl = 0.0;
    for (int it = G.ib; it < G.ie; ++it) {
      const GItem I = items[it];
      if (I.abuf >= 0 && !tab[I.abuf * P + p]) continue;
      if (I.bbuf >= 0 && !tab[I.bbuf * P + p]) continue;
      const int k = dimv(I.k_st, I.k_rb, I.k_ri, rtab, P, p);
      const int rows = dimv(I.r_st, I.r_rb, I.r_ri, rtab, P, p);
      if (k > 0 && rows > 0) fl += 2.0 * rows * n * k;
    }
    if (fl > 0.0) atomicAdd(flops, fl);
  }
  for (int u = warp; u < units; u += 8) {
    const int tile = u % ntile, ks = u / ntile;
    const int i0 = (tile % TM) * 4, j0 = (tile / TM) * 4;
    Acc acc[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[r][c] = Acc(0);
    for (int it = G.ib; it < G.ie; ++it) {
      const GItem I = items[it];
      if (I.guard0 >= 0 && !tab[I.guard0 * P + p]) continue;
      if (I.guard1 >= 0 && !tab[I.guard1 * P + p]) continue;
      const T* A = tab[I.abuf * P + p];
      if (!A) continue;
      A += I.aoff;
      const T* B = nullptr;
      const bool bo = I.bflags & FL_OMEGA;
      if (!bo) {
        B = tab[I.bbuf * P + p];
        if (!B) continue;
        B += I.boff;
      }
      const int k = dimv(I.k_st, I.k_rb, I.k_ri, rtab, P, p);
      const int rows = dimv(I.r_st, I.r_rb, I.r_ri, rtab, P, p);
      if (k <= 0 || rows <= 0) continue;
      const Acc cf = (Acc)coefs[I.coef];
      const T* ar[4];
      const T* bc[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) ar[r] = (i0 + r < rows) ? A + (int64_t)(i0 + r) * I.lda : nullptr;
#pragma unroll
      for (int c = 0; c < 4; ++c) bc[c] = (!bo && j0 + c < n) ? B + (int64_t)(j0 + c) * I.ldb : nullptr;
      for (int l = ks * 32 + lane; l < k; l += 32 * KS) {
        Acc av[4], bv[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) av[r] = ar[r] ? cf * (Acc)ar[r][l] : Acc(0);
        if (bo) {   // j0 is a multiple of 4: two hash words serve its 4 columns
          const uint32_t row = (uint32_t)(I.omega_row0 + l);
          const uint32_t b0 = omega_bits((uint32_t)I.seed, row, (uint32_t)j0 >> 1);
          const uint32_t b1 = omega_bits((uint32_t)I.seed, row, ((uint32_t)j0 >> 1) + 1);
#pragma unroll
          for (int c = 0; c < 4; ++c)
            bv[c] = (j0 + c < n) ? (Acc)omega_half(c < 2 ? b0 : b1, (uint32_t)(j0 + c)) : Acc(0);
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) bv[c] = bc[c] ? (Acc)bc[c][l] : Acc(0);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[r][c] += av[r] * bv[c];
      }
    }
    // all-lane butterfly reductions; lane e keeps element e
    Acc mine = Acc(0);
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      Acc v = acc[e & 3][e >> 2];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == e) mine = v;
    }
    if (KS == 1) {
      if (lane < 16) {
        const int i = i0 + (lane & 3), j = j0 + (lane >> 2);
        if (i < m && j < n) {
          T* c = C + i + (int64_t)j * G.ldc;
          Acc v = mine;
          if (G.beta >= 0) v += beta * (Acc)(*c);
          *c = (T)v;
        }
      }
    } else if (lane < 16) {
      red[u * 16 + lane] = mine;
    }
  }
  if (KS > 1) {
    __syncthreads();
    for (int t = threadIdx.x; t < ntile * 16; t += NT) {
      const int tile = t >> 4, e = t & 15;
      Acc v = Acc(0);
      for (int ks = 0; ks < KS; ++ks) v += red[(tile + ks * ntile) * 16 + e];
      const int i0 = (tile % TM) * 4, j0 = (tile / TM) * 4;
      const int i = i0 + (e & 3), j = j0 + (e >> 2);
      if (i < m && j < n) {
        T* c = C + i + (int64_t)j * G.ldc;
        if (G.beta >= 0) v += beta * (Acc)(*c);
        *c = (T)v;
      }
    }
  }
}

// Warp-per-group form of the dot kernel for stages made of very many tiny
// groups (U^T V, Z^T Omega, X^T Q): eight groups per CTA, each warp walks
// its group's output in 4 x 8 tiles with lanes striding the contraction;
// no shared memory, no barriers.
// TM output rows per tile (4, or 8: one pass over the items covers ranks up
// to 8 and every sketch column is generated once per row tile)
template <typename T, typename Acc, int TM>
__global__ void __launch_bounds__(NT, sizeof(Acc) == 4 ? (TM == 4 ? 4 : 2) : 1) k_gdot_warp(const GGroup* __restrict__ groups,
                                                  const GItem* __restrict__ items,
                                                  T* const* __restrict__ tab,
                                                  const int* const* __restrict__ rtab, int P,
                                                  int gbase, int gend,
                                                  const double* __restrict__ coefs,
                                                  double* __restrict__ flops) {
  const int p = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gi = gbase + blockIdx.x * (NT / 32) + warp;
  if (gi >= gend) return;
  const GGroup G = groups[gi];
  T* C = tab[G.cbuf * P + p];
  if (!C) return;
  const int m = dimv(G.m_st, G.m_rb, G.m_ri, rtab, P, p);
  const int n = dimv(G.n_st, G.n_rb, G.n_ri, rtab, P, p);
  if (m <= 0 || n <= 0) return;
  C += G.coff;
  const Acc beta = G.beta >= 0 ? (Acc)coefs[G.beta] : Acc(0);
  long long fl = 0;
  for (int i0 = 0; i0 < m; i0 += TM) {
    for (int j0 = 0; j0 < n; j0 += 8) {
      Acc acc[TM][8];
#pragma unroll
      for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < 8; ++c) acc[r][c] = Acc(0);
      for (int it = G.ib; it < G.ie; ++it) {
        const GItem I = items[it];
        if (I.guard0 >= 0 && !tab[I.guard0 * P + p]) continue;
        if (I.guard1 >= 0 && !tab[I.guard1 * P + p]) continue;
        const T* A = tab[I.abuf * P + p];
        if (!A) continue;
        A += I.aoff;
        const bool bo = I.bflags & FL_OMEGA;
        const T* B = nullptr;
        if (!bo) {
          B = tab[I.bbuf * P + p];
          if (!B) continue;
          B += I.boff;
        }
        const int k = dimv(I.k_st, I.k_rb, I.k_ri, rtab, P, p);
        const int rows = dimv(I.r_st, I.r_rb, I.r_ri, rtab, P, p);
        if (k <= 0 || rows <= 0) continue;
        if (i0 == 0 && j0 == 0) fl += 2LL * rows * n * k;
        const Acc cf = (Acc)coefs[I.coef];
        const T* ar[TM];
#pragma unroll
        for (int r = 0; r < TM; ++r) ar[r] = (i0 + r < rows) ? A + (int64_t)(i0 + r) * I.lda : nullptr;
        for (int l = lane; l < k; l += 32) {
          Acc av[TM], bv[8];
#pragma unroll
          for (int r = 0; r < TM; ++r) av[r] = ar[r] ? cf * (Acc)ar[r][l] : Acc(0);
          if (bo) {
            const uint32_t row = (uint32_t)(I.omega_row0 + l);
#pragma unroll
            for (int w = 0; w < 4; ++w) {
              const uint32_t bits = omega_bits((uint32_t)I.seed, row, ((uint32_t)j0 >> 1) + w);
              bv[2 * w] = (j0 + 2 * w < n) ? (Acc)omega_half(bits, 0u) : Acc(0);
              bv[2 * w + 1] = (j0 + 2 * w + 1 < n) ? (Acc)omega_half(bits, 1u) : Acc(0);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 8; ++c)
              bv[c] = (j0 + c < n) ? (Acc)B[l + (int64_t)(j0 + c) * I.ldb] : Acc(0);
          }
#pragma unroll
          for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[r][c] += av[r] * bv[c];
        }
      }
      // transposing reduction per 32 tile elements (element e = row e % TM,
      // column e / TM): 32 sums over the 32 lanes, lane e ending with element
      // e (recursive halving, 31 shuffles instead of 32 x 5)
#pragma unroll
      for (int h = 0; h < TM / 4; ++h) {
        Acc v[32];
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = acc[(32 * h + e) % TM][(32 * h + e) / TM];
#pragma unroll
        for (int sft = 16; sft > 0; sft >>= 1) {
          const bool up = (lane & sft) != 0;
#pragma unroll
          for (int e = 0; e < sft; ++e) {
            const Acc keep = up ? v[e + sft] : v[e];
            const Acc send = up ? v[e] : v[e + sft];
            v[e] = keep + __shfl_xor_sync(0xffffffffu, send, sft);
          }
        }
        const int e = 32 * h + lane;
        const int i = i0 + e % TM, j = j0 + e / TM;
        if (i < m && j < n) {
          T* c = C + i + (int64_t)j * G.ldc;
          Acc w = v[0];
          if (G.beta >= 0) w += beta * (Acc)(*c);
          *c = (T)w;
        }
      }
    }
  }
  if (flops && lane == 0 && fl > 0) atomicAdd(flops, (double)fl);
}

// The inner products of a low-rank target with its common right factor: the
// sketch rows S_i = Z_i^T Omega (SK) or the projections P_i = X_i^T Q of all
// summed terms i.  One CTA per target holds the common factor (generated once,
// instead of once per term, for Omega) in shared memory, row by row; a warp takes 8 columns of
// one Z_i at a time: 32 rows of them pass through the warp's own shared
// slice, and each lane accumulates 8 products of its own output column -- no
// shuffles per output, 3 shared loads per 8 multiply-adds.  Narrow outputs (W < 32
// columns) split the 32 rows over the lanes' spare groups.  Sums are per 32 rows, then
// over the blocks.  Factors of more than 512 (FP64: 256) rows go through in blocks, added
// in global memory.  n = 64 setup: sketches 33 -> 20 ms, projections 39 -> 22 ms (n = 80: 118 -> 59, 100 -> 60)
// against one warp per term with lanes along the rows.
// rows of the common factor held at a time
template <typename T>
__host__ __device__ constexpr int tdr() { return sizeof(T) == 4 ? 512 : 256; }
constexpr int TDI = 64;        // terms resolved at a time

template <typename T>
constexpr size_t tdot_smem(int rows, int p) {
  const int w = p <= 8 ? 8 : p <= 16 ? 16 : p <= 32 ? 32 : 64;
  return ((size_t)(rows < tdr<T>() ? rows : tdr<T>()) * (w + 1) + (NT / 32) * 32 * 8) * sizeof(T) + 16;
}

template <typename T, bool SK>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 4 : 2)
    k_tdot(const TInfo* __restrict__ tis, const int* __restrict__ order,
           const GGroup* __restrict__ groups, const GItem* __restrict__ items,
           T* const* __restrict__ tab, const int* const* __restrict__ rtab, int P, int scr_buf,
           int scr_rbuf, double* __restrict__ flops) {
  const int p = blockIdx.y;
  const TInfo ti = tis[order[blockIdx.x]];
  T* scr = tab[scr_buf * P + p];
  const int* rs = rtab[scr_rbuf * P + p];
  const int gb = SK ? ti.s_beg : ti.x_beg, ge = SK ? ti.s_end : ti.x_end;
  if (!scr || !rs || ge <= gb) return;
  const int nc = SK ? ti.p : rs[ti.r_ri];       // output columns
  if (nc <= 0) return;
  const int rows = SK ? ti.n : ti.m;            // rows of the common factor
  const int W = nc <= 8 ? 8 : nc <= 16 ? 16 : nc <= 32 ? 32 : 64, LD = W + 1;
  extern __shared__ __align__(16) unsigned char td_raw[];
  T* zsall = reinterpret_cast<T*>(td_raw);      // 32 x 8 per warp
  T* F = zsall + (NT / 32) * 32 * 8;            // F(row, col) = F[row * LD + col]
  struct Term {
    const T* Z;
    T* C;
    int k, rows, lda, ldc, off;
  };
  __shared__ Term term[TDI];
  __shared__ int uoff[TDI + 1];                 // first unit (8 columns of Z) of each term
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  T* zs = zsall + warp * 32 * 8;
  const int w32 = min(W, 32), col = lane & (w32 - 1), sub = lane / w32, RS = 32 / w32;
  for (int f0 = 0; f0 < rows; f0 += tdr<T>()) {
    const int fr = min(tdr<T>(), rows - f0);
    __syncthreads();
    if (SK) {
      for (int e = tid; e < fr * (W / 2); e += NT) {
        const int r = e / (W / 2), c = e - r * (W / 2);     // (W a power of two)
        if (2 * c < nc) {
          const uint32_t b = omega_bits((uint32_t)ti.seed, (uint32_t)(f0 + r), (uint32_t)c);
          F[r * LD + 2 * c] = (T)omega_half(b, 0u);
          F[r * LD + 2 * c + 1] = (T)omega_half(b, 1u);
        }
      }
    } else {
      const T* Q = scr + ti.y_off + f0;
      for (int c = warp; c < nc; c += NT / 32)
        for (int r = lane; r < fr; r += 32) F[r * LD + c] = Q[r + (int64_t)c * rows];
    }
    for (int base = gb; base < ge; base += TDI) {
      const int cnt = min(TDI, ge - base);
      __syncthreads();
      if (tid < TDI) {
        Term R{};
        if (tid < cnt) {
          const GGroup G = groups[base + tid];
          const GItem I = items[G.ib];
          const T* Z = tab[I.abuf * P + p];
          if (Z) {
            R.Z = Z + I.aoff;
            R.C = scr + G.coff;
            R.k = dimv(G.m_st, G.m_rb, G.m_ri, rtab, P, p);
            R.rows = I.k_st;
            R.off = SK ? I.omega_row0 : (int)(I.boff - ti.y_off);
            R.lda = I.lda; R.ldc = G.ldc;
            if (flops && f0 == 0 && blockIdx.z == 0 && R.k > 0)
              atomicAdd(flops, 2.0 * R.rows * nc * R.k);
          }
          // (a term without rows in this block has no units here)
          if (R.k <= 0 || R.off >= f0 + fr || R.off + R.rows <= f0) R.k = 0;
        }
        term[tid] = R;
        int inc = (R.k + 7) >> 3;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += v;
        }
        uoff[tid + 1] = inc;
        if (tid == 0) uoff[0] = 0;
      }
      __syncthreads();
      const int half = uoff[32], units = half + uoff[TDI];
      for (int u = warp + (NT / 32) * blockIdx.z; u < units; u += (NT / 32) * gridDim.z) {
        // the term of unit u (the second half's offsets are its own)
        int lo, hi, add;
        if (u < half) { lo = 0; hi = 32; add = 0; } else { lo = 32; hi = TDI; add = half; }
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if ((mid == 32 ? 0 : uoff[mid]) <= u - add) lo = mid;
          else hi = mid;
        }
        const Term R = term[lo];
        const int i0 = 8 * (u - add - (lo == 32 ? 0 : uoff[lo]));
        const int kc = min(8, R.k - i0);
        // rows [l0, l1) of the term lie in this block; F row of term row l: l + sh
        const int l0 = max(0, f0 - R.off), l1 = min(R.rows, f0 + fr - R.off), sh = R.off - f0;
        const T* Z = R.Z + (int64_t)i0 * R.lda;
        for (int h = 0; h < W; h += 32) {
          T acc[8], z[8];
#pragma unroll
          for (int c = 0; c < 8; ++c) acc[c] = T(0);
#pragma unroll
          for (int c = 0; c < 8; ++c)
            z[c] = (c < kc && l0 + lane < l1) ? Z[l0 + lane + (int64_t)c * R.lda] : T(0);
          for (int l = l0; l < l1; l += 32) {
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 8; c += 16 / (int)sizeof(T)) {
              if (sizeof(T) == 4)
                *reinterpret_cast<float4*>(zs + lane * 8 + c) =
                    make_float4((float)z[c], (float)z[c + 1], (float)z[c + 2], (float)z[c + 3]);
              else
                *reinterpret_cast<double2*>(zs + lane * 8 + c) = make_double2((double)z[c], (double)z[c + 1]);
            }
            __syncwarp();
#pragma unroll
            for (int c = 0; c < 8; ++c)   // the next rows, while these are multiplied
              z[c] = (c < kc && l + 32 + lane < l1) ? Z[l + 32 + lane + (int64_t)c * R.lda] : T(0);
            const int nr = min(32, l1 - l), per = 32 / RS;
            const T* f = F + (int64_t)(l + sh + sub * per) * LD + h + col;
            const T* zr = zs + sub * per * 8;
            const int my = min(per, nr - sub * per);
            T s[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) s[c] = T(0);
            if (kc > 4) {
#pragma unroll 4
              for (int r = 0; r < my; ++r) {
                T a[4], b[4];
                ld4(zr + r * 8, a);
                ld4(zr + r * 8 + 4, b);
                const T t = f[r * LD];
#pragma unroll
                for (int c = 0; c < 4; ++c) { s[c] += a[c] * t; s[c + 4] += b[c] * t; }
              }
            } else {
#pragma unroll 4
              for (int r = 0; r < my; ++r) {
                T a[4];
                ld4(zr + r * 8, a);
                const T t = f[r * LD];
#pragma unroll
                for (int c = 0; c < 4; ++c) s[c] += a[c] * t;
              }
            }
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] += s[c];
          }
          for (int o = w32; o < 32; o <<= 1)
#pragma unroll
            for (int c = 0; c < 8; ++c) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
          // through the warp's slice: the 8 rows of a column are contiguous
          __syncwarp();
          if (sub == 0)
#pragma unroll
            for (int c = 0; c < 8; ++c) zs[col * 8 + c] = acc[c];
          __syncwarp();
          const int i = lane & 7;
          for (int j = lane >> 3; j < w32; j += 4) {
            if (i >= kc || h + j >= nc) continue;
            T* c = R.C + i0 + i + (int64_t)(h + j) * R.ldc;
            const T v = zs[j * 8 + i];
            *c = l0 > 0 ? *c + v : v;
          }
        }
      }
    }
  }
}

}  // namespace

template <typename T>
void launch_tdot(const Plan& pl, bool sketch, T* const* d_tab, const int* const* d_rtab, int P,
                 cudaStream_t st, double* d_fl) {
  const int nt = (int)pl.torder.size();
  if (nt <= 0 || P <= 0) return;
  auto kern = sketch ? k_tdot<T, true> : k_tdot<T, false>;
  auto smem = [&](int q) {
    const TInfo& ti = pl.targets[pl.torder[q]];
    return tdot_smem<T>(std::max(ti.m, ti.n), ti.p);
  };
  // targets by increasing size: those that leave room for 4 (double: 2) CTAs per
  // SM first, then the larger ones; few targets go in one launch
  const size_t small = sizeof(T) == 4 ? 56320 : 112640;
  const bool few = (int64_t)nt * P <= device_sm_count();
  ACR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)tdot_smem<T>(tdr<T>(), 64)));
  for (int beg = 0; beg < nt;) {
    int end = nt;
    if (!few && smem(beg) <= small)
      for (end = beg + 1; end < nt && smem(end) <= small; ++end) {}
    size_t need = 0;
    int rows = 0;
    for (int q = beg; q < end; ++q) {
      need = std::max(need, smem(q));
      rows = std::max({rows, pl.targets[pl.torder[q]].m, pl.targets[pl.torder[q]].n});
    }
    // few targets: their units dealt to up to 8 CTAs each (a unit's sums are the
    // same wherever it runs; with more than one block of rows its partial sums
    // meet in global memory and stay in one CTA)
    int z = 1;
    if (rows <= tdr<T>())
      while (z < 8 && (int64_t)(end - beg) * P * z < 2 * device_sm_count()) z *= 2;
    for (int t0 = beg; t0 < end; t0 += 65535) {
      const dim3 grid(std::min(65535, end - t0), P, z);
      kern<<<grid, NT, need, st>>>((const TInfo*)pl.d_targets, (const int*)pl.d_torder + t0,
                                   (const GGroup*)pl.d_groups, (const GItem*)pl.d_items, d_tab,
                                   d_rtab, P, 3 * pl.nroles, pl.nroles, d_fl);
      ACR_LAUNCHED(1);
    }
    beg = end;
  }
}

template <typename T>
void launch_gbundle(const Plan& pl, int bbeg, int bend, T* const* d_tab, const int* const* d_rtab,
                    int P, const double* d_coefs, cudaStream_t st, double* d_fl) {
  if (bend <= bbeg || P <= 0) return;
  if (cat_bytes<T>() > 48 * 1024)
    ACR_CUDA(cudaFuncSetAttribute(k_gbundle<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  cat_bytes<T>()));
  for (int b0 = bbeg; b0 < bend; b0 += 65535) {
    const dim3 grid(std::min(65535, bend - b0), P);
    k_gbundle<T><<<grid, NT, cat_bytes<T>(), st>>>(
        (const int*)pl.d_bundles + 2 * b0, (const GGroup*)pl.d_groups, (const GItem*)pl.d_items,
        d_tab, d_rtab, P, d_coefs, d_fl);
    ACR_LAUNCHED(1);
  }
}

template <typename T>
void launch_ggemm(const Plan& pl, int gbeg, int gend, T* const* d_tab, const int* const* d_rtab,
                  int P, const double* d_coefs, cudaStream_t st, double* d_fl, int tag,
                  int variant, int* d_err, int nwide) {
  int ng = gend - gbeg;
  if (ng <= 0 || P <= 0) return;
  if ((variant == 2 || variant == 3 || variant == 4) && nwide > 0 && sizeof(T) == 4 &&
      !tag_is_dot(tag)) {
    // the stage's wide groups (64-column outputs: dense products) in the
    // staged CTA kernel (shape 2) or on the tensor cores (shape 3), the rest
    // one warp per group
    const int w = std::min(nwide, ng);
    if (variant == 3 && d_err)
      launch_ggemm_tc(pl, gbeg, gbeg + w, (float* const*)d_tab, d_rtab, P, d_coefs, st, d_fl,
                      d_err);
    else
      launch_ggemm<T>(pl, gbeg, gbeg + w, d_tab, d_rtab, P, d_coefs, st, d_fl, tag, 0, d_err, 0);
    launch_ggemm<T>(pl, gbeg + w, gend, d_tab, d_rtab, P, d_coefs, st, d_fl, tag,
                    variant == 4 ? 4 : 2, d_err, 0);
    return;
  }
  if (variant == 3) variant = 2;   // no wide groups: shape 3 is shape 2
  using Acc = T;
  if (cat_bytes<T>() > 48 * 1024)
    ACR_CUDA(cudaFuncSetAttribute(k_gcat<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  cat_bytes<T>()));
  // A stage of few groups per plane leaves most of the SMs idle whenever few
  // planes are left: its outputs' columns are then split over 2 or 4 CTAs.  (By the
  // plan alone, not by P: a plane's result must not depend on the batch.)
  const int zsplit = 4 * ng <= PART_SMS ? 4 : 2 * ng <= PART_SMS ? 2 : 1;
  const int maxg = 65535;
  for (int g0 = 0; g0 < ng; g0 += maxg) {
    dim3 grid(std::min(maxg, ng - g0), P);
    const GGroup* gr = (const GGroup*)pl.d_groups;
    const GItem* it = (const GItem*)pl.d_items;
    // warp per group for the inner products, and for the small-output
    // sketch / projection stages where the multiply type is float (the FP64
    // instance of the warp kernel holds ~200 registers: one CTA per SM)
    // Variant 0: k_gcat.  Variant 1 swaps the warp-per-group and CTA-per-group
    // inner-product kernels and takes k_ggemm, item by item, for the others
    // (float: 3 CTAs per SM and 80 registers; double: half the staging per
    // K-step).  Variant 2 (float, non-dot stages) runs
    // one warp per group (k_gwarp, 8 columns per pass); variant 3 as 2, with
    // the wide groups on the tensor cores; variant 4 as 2 with 32 columns per
    // pass; variant 5 (float, inner-product stages) 8 x 8 warp tiles.
    const bool warp_dot = (tag == TAG_M || (sizeof(T) == 4 && (tag == TAG_S || tag == TAG_P)));
    if ((variant == 2 || variant == 4) && sizeof(T) == 4 && d_err && !tag_is_dot(tag)) {
      const int cnt = std::min(maxg, ng - g0);
      dim3 gw((cnt + NT / 32 - 1) / (NT / 32), P);
      if (variant == 4)
        k_gwarp<32, 2><<<gw, NT, 0, st>>>(gr, it, (float* const*)d_tab, d_rtab, P, gbeg + g0,
                                          gbeg + g0 + cnt, d_coefs, d_fl, d_err);
      else
        k_gwarp<8, 3><<<gw, NT, 0, st>>>(gr, it, (float* const*)d_tab, d_rtab, P, gbeg + g0,
                                         gbeg + g0 + cnt, d_coefs, d_fl, d_err);
    } else if (tag_is_dot(tag) && variant == 5 && sizeof(T) == 4) {
      const int cnt = std::min(maxg, ng - g0);
      dim3 gw((cnt + NT / 32 - 1) / (NT / 32), P);
      k_gdot_warp<T, Acc, 8><<<gw, NT, 0, st>>>(gr, it, d_tab, d_rtab, P, gbeg + g0,
                                                gbeg + g0 + cnt, d_coefs, d_fl);
    } else if (tag_is_dot(tag) && (warp_dot != (variant == 1))) {
      const int cnt = std::min(maxg, ng - g0);
      dim3 gw((cnt + NT / 32 - 1) / (NT / 32), P);
      k_gdot_warp<T, Acc, 4><<<gw, NT, 0, st>>>(gr, it, d_tab, d_rtab, P, gbeg + g0,
                                                gbeg + g0 + cnt, d_coefs, d_fl);
    } else if (tag_is_dot(tag))
      k_gdot<T, Acc><<<grid, NT, 0, st>>>(gr, it, d_tab, d_rtab, P, gbeg + g0, d_coefs, d_fl);
    else if (variant == 1 && sizeof(Acc) == 4)
      k_ggemm<T, Acc, STAGE_BYTES, 3>
          <<<grid, NT, 0, st>>>(gr, it, d_tab, d_rtab, P, gbeg + g0, d_coefs, d_fl);
    else if (variant == 1)
      k_ggemm<T, Acc, STAGE_BYTES / 2, 2>
          <<<grid, NT, 0, st>>>(gr, it, d_tab, d_rtab, P, gbeg + g0, d_coefs, d_fl);
    else
      k_gcat<T><<<dim3(grid.x, grid.y, zsplit), NT, cat_bytes<T>(), st>>>(gr, it, d_tab, d_rtab, P,
                                                                          gbeg + g0, d_coefs, d_fl);
    ACR_LAUNCHED(1);
  }
}

template void launch_tdot<double>(const Plan&, bool, double* const*, const int* const*, int,
                                  cudaStream_t, double*);
template void launch_tdot<float>(const Plan&, bool, float* const*, const int* const*, int,
                                 cudaStream_t, double*);
template void launch_gbundle<double>(const Plan&, int, int, double* const*, const int* const*, int,
                                     const double*, cudaStream_t, double*);
template void launch_gbundle<float>(const Plan&, int, int, float* const*, const int* const*, int,
                                    const double*, cudaStream_t, double*);
template void launch_ggemm<double>(const Plan&, int, int, double* const*, const int* const*, int,
                                   const double*, cudaStream_t, double*, int, int, int*, int);
template void launch_ggemm<float>(const Plan&, int, int, float* const*, const int* const*, int,
                                  const double*, cudaStream_t, double*, int, int, int*, int);

}  // namespace acr
