// Check of the recompression cores (acr_core_kernels.cu) on their own: the basis
// kernel on sketches whose exact ranks and ranges are known in FP64, the core kernel on
// factors with given singular values.  Prints one line per case; exits 1 on a failure.
// Links the library; test infrastructure only.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "acr_internal.h"
#include "acr_plan.h"

using namespace acr;

namespace {

bool fail = false;
std::mt19937_64 rng(11);
double rnd() { return std::uniform_real_distribution<double>(-1.0, 1.0)(rng); }

void cu(cudaError_t e) {
  if (e != cudaSuccess) { std::printf("CUDA: %s\n", cudaGetErrorString(e)); std::exit(2); }
}
template <typename V>
V* dev(const std::vector<V>& h) {
  V* p = nullptr;
  cu(cudaMalloc(&p, std::max<size_t>(h.size(), 1) * sizeof(V)));
  cu(cudaMemcpy(p, h.data(), h.size() * sizeof(V), cudaMemcpyHostToDevice));
  return p;
}
template <typename V>
std::vector<V> host(const V* p, size_t n) {
  std::vector<V> h(n);
  cu(cudaDeviceSynchronize());
  cu(cudaMemcpy(h.data(), p, n * sizeof(V), cudaMemcpyDeviceToHost));
  return h;
}
void check(const char* what, double got, double bound) {
  const bool ok = got <= bound;
  if (!ok) fail = true;
  std::printf("  %s %.3e (at most %.1e)%s", what, got, bound, ok ? "" : " FAIL");
}

// One target of m x p sketch and n x p B^T in one plane's scratch; the second plane of
// the launch is absent.
template <typename T>
struct Setup {
  Plan pl;
  TInfo ti{};
  std::vector<T*> tab;
  std::vector<int*> rtab;
  T* scr = nullptr;
  T *U = nullptr, *V = nullptr;
  int *rs = nullptr, *crank = nullptr, *err = nullptr;
  T** d_tab = nullptr;
  int** d_rtab = nullptr;
  Setup(int m, int n, int p, const std::vector<T>& scratch, int64_t bt_off, int r) {
    ti.m = m; ti.n = n; ti.p = p;
    ti.y_off = 0; ti.bt_off = bt_off;
    pl.nroles = 1;
    pl.targets = {ti};
    pl.torder = {0};
    pl.max_p = p;
    pl.d_targets = dev(pl.targets);
    pl.d_torder = dev(pl.torder);
    scr = dev(scratch);
    U = dev(std::vector<T>((size_t)m * p));
    V = dev(std::vector<T>((size_t)n * p));
    rs = dev(std::vector<int>{r});
    crank = dev(std::vector<int>{-1});
    err = dev(std::vector<int>{0});
    tab = {nullptr, nullptr, U, nullptr, V, nullptr, scr, nullptr};   // [buffer][plane]
    rtab = {crank, nullptr, rs, nullptr};
    d_tab = dev(tab);
    d_rtab = dev(rtab);
  }
};

// Columns a_k y_0 + delta_k e_k, delta_k in steps of 1e-3 across tau, and a scale of the
// whole sketch: as many of them as exceed tau in exact arithmetic belong to the basis.
void orth_ranks(int m, int p, double tau, double scale) {
  std::vector<float> Y((size_t)m * p, 0.f);
  for (int i = p; i < m; ++i) Y[i] = (float)(scale * rnd());
  double n0 = 0.0;
  for (int i = 0; i < m; ++i) n0 += (double)Y[i] * Y[i];
  n0 = std::sqrt(n0);
  for (int k = 1; k < p; ++k) {
    const double a = 0.3 + 0.6 * k / p;
    for (int i = p; i < m; ++i) Y[i + (size_t)k * m] = (float)(a * Y[i]);
    Y[k + (size_t)k * m] = (float)(tau * n0 * (1.0 + 1e-3 * (k - p / 2 - 0.5)));
  }
  // pivoted Gram-Schmidt in FP64 (twice)
  std::vector<double> W(Y.begin(), Y.end());
  std::vector<char> used(p, 0);
  int rank = 0;
  double near = 1.0;
  for (int j = 0; j < p; ++j) {
    int q = -1;
    double best = -1.0;
    for (int c = 0; c < p; ++c) {
      if (used[c]) continue;
      double s = 0.0;
      for (int i = 0; i < m; ++i) s += W[i + (size_t)c * m] * W[i + (size_t)c * m];
      if (s > best) { best = s; q = c; }
    }
    const double rel = std::sqrt(best) / (tau * n0);
    near = std::min(near, std::fabs(rel - 1.0));
    if (j > 0 && rel <= 1.0) break;
    used[q] = 1;
    ++rank;
    for (int pass = 0; pass < 2; ++pass)
      for (int c = 0; c < p; ++c) {
        if (used[c]) continue;
        double s = 0.0;
        for (int i = 0; i < m; ++i) s += W[i + (size_t)c * m] * W[i + (size_t)q * m];
        for (int i = 0; i < m; ++i) W[i + (size_t)c * m] -= s / best * W[i + (size_t)q * m];
      }
  }
  std::vector<float> scratch(Y);
  scratch.resize((size_t)2 * m * p, 0.f);
  Setup<float> su(m, m, p, scratch, (int64_t)m * p, 0);
  launch_orth(su.pl, tau, su.d_tab, su.d_rtab, 2, 0, nullptr);
  const int r = host(su.rs, 1)[0];
  const std::vector<float> Q = host(su.scr, (size_t)m * p);
  double orth = 0.0, range = 0.0;
  for (int a = 0; a < r; ++a)
    for (int b = 0; b <= a; ++b) {
      double s = 0.0;
      for (int i = 0; i < m; ++i) s += (double)Q[i + (size_t)a * m] * Q[i + (size_t)b * m];
      orth = std::max(orth, std::fabs(s - (a == b)));
    }
  for (int c = 0; c < p; ++c) {
    std::vector<double> y(Y.begin() + (size_t)c * m, Y.begin() + (size_t)(c + 1) * m);
    for (int pass = 0; pass < 2; ++pass)
      for (int a = 0; a < r; ++a) {
        double s = 0.0;
        for (int i = 0; i < m; ++i) s += y[i] * Q[i + (size_t)a * m];
        for (int i = 0; i < m; ++i) y[i] -= s * Q[i + (size_t)a * m];
      }
    double s = 0.0;
    for (double v : y) s += v * v;
    range = std::max(range, std::sqrt(s) / n0);
  }
  std::printf("orth m %d p %d tau %.0e scale %.0e: rank %d, exact %d (nearest %.1e)%s", m, p, tau,
              scale, r, rank, near, r == rank ? "" : " FAIL");
  if (r != rank) fail = true;
  // Q's entries rounded to float: 2^-24 of each of the two vectors, and the basis' own 3e-8
  check("orthogonality", orth, 2 * 0x1p-24 + 3e-8);
  // what is left out (tau), and the rounding of Q's entries against a column
  check("range", range, tau * 1.0001 + 0x1p-23);
  std::printf("\n");
}

// B^T = X S W^T (n x r) with given singular values, Q (m x r) orthonormal: the factors
// U V^T are Q B without the singular values up to eps, and U is orthonormal.
template <typename T>
void core(int m, int n, int r, double eps, double ratio) {
  auto ortho = [&](int rows, int cols) {
    std::vector<double> A((size_t)rows * cols);
    for (double& x : A) x = rnd();
    for (int c = 0; c < cols; ++c)
      for (int pass = 0; pass < 2; ++pass) {
        for (int q = 0; q < c; ++q) {
          double s = 0.0;
          for (int i = 0; i < rows; ++i) s += A[i + (size_t)c * rows] * A[i + (size_t)q * rows];
          for (int i = 0; i < rows; ++i) A[i + (size_t)c * rows] -= s * A[i + (size_t)q * rows];
        }
        double s = 0.0;
        for (int i = 0; i < rows; ++i) s += A[i + (size_t)c * rows] * A[i + (size_t)c * rows];
        for (int i = 0; i < rows; ++i) A[i + (size_t)c * rows] /= std::sqrt(s);
      }
    return A;
  };
  const std::vector<double> Q = ortho(m, r), X = ortho(n, r), W = ortho(r, r);
  std::vector<T> scratch((size_t)(m + n) * r);
  for (size_t e = 0; e < Q.size(); ++e) scratch[e] = (T)Q[e];
  int keep = 0;
  std::vector<double> sv(r);
  for (int q = 0; q < r; ++q) {
    sv[q] = std::pow(ratio, q);
    if (sv[q] > eps) ++keep;
  }
  for (int i = 0; i < n; ++i)
    for (int j = 0; j < r; ++j) {
      double s = 0.0;
      for (int q = 0; q < r; ++q) s += X[i + (size_t)q * n] * sv[q] * W[j + (size_t)q * r];
      scratch[(size_t)m * r + i + (size_t)j * n] = (T)s;
    }
  Setup<T> su(m, n, r, scratch, (int64_t)m * r, r);
  launch_core<T>(su.pl, eps, r, 0, su.d_tab, su.d_rtab, 2, su.err, 0);
  const int k = host(su.crank, 1)[0];
  const std::vector<T> U = host(su.U, (size_t)m * r), V = host(su.V, (size_t)n * r);
  double orth = 0.0, rec = 0.0;
  for (int a = 0; a < k; ++a)
    for (int b = 0; b <= a; ++b) {
      double s = 0.0;
      for (int i = 0; i < m; ++i) s += (double)U[i + (size_t)a * m] * U[i + (size_t)b * m];
      orth = std::max(orth, std::fabs(s - (a == b)));
    }
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < n; ++j) {
      double s = 0.0;
      for (int q = 0; q < k; ++q) s += (double)U[i + (size_t)q * m] * V[j + (size_t)q * n];
      for (int l = 0; l < r; ++l)
        s -= (double)scratch[i + (size_t)l * m] * scratch[(size_t)m * r + j + (size_t)l * n];
      rec += s * s;
    }
  const bool f64 = sizeof(T) == 8;
  const double u = f64 ? 0x1p-53 : 0x1p-24;
  std::printf("core %s m %d n %d r %d eps %.0e: rank %d, exact %d%s", f64 ? "fp64" : "float", m, n, r,
              eps, k, keep, k == keep ? "" : " FAIL");
  if (k != keep) fail = true;
  // a row of U or V sums r products, U's entries and those of W are rounded: (r + 4) u of
  // the norms; FP64's rotations themselves ~7 sweeps of r - 1 rounds at 3 u
  const double c = (r + 4) * u * 4 + (f64 ? 21.0 * r * u : 0.0);
  check("orthogonality", orth, c);
  double left = 0.0;
  for (int q = k; q < r; ++q) left += sv[q] * sv[q];
  double total = 0.0;
  for (double s : sv) total += s * s;
  check("reconstruction", std::sqrt(rec), std::sqrt(left) * 1.0001 + c * std::sqrt(total));
  std::printf("\n");
}

}  // namespace

int main() {
  for (double scale : {1.0, 1e-25, 1e25}) {
    orth_ranks(36, 27, 1e-6, scale);
    orth_ranks(64, 32, 1e-5, scale);
    orth_ranks(100, 56, 1e-6, scale);
    orth_ranks(144, 40, 1e-5, scale);    // 47.5 KB, beside the kernel's own arrays
    orth_ranks(288, 42, 1e-5, scale);
    orth_ranks(400, 32, 1e-6, scale);
    orth_ranks(800, 34, 1e-5, scale);    // a cluster's, with rows to spare
    orth_ranks(1152, 56, 1e-5, scale);
  }
  orth_ranks(1001, 30, 1e-5, 1.0);       // a cluster's, whose last CTA has fewer rows
  orth_ranks(4096, 56, 1e-5, 1.0);       // beyond a cluster's shared memory
  for (int r : {1, 2, 3, 12, 31, 56}) {
    core<double>(64, 50, r, 1e-2, 0.5);
    core<double>(100, 300, r, 1e-7, 0.8);
    core<float>(64, 50, r, 1e-2, 0.5);
    core<float>(100, 300, r, 1e-5, 0.8);
  }
  for (int k = 0; k < 6; ++k) core<float>(100, 300, 56, 1e-5, 0.8);   // eigenvalues down to eps^2
  std::printf(fail ? "FAILED\n" : "all ok\n");
  return fail ? 1 : 0;
}
