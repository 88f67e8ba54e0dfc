// The plans as the engine builds them (PlanParams::fused and fused_core), executed on the CPU
// in FP64 the way the kernels read them: sketches and projections by each target's own
// range of groups, factor products by bundles (the items of the bundle's first group
// give the A operands of all), bases and cores from the targets' records.  The operations
// and their exact results are those of plan_emulator.cpp.  Also checks what the kernels
// rely on: bundles that cover a factor stage's narrow groups once, target ranges that
// cover the sketch and projection stages once, sizes in order.
#define main plan_emulator_main
#include "plan_emulator.cpp"
#undef main

namespace {

const double signs[3] = {1.0, -1.0, 1.0};

double* buf(int b) { return tab[b]; }

// sum over items of coef A B into a C of the group; A from the items of `lead`
void product(const Plan& pl, const GGroup& G, const GGroup& lead) {
  double* C = buf(G.cbuf);
  if (!C) return;
  const int m = dimv(lead.m_st, lead.m_rb, lead.m_ri), n = dimv(G.n_st, G.n_rb, G.n_ri);
  if (m <= 0 || n <= 0) return;
  C += G.coff;
  std::vector<double> acc((size_t)m * n, 0.0);
  for (int e = 0; e < G.ie - G.ib; ++e) {
    const GItem &I = pl.items[lead.ib + e], &J = pl.items[G.ib + e];
    if ((I.guard0 >= 0 && !buf(I.guard0)) || (I.guard1 >= 0 && !buf(I.guard1))) continue;
    const double* A = I.abuf >= 0 ? buf(I.abuf) : nullptr;
    const double* B = J.bbuf >= 0 ? buf(J.bbuf) : nullptr;
    if ((I.abuf >= 0 && !A) || (J.bbuf >= 0 && !B)) continue;
    const int k = dimv(I.k_st, I.k_rb, I.k_ri), rows = dimv(I.r_st, I.r_rb, I.r_ri);
    if (k <= 0 || rows <= 0) continue;
    if (I.row_off + rows > m) { fail = true; return; }
    for (int i = 0; i < rows; ++i)
      for (int j = 0; j < n; ++j) {
        double s = 0.0;
        if (I.aflags & FL_IDENT) s = B[J.boff + i + (int64_t)j * J.ldb];
        else if (J.bflags & FL_IDENT) s = A[I.aoff + i + (int64_t)j * I.lda];
        else
          for (int l = 0; l < k; ++l)
            s += ((I.aflags & FL_T) ? A[I.aoff + l + (int64_t)i * I.lda] : A[I.aoff + i + (int64_t)l * I.lda]) *
                 ((J.bflags & FL_OMEGA) ? sketch(J.omega_row0 + l, j)
                  : (J.bflags & FL_T)   ? B[J.boff + j + (int64_t)l * J.ldb]
                                        : B[J.boff + l + (int64_t)j * J.ldb]);
        acc[i + (size_t)m * j] += signs[I.coef] * s;
      }
  }
  for (int i = 0; i < m; ++i)
    for (int j = 0; j < n; ++j) {
      double& c = C[i + (int64_t)j * G.ldc];
      c = acc[i + (size_t)m * j] + (G.beta >= 0 ? signs[G.beta] * c : 0.0);
    }
}

// S_i = Z_i^T Omega or P_i = X_i^T Q of one target, with its common right factor
void target_dots(const Plan& pl, const TInfo& ti, bool sk) {
  const double* scr = tab[3 * pl.nroles];
  const int cols = sk ? ti.p : rtab[pl.nroles][ti.r_ri], rows = sk ? ti.n : ti.m;
  for (int g = sk ? ti.s_beg : ti.x_beg; g < (sk ? ti.s_end : ti.x_end); ++g) {
    const GGroup& G = pl.groups[g];
    const GItem& I = pl.items[G.ib];
    if (G.cbuf != 3 * pl.nroles || G.ie - G.ib != 1 || !(I.aflags & FL_T) || I.k_rb >= 0) {
      std::printf("not an inner product of a target\n");
      fail = true;
      return;
    }
    if (!buf(I.abuf)) continue;
    const int off = sk ? I.omega_row0 : (int)(I.boff - ti.y_off);
    if (off < 0 || off + I.k_st > rows) { std::printf("rows outside the factor\n"); fail = true; return; }
    const double* Z = buf(I.abuf) + I.aoff;
    double* C = tab[3 * pl.nroles] + G.coff;
    for (int i = 0; i < dimv(G.m_st, G.m_rb, G.m_ri); ++i)
      for (int j = 0; j < cols; ++j) {
        double s = 0.0;
        for (int l = 0; l < I.k_st; ++l)
          s += Z[l + (int64_t)i * I.lda] *
               (sk ? sketch(off + l, j) : scr[ti.y_off + off + l + (int64_t)j * ti.m]);
        C[i + (int64_t)j * G.ldc] = s;
      }
  }
}

// Gram-Schmidt (twice) of the sketch, in place, with pivots
void basis(const Plan& pl, const TInfo& ti, double tau) {
  double* Y = tab[3 * pl.nroles] + ti.y_off;
  const int m = ti.m;
  auto dot = [&](int a, int b) {
    double s = 0.0;
    for (int i = 0; i < m; ++i) s += Y[i + (int64_t)a * m] * Y[i + (int64_t)b * m];
    return s;
  };
  double first = 0.0;
  int r = 0;
  for (; r < ti.p; ++r) {
    int q = r;
    for (int c = r; c < ti.p; ++c)
      if (dot(c, c) > dot(q, q)) q = c;
    for (int i = 0; i < m; ++i) std::swap(Y[i + (int64_t)q * m], Y[i + (int64_t)r * m]);
    if (r == 0) first = dot(0, 0);
    if (!(dot(r, r) > tau * tau * first)) break;
    const double f = 1.0 / std::sqrt(dot(r, r));
    for (int i = 0; i < m; ++i) Y[i + (int64_t)r * m] *= f;
    for (int pass = 0; pass < 2; ++pass)
      for (int c = r + 1; c < ti.p; ++c) {
        const double s = dot(c, r);
        for (int i = 0; i < m; ++i) Y[i + (int64_t)c * m] -= s * Y[i + (int64_t)r * m];
      }
  }
  rtab[pl.nroles][ti.r_ri] = r;
}

// Gram of B^T, its eigenvectors (eig of plan_emulator.cpp, in a scratch of its own), the factors
void core(const Plan& pl, TInfo ti, double eps, int crole) {
  const int r = rtab[pl.nroles][ti.r_ri], m = ti.m, n = ti.n;
  double* scr = tab[3 * pl.nroles];
  std::vector<double> own((size_t)2 * ti.p * ti.p + 1);
  for (int i = 0; i < r; ++i)
    for (int j = 0; j < r; ++j)
      for (int l = 0; l < n; ++l)
        own[i + (size_t)j * ti.p] += scr[ti.bt_off + l + (int64_t)i * n] * scr[ti.bt_off + l + (int64_t)j * n];
  ti.h_off = 0;
  ti.w_off = (int64_t)ti.p * ti.p;
  tab[3 * pl.nroles] = own.data();
  eig(pl, ti, eps, crole);
  tab[3 * pl.nroles] = scr;
  const int k = rtab[crole] ? rtab[crole][ti.c_leaf] : 0;
  for (int j = 0; j < k; ++j) {
    const double* w = &own[ti.w_off + (size_t)j * ti.p];
    for (int i = 0; i < m + n; ++i) {
      double s = 0.0;
      for (int l = 0; l < r; ++l)
        s += w[l] * (i < m ? scr[ti.y_off + i + (int64_t)l * m] : scr[ti.bt_off + i - m + (int64_t)l * n]);
      if (i < m) tab[3 * crole + 1][ti.u_off + i + (int64_t)j * m] = s;
      else tab[3 * crole + 2][ti.v_off + i - m + (int64_t)j * n] = s;
    }
  }
}

void execute_engine(const Plan& pl, const std::vector<HMat*>& roles, int crole, double eps) {
  std::vector<double> scr(pl.scratch + 16, 1e300);
  std::vector<int> sr(pl.scratch_ranks + 1, 0);
  tab.assign(3 * pl.nroles + 1, nullptr);
  rtab.assign(pl.nroles + 1, nullptr);
  for (int r = 0; r < pl.nroles; ++r)
    if (roles[r]) {
      tab[3 * r] = roles[r]->d.data();
      tab[3 * r + 1] = roles[r]->U.data();
      tab[3 * r + 2] = roles[r]->V.data();
      rtab[r] = roles[r]->rank.data();
    }
  tab[3 * pl.nroles] = scr.data();
  rtab[pl.nroles] = sr.data();
  const double tau = std::max(1e-3 * eps, 1e-7);
  for (const Stage& sg : pl.stages) {
    if (sg.kind == ST_GEMM && (sg.tag == TAG_S || sg.tag == TAG_P)) {
      for (int t : pl.torder) target_dots(pl, pl.targets[t], sg.tag == TAG_S);
    } else if (sg.kind == ST_GEMM && sg.bend > sg.bbeg) {
      for (int g = sg.beg; g < sg.beg + sg.nwide; ++g) product(pl, pl.groups[g], pl.groups[g]);
      for (int b = sg.bbeg; b < sg.bend; ++b)
        for (int g = pl.bundles[2 * b]; g < pl.bundles[2 * b + 1]; ++g)
          product(pl, pl.groups[g], pl.groups[pl.bundles[2 * b]]);
    } else if (sg.kind == ST_GEMM) {
      for (int g = sg.beg; g < sg.end; ++g) product(pl, pl.groups[g], pl.groups[g]);
    } else if (sg.kind == ST_PCHOL || sg.kind == ST_PCHOL + 16) {
      for (int t = sg.beg; t < sg.end; ++t) pchol(pl, pl.targets[t], sg.kind == ST_PCHOL, tau);
    } else if (sg.kind == ST_ORTH) {
      for (int t : pl.torder) basis(pl, pl.targets[t], tau);
    } else if (sg.kind == ST_CORE) {
      for (const TInfo& ti : pl.targets) core(pl, ti, eps, crole);
    } else {
      std::printf("a stage of kind %d that the engine does not run\n", sg.kind);
      fail = true;
    }
  }
}

// what the kernels rely on
int check_records(const Plan& pl) {
  int bad = 0;
  for (const Stage& sg : pl.stages) {
    if (sg.kind != ST_GEMM) continue;
    std::vector<int> seen(sg.end - sg.beg, 0);
    if (sg.tag == TAG_S || sg.tag == TAG_P) {
      for (const TInfo& ti : pl.targets)
        for (int g = sg.tag == TAG_S ? ti.s_beg : ti.x_beg; g < (sg.tag == TAG_S ? ti.s_end : ti.x_end); ++g) {
          if (g < sg.beg || g >= sg.end) ++bad;
          else ++seen[g - sg.beg];
        }
      for (int s : seen) bad += s != 1;
    }
    if (sg.tag == TAG_FACT) {
      for (int b = sg.bbeg; b < sg.bend; ++b) {
        const int g0 = pl.bundles[2 * b], g1 = pl.bundles[2 * b + 1];
        if (g1 - g0 < 1 || g1 - g0 > BUNDLE_MAX || g0 < sg.beg + sg.nwide || g1 > sg.end) { ++bad; continue; }
        for (int g = g0; g < g1; ++g) {
          ++seen[g - sg.beg];
          bad += pl.groups[g].ie - pl.groups[g].ib != pl.groups[g0].ie - pl.groups[g0].ib;
        }
      }
      for (int g = sg.beg; g < sg.end; ++g) bad += seen[g - sg.beg] != (g >= sg.beg + sg.nwide);
    }
  }
  for (size_t i = 1; i < pl.torder.size(); ++i) {
    const TInfo &a = pl.targets[pl.torder[i - 1]], &b = pl.targets[pl.torder[i]];
    bad += (int64_t)a.m * a.p > (int64_t)b.m * b.p;
  }
  for (const TInfo& ti : pl.targets)   // the low parts of a sketch lie in B^T's place
    bad += ti.bt_off < ti.y_off + (int64_t)ti.m * ti.p ||
           ti.bt_off + (int64_t)ti.m * ti.p > pl.scratch;
  return bad;
}

}  // namespace

int main(int argc, char** argv) {
  const int n = argc > 1 ? std::atoi(argv[1]) : 16;
  const double eta = argc > 2 ? std::atof(argv[2]) : 2.0;
  const int leaf = argc > 3 ? std::atoi(argv[3]) : 16;
  const bool fused = argc > 4 && std::atoi(argv[4]);
  const double eps = 1e-10, tol = 1e-8;
  S.build(n, eta, leaf);
  PlanParams pp{kc, 8, true};
  pp.fused = fused;
  pp.fused_core = true;
  OpDesc prod = product_op(0, 0, 0, 1, 0, 2);
  prod.prods[0].coef = 2;
  Plan pl;
  build_plan(S, prod, pp, pl);
  HMat A = random_h(3), I = block_diagonal(false), G = block_diagonal(true);
  const std::vector<double> Ad = to_dense(A), Gd = to_dense(G);
  auto run = [&](const char* name, HMat* a, HMat* b, const std::vector<double>& want) {
    HMat C = zero_h();
    execute_engine(pl, {&C, a, b}, 0, eps);
    report(name, rel(to_dense(C), want), tol);
  };
  run("A * I = A", &A, &I, Ad);
  run("I * B = B", &I, &A, Ad);
  run("A * G (G block diagonal)", &A, &G, matmul(Ad, Gd));
  OpDesc sum;
  sum.c_node = 0; sum.c_role = 0; sum.alpha = 0; sum.nroles = 3;
  sum.adds.push_back(OpDesc::Add{1, 1});
  sum.adds.push_back(OpDesc::Add{2, 1});
  Plan ps;
  build_plan(S, sum, pp, ps);
  {
    HMat C = random_h(3), T1 = random_h(2);
    const std::vector<double> Cd = to_dense(C), T1d = to_dense(T1);
    std::vector<double> want(Cd.size());
    for (size_t i = 0; i < want.size(); ++i) want[i] = Cd[i] - T1d[i];
    execute_engine(ps, {&C, &T1, nullptr}, 0, eps);   // (a plane without its second term)
    report("C - T1 (second term absent)", rel(to_dense(C), want), tol);
  }
  const int t1 = S.cl[0].child[0], t2 = S.cl[0].child[1];
  const int n11 = S.node(t1, t1), n12 = S.node(t1, t2), n21 = S.node(t2, t1);
  OpDesc a, b;
  a.c_node = n12; a.c_role = 1; a.alpha = -1; a.nroles = 2;
  a.prods.push_back(OpDesc::Prod{n11, n12, 0, 0, 0});
  b.c_node = n21; b.c_role = 1; b.alpha = -1; b.nroles = 2;
  b.prods.push_back(OpDesc::Prod{n21, n11, 0, 0, 0});
  Plan pa, pb, pm;
  build_plan(S, a, pp, pa);
  build_plan(S, b, pp, pb);
  merge_plans({&pa, &pb}, pm);
  {
    HMat X = random_h(2), T1 = zero_h(), T2 = zero_h();
    allow_cap = true;
    execute_engine(pa, {&X, &T1}, 1, eps);
    execute_engine(pb, {&X, &T1}, 1, eps);
    execute_engine(pm, {&X, &T2}, 1, eps);
    allow_cap = false;
    report("merged plans = separate plans", rel(to_dense(T2), to_dense(T1)), 1e-13);
  }
  int bad = 0;
  for (const Plan* p : {&pl, &ps, &pa, &pb, &pm}) bad += check_records(*p) + check_plan_order(*p);
  report("records of the plans", (double)bad, 0.0);
  return fail ? 1 : 0;
}
