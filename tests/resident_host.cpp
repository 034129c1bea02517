// Host execution of a resident plan (csrc/resident.cpp) for the CPU tests: the
// rounds of every part run level by level on a random block matrix, with the
// checks that make the parallel execution well defined (the items of a target
// on one thread, no item of a level reading what that level writes, every row
// and Jacobian entry assembled once), and the residual of the solution.
#include <algorithm>
#include <array>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "../paper_1711_10579_gb300/csrc/resident.h"

using namespace pf;
using B4 = std::array<double, 4>;
using B2 = std::array<double, 2>;

namespace {

void invert(B4& a) {
  const double d = a[0] * a[3] - a[1] * a[2];
  a = B4{a[3] / d, -a[1] / d, -a[2] / d, a[0] / d};
}

struct Run {
  const ResPlanHost& p;
  std::vector<std::vector<B4>>& M;
  std::vector<std::vector<B2>>& V;

  // The rounds [r0, r0 + nr) of part R in CTA c; 0, or the rule broken.
  int rounds(int c, const ResPart& R, int r0, int nr, bool backward) {
    B4* a = M[c].data() + R.blk0;
    B2* v = V[c].data() + R.vec0;
    for (int r = r0; r < r0 + nr;) {
      int e = r;
      while (p.rnd[2 * e + 1] >= 0) ++e;  // the level ends with a barrier
      if (e >= r0 + nr) return 1;
      std::vector<int> wb(R.nblk, -1), wv(R.np + R.nb, -1);
      for (int pass = 0; pass < 2; ++pass)
        for (int rr = r; rr <= e; ++rr) {
          const int off = p.rnd[2 * rr], cnt = p.rnd[2 * rr + 1] & 0xffff;
          if (cnt > p.threads) return 2;
          for (int th = 0; th < cnt; ++th) {
            const uint32_t x = p.rec[2 * (size_t)(off + th)], y = p.rec[2 * (size_t)(off + th) + 1];
            const int t = x & 0xffff, b = x >> 16, k = (y >> 16) & (kResMaxRows - 1), u = y & 0xffff;
            if (t == kResNone) continue;
            const bool vec = backward || (y & kResVec);
            if (t >= (vec ? R.np + R.nb : R.nblk)) return 3;
            if (pass == 0) {  // who writes what
              int& w = vec ? wv[t] : wb[t];
              if (w >= 0 && w != th) return 4;
              w = th;
              continue;
            }
            if (backward) {
              if (b != kResNone) {
                if (b >= R.nblk || u >= R.np + R.nb || wv[u] >= 0) return 5;
                v[t][0] -= a[b][0] * v[u][0] + a[b][1] * v[u][1];
                v[t][1] -= a[b][2] * v[u][0] + a[b][3] * v[u][1];
              }
              if (y & kResFinal) {
                const B2 z = v[t];
                v[t] = B2{a[t][0] * z[0] + a[t][1] * z[1], a[t][2] * z[0] + a[t][3] * z[1]};
              }
              continue;
            }
            if (k >= R.np || b >= R.nblk || wb[b] >= 0 || wb[k] >= 0) return 6;
            const B4 D = a[k], L = a[b];
            if (vec) {
              if (wv[k] >= 0) return 7;
              const double m0 = D[0] * v[k][0] + D[1] * v[k][1], m1 = D[2] * v[k][0] + D[3] * v[k][1];
              v[t][0] -= L[0] * m0 + L[1] * m1;
              v[t][1] -= L[2] * m0 + L[3] * m1;
              continue;
            }
            if (u >= R.nblk || wb[u] >= 0) return 8;
            const B4 U = a[u], m{D[0] * U[0] + D[1] * U[2], D[0] * U[1] + D[1] * U[3],
                                 D[2] * U[0] + D[3] * U[2], D[2] * U[1] + D[3] * U[3]};
            a[t][0] -= L[0] * m[0] + L[1] * m[2];
            a[t][1] -= L[0] * m[1] + L[1] * m[3];
            a[t][2] -= L[2] * m[0] + L[3] * m[2];
            a[t][3] -= L[2] * m[1] + L[3] * m[3];
            if (y & kResFinal) invert(a[t]);
          }
        }
      r = e + 1;
    }
    return 0;
  }
};

}  // namespace

// A grid of n buses and m branches, P CTAs of T threads: solves J x = b twice
// (the factorisation with its forward sweep, then the forward sweep alone) on
// random blocks.  Returns 0 and the largest residual, or the rule broken.
extern "C" int resident_check(int n, int m, const int* f, const int* t, int P, int T, double* err,
                              int* parts) {
  Ybus y;
  y.n = n;
  std::vector<std::vector<int>> adj(n);
  for (int i = 0; i < n; ++i) adj[i].push_back(i);
  for (int e = 0; e < m; ++e) {
    adj[f[e]].push_back(t[e]);
    adj[t[e]].push_back(f[e]);
  }
  y.rowptr.push_back(0);
  for (auto& a : adj) {
    std::sort(a.begin(), a.end());
    a.erase(std::unique(a.begin(), a.end()), a.end());
    for (int j : a) y.col.push_back(j);
    y.rowptr.push_back((int)y.col.size());
  }
  y.val.assign(2 * y.col.size(), 1.0);
  Symbolic s;
  analyze(y, Ordering::MinDegree, true, s);
  ResPlanHost p;
  if (!res_plan(s, P, T, p)) return 100;
  *parts = 0;
  for (const ResPart& R : p.part) *parts += R.np > 0;

  std::mt19937 g(7);
  std::normal_distribution<double> N;
  std::vector<B4> A(s.nnz_lu(), B4{0, 0, 0, 0});
  std::vector<int> rowof(s.nnz_lu()), entry(s.nnz_y(), -1);
  for (int i = 0; i < n; ++i)
    for (int q = s.lu_rowptr[i]; q < s.lu_rowptr[i + 1]; ++q) {
      rowof[q] = i;
      if (s.lu2y[q] < 0) continue;
      entry[s.lu2y[q]] = q;
      for (double& v : A[q]) v = 0.2 * N(g);
      if (s.lu_col[q] == i) {
        A[q][0] += 4;
        A[q][3] += 4;
      }
    }
  // poisoned memory: what is not assembled, zeroed or written shows
  std::vector<std::vector<B4>> M(P, std::vector<B4>(p.max_blk, B4{NAN, NAN, NAN, NAN}));
  std::vector<std::vector<B2>> V(P, std::vector<B2>(p.max_vec, B2{NAN, NAN}));
  Run run{p, M, V};
  for (size_t q = 0; q < p.part.size(); ++q) {
    const ResPart& R = p.part[q];
    const int c = q < (size_t)P ? (int)q : 0;
    for (int k = R.z0; k < R.nblk; ++k) M[c][R.blk0 + k] = B4{0, 0, 0, 0};
  }
  std::vector<std::array<int, 2>> where(n, std::array<int, 2>{-1, -1});
  int jac = 0;
  for (int c = 0; c < P; ++c) {
    const ResCta& C = p.cta[c];
    for (int k = 0; k < 32 * C.ngrp; ++k) {
      const int* r = &p.row[4 * (size_t)(32 * C.grp + k)];
      if (r[0] < 0) continue;
      const int i = r[0] & ~kResRowLevel0;
      if (where[i][0] >= 0 || r[3] != s.lu2y[s.lu_diag[i]]) return 20;
      where[i] = {c, r[2]};
      M[c][r[1]] = A[s.lu_diag[i]];
      if (r[0] & kResRowLevel0) invert(M[c][r[1]]);
      const ResGroup& G = p.grp[C.grp + k / 32];
      std::vector<int> ys;
      for (int e = 0; e < G.width; ++e) {
        const int ye = p.ell_y[G.ell + 32 * e + k % 32];
        if (ye < 0) continue;
        if (p.ell_col[G.ell + 32 * e + k % 32] != s.y_col[ye]) return 21;
        ys.push_back(ye);
      }
      if (ys.empty() || ys[0] != r[3]) return 22;  // the diagonal first
      std::sort(ys.begin(), ys.end());
      if ((int)ys.size() != s.y_rowptr[i + 1] - s.y_rowptr[i] || ys[0] != s.y_rowptr[i]) return 23;
    }
    for (int e = 0; e < C.njac; ++e, ++jac) {
      const int* r = &p.jac[4 * (size_t)(C.jac + e)];
      const int q = entry[r[3]];
      if (rowof[q] != r[1] || s.lu_col[q] != r[2] || !std::isnan(M[c][r[0]][0])) return 24;
      M[c][r[0]] = A[q];
    }
  }
  if (jac + n != s.nnz_y()) return 25;

  *err = 0.0;
  for (int pass = 0; pass < 2; ++pass) {
    std::vector<B2> b(n);
    for (int i = 0; i < n; ++i) {
      b[i] = B2{N(g), N(g)};
      if (where[i][0] < 0) return 26;
      V[where[i][0]][where[i][1]] = b[i];
    }
    for (int c = 0; c < P; ++c) {
      const ResPart& R = p.part[c];
      for (int k = 0; k < R.nb; ++k) V[c][R.vec0 + R.np + k] = B2{0, 0};
      const int rc = pass == 0 ? run.rounds(c, R, R.rf, R.nrf, false) : run.rounds(c, R, R.rw, R.nrw, false);
      if (rc) return rc;
    }
    if (P > 1) {
      const ResPart& R = p.part[P];
      for (int k = 0; k < p.ngat_blk + p.ngat_vec; ++k) {
        const int* q = &p.gat[4 * k];
        if (k < p.ngat_blk && pass > 0) continue;
        for (int u = q[1]; u < q[2]; ++u) {
          const int c = p.gsrc[2 * u], at = p.gsrc[2 * u + 1];
          if (k < p.ngat_blk)
            for (int d = 0; d < 4; ++d) M[0][R.blk0 + q[0]][d] += M[c][at][d];
          else
            for (int d = 0; d < 2; ++d) V[0][R.vec0 + q[0]][d] += V[c][at][d];
        }
        if (q[3]) invert(M[0][R.blk0 + q[0]]);
      }
      int rc = pass == 0 ? run.rounds(0, R, R.rf, R.nrf, false) : run.rounds(0, R, R.rw, R.nrw, false);
      if (rc == 0) rc = run.rounds(0, R, R.rb, R.nrb, true);
      if (rc) return 40 + rc;
      for (int c = 0; c < P; ++c) {
        const ResPart& Q = p.part[c];
        for (int k = 0; k < Q.nb; ++k) V[c][Q.vec0 + Q.np + k] = V[0][R.vec0 + p.bnd[Q.bnd + k]];
      }
    }
    for (int c = 0; c < P; ++c) {
      const int rc = run.rounds(c, p.part[c], p.part[c].rb, p.part[c].nrb, true);
      if (rc) return 60 + rc;
    }
    for (int i = 0; i < n; ++i) {
      B2 r = b[i];
      for (int q = s.lu_rowptr[i]; q < s.lu_rowptr[i + 1]; ++q) {
        if (s.lu2y[q] < 0) continue;
        const auto& w = where[s.lu_col[q]];
        const B2& x = V[w[0]][w[1]];
        r[0] -= A[q][0] * x[0] + A[q][1] * x[1];
        r[1] -= A[q][2] * x[0] + A[q][3] * x[1];
      }
      for (double d : r)
        if (!(std::fabs(d) <= *err)) *err = std::isnan(d) ? INFINITY : std::fabs(d);
    }
  }
  return 0;
}
