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

#include "../paper_1711_10579_gb300/csrc/feeder.h"
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
          if (cnt > p.slots) return 2;
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
// ilu: an ILU(0) pattern instead (P = 1), and err its defining property (the
// product of the factors equals the matrix on the pattern).
extern "C" int resident_check(int n, int m, const int* f, const int* t, int P, int T, int ilu,
                              double* err, int* parts) {
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
  if (ilu) analyze(y, Ordering::RCM, false, s);
  else analyze(y, Ordering::MinDegree, true, s);
  ResPlanHost p;
  if (!res_plan(s, P, T, n % 2 ? 1.0 : 0.3, p)) return 100;
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
    if (ilu) {
      // sum_k A_ik D_k^-1 A_kj + A_ij (D_i) = the matrix, (i, j) in the pattern
      std::vector<int> at(s.nnz_lu(), -1);
      for (int e = 0; e < p.cta[0].njac; ++e) at[entry[p.jac[4 * (size_t)e + 3]]] = p.jac[4 * (size_t)e];
      for (int k = 0; k < 32 * p.cta[0].ngrp; ++k)
        if (p.row[4 * (size_t)k] >= 0) at[entry[p.row[4 * (size_t)k + 3]]] = p.row[4 * (size_t)k + 1];
      auto mul = [](const B4& a, const B4& b) {
        return B4{a[0] * b[0] + a[1] * b[2], a[0] * b[1] + a[1] * b[3], a[2] * b[0] + a[3] * b[2],
                  a[2] * b[1] + a[3] * b[3]};
      };
      auto entry_of = [&](int i, int j) {
        for (int q = s.lu_rowptr[i]; q < s.lu_rowptr[i + 1]; ++q)
          if (s.lu_col[q] == j) return q;
        return -1;
      };
      for (int i = 0; i < n; ++i)
        for (int q = s.lu_rowptr[i]; q < s.lu_rowptr[i + 1]; ++q) {
          const int j = s.lu_col[q];
          B4 sum = M[0][at[q]];
          if (i == j) invert(sum);
          for (int k = 0; k < std::min(i, j); ++k) {
            const int a = entry_of(i, k), c = a < 0 ? -1 : entry_of(k, j);
            if (c < 0) continue;
            const B4 t = mul(M[0][at[a]], mul(M[0][at[s.lu_diag[k]]], M[0][at[c]]));
            for (int d = 0; d < 4; ++d) sum[d] += t[d];
          }
          for (int d = 0; d < 4; ++d) *err = std::max(*err, std::fabs(sum[d] - A[q][d]));
        }
      return 0;
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

// The same for a feeder plan (csrc/feeder.cpp): a tree of n nodes with random
// diagonally dominant scalar blocks (the order of the operations is what the
// plan decides).  kinds[n]: bus types as the library packs them.
extern "C" int feeder_check(int n, const int* f, const int* t, const int8_t* kinds, int P, int G,
                            double* err, int* levels) {
  Ybus y;
  y.n = n;
  std::vector<std::vector<int>> adj(n);
  for (int i = 0; i < n; ++i) adj[i].push_back(i);
  for (int e = 0; e < n - 1; ++e) {
    adj[f[e]].push_back(t[e]);
    adj[t[e]].push_back(f[e]);
  }
  y.rowptr.push_back(0);
  for (auto& a : adj) {
    std::sort(a.begin(), a.end());
    for (int j : a) y.col.push_back(j);
    y.rowptr.push_back((int)y.col.size());
  }
  y.ybs = 3;
  y.val.assign(18 * y.col.size(), 1.0);
  Symbolic s;
  analyze(y, Ordering::MinDegree, true, s);
  std::vector<int8_t> bt(n);
  for (int i = 0; i < n; ++i) bt[i] = kinds[s.perm[i]];
  FeedPlanHost p;
  if (!feed_plan(s, bt, P, G, p)) return 100;
  std::mt19937 g(5);
  std::normal_distribution<double> N;
  std::vector<double> D(n), br(n, 0.0), b(n);
  std::vector<int> parent(n, -1), cta(n, -1), slot(n, -1);
  for (int i = 0; i < n; ++i) {
    D[i] = 4.0 + 0.3 * N(g);
    b[i] = N(g);
    if (p.branch[i] >= 0) {
      parent[i] = s.y_col[p.branch[i]];
      br[i] = 0.5 * N(g);
    }
  }
  const double poison = NAN;
  std::vector<std::vector<double>> H(P, std::vector<double>(p.max_slots, poison)), W = H;
  std::vector<std::vector<int>> who(P, std::vector<int>(p.max_slots, -1));
  std::vector<int> phases(n, 0);
  for (int c = 0; c < P; ++c) {
    const FeedCta& C = p.cta[c];
    for (int k = C.own; k < C.own + C.nown; ++k) {
      const int i = p.node[2 * k], at = p.node[2 * k + 1];
      if (cta[i] >= 0 || at >= p.max_slots || who[c][at] >= 0) return 1;
      cta[i] = c;
      slot[i] = at;
      who[c][at] = i;
      H[c][at] = D[i];
      W[c][at] = b[i];
    }
    for (int q = 0; q < 32 * C.ngrp; ++q) {
      const int id = p.item[2 * (size_t)(32 * C.grp + q)];
      if (id < 0) continue;
      const int i = id & (kFeedMaxNodes - 1), a = (id >> 28) & 3;
      const bool fr = ((bt[i] >> a) & 1) && !(bt[i] & 8);
      if (cta[i] != c || p.item[2 * (size_t)(32 * C.grp + q) + 1] != slot[i] || fr != ((id >> 30) == 1)) return 2;
      ++phases[i];
      const FeedGroup& gr = p.grp[C.grp + q / 32];
      int seen = 0;
      for (int e = 0; e < gr.width; ++e) {
        const int ye = p.ell_y[gr.ell + 32 * e + q % 32];
        if (ye < 0) continue;
        if (ye != s.y_rowptr[i] + e || p.ell_col[gr.ell + 32 * e + q % 32] != s.y_col[ye]) return 3;
        ++seen;
      }
      if (fr && seen != s.y_rowptr[i + 1] - s.y_rowptr[i]) return 4;
    }
  }
  for (int i = 0; i < n; ++i)
    if (cta[i] < 0 || phases[i] != 3) return 5;
  *levels = 0;
  std::vector<int> done(n, 0);  // 1 eliminated, 2 substituted
  auto run = [&](int c, const FeedPart& R, bool backward) {
    const int r0 = backward ? R.rb : R.rf, nr = backward ? R.nrb : R.nrf;
    for (int r = r0; r < r0 + nr;) {
      int e = r;
      while (p.rnd[2 * e + 1] >= 0) ++e;
      if (e >= r0 + nr) return 10;
      ++*levels;
      std::vector<int> now;  // what this level finishes is not read by it
      std::vector<double> acc(G, poison), rhs = acc;
      std::vector<int> on(G, -1);
      for (int rr = r; rr <= e; ++rr) {
        const int off = p.rnd[2 * rr], cnt = p.rnd[2 * rr + 1] & 0xffff;
        if (cnt > G) return 11;
        for (int q = 0; q < cnt; ++q) {
          const uint32_t x = p.rec[2 * (size_t)(off + q)], yv = p.rec[2 * (size_t)(off + q) + 1];
          if (x == kFeedNone) continue;
          const int at = x & 0xffff, other = x >> 16, rank = (yv >> kFeedRankShift) & 15;
          const int k = who[c][at], id = yv & (kFeedMaxNodes - 1);
          if (k < 0) return 12;
          if (backward) {
            const int pk = who[rank][other];
            if (pk != parent[k] || id != k || done[pk] != 2 || done[k] != 1) return 13;
            W[c][at] -= H[c][at] * W[rank][other];
            now.push_back(k);
            continue;
          }
          if (yv & kFeedFirst) {
            acc[q] = H[c][at];
            rhs[q] = W[c][at];
            on[q] = k;
          }
          if (on[q] != k) return 14;
          if (!(yv & kFeedFactor)) {
            const int ch = who[rank][other];
            if (ch != id || parent[ch] != k || done[ch] != 1) return 15;
            acc[q] -= br[ch] * H[rank][other];
            rhs[q] -= br[ch] * W[rank][other];
          } else {
            if (id != k || ((yv & kFeedRoot) != 0) != (parent[k] < 0)) return 16;
            H[c][at] = br[k] / acc[q];
            W[c][at] = rhs[q] / acc[q];
            now.push_back(k);
          }
        }
      }
      for (int k : now) done[k] = backward ? 2 : 1;
      r = e + 1;
    }
    return 0;
  };
  for (int c = 0; c < P; ++c)
    if (int rc = run(c, p.part[c], false)) return rc;
  if (P > 1)
    if (int rc = run(0, p.part[P], false)) return 20 + rc;
  for (int i = 0; i < n; ++i) {
    if (done[i] != 1) return 30;
    if (parent[i] < 0) done[i] = 2;
  }
  if (P > 1)
    if (int rc = run(0, p.part[P], true)) return 40 + rc;
  for (int c = 0; c < P; ++c)
    if (int rc = run(c, p.part[c], true)) return 60 + rc;
  *err = 0.0;
  for (int i = 0; i < n; ++i) {
    double r = b[i] - D[i] * W[cta[i]][slot[i]];
    if (done[i] != 2) return 31;
    if (parent[i] >= 0) r -= br[i] * W[cta[parent[i]]][slot[parent[i]]];
    for (int k = 0; k < n; ++k)
      if (parent[k] == i) r -= br[k] * W[cta[k]][slot[k]];
    if (!(std::fabs(r) <= *err)) *err = std::isnan(r) ? INFINITY : std::fabs(r);
  }
  return 0;
}
