// Host execution of the factorisation's packed records (csrc/records.cpp) for
// the CPU tests: the items of each level as the batched kernels that invert a
// pivot once run them, on scalars instead of 2x2 blocks.
#include <algorithm>
#include <cmath>
#include <random>
#include <vector>

#include "../paper_1711_10579_gb300/csrc/records.h"

using namespace pf;

// A grid of n buses and m branches; ilu: the ILU(0) pattern.  sorted: the items
// sorted by work.  Returns 0 and the largest |(L U - A)_ij| of the pattern, or
// the rule broken; *descents: items out of the order of their entries (column by
// column, targets row by row) in a level.
extern "C" int records_check(int n, int m, const int* f, const int* t, int ilu, int sorted,
                             double* err, int* descents) {
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
  std::vector<int4> fwd, bwd, fac, tgt;
  std::vector<int2> con;
  pack_records(s, fwd, bwd, fac, tgt, con);
  if (sorted) sort_records(s, fac, tgt, con);

  std::mt19937 g(11);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  std::vector<double> A(s.nnz_lu(), 0.0), lu(s.nnz_lu(), NAN), uinv(n, NAN);  // NAN: not written yet
  for (int i = 0; i < n; ++i)
    for (int e = s.lu_rowptr[i]; e < s.lu_rowptr[i + 1]; ++e)
      if (s.lu2y[e] >= 0)
        lu[e] = A[e] = s.lu_col[e] == i ? 2.0 * (s.lu_rowptr[i + 1] - s.lu_rowptr[i]) + U(g) : U(g);
  *descents = 0;
  for (size_t l = 0; l + 1 < s.fac_ptr.size(); ++l) {
    const std::vector<double> lu0 = lu, uinv0 = uinv;  // a step reads the state before it
    for (int q = s.fac_ptr[l]; q < s.fac_ptr[l + 1]; ++q) {
      const int4 r = fac[q];
      if (q > s.fac_ptr[l] && (r.y < fac[q - 1].y || (r.y == fac[q - 1].y && r.x < fac[q - 1].x)))
        ++*descents;
      if (r.z != s.lu_diag[r.y] || s.lu_col[r.x] != r.y) return 1;
      if (r.w && std::isnan(uinv0[r.y])) return 2;  // said to be ready
      if (r.w && r.x == r.z) continue;
      const double di = r.w ? uinv0[r.y] : 1.0 / lu0[r.z];
      if (r.x != r.z) lu[r.x] = lu0[r.x] * di;
      else if (!std::isnan(uinv[r.y])) return 3;
      else uinv[r.y] = di;
    }
    const std::vector<double> lu1 = lu;
    for (int q = s.tgt_ptr[l]; q < s.tgt_ptr[l + 1]; ++q) {
      const int4 r = tgt[q];
      const int e = r.x & ~kFillFirst;
      if (q > s.tgt_ptr[l] && e < (tgt[q - 1].x & ~kFillFirst)) ++*descents;
      double c = (r.x & kFillFirst) ? 0.0 : lu1[e];
      c -= lu1[r.y] * lu1[r.z];
      int mark = r.w;
      if (r.w >= 0)
        for (int p = r.w;; ++p) {
          mark = con[p].y;
          if (con[p].x < 0) break;
          c -= lu1[con[p].x] * lu1[con[p].y];
        }
      if (mark < -1) {  // finishes a pivot: only its inverse is read from here on
        const int k = -2 - mark;
        if (e != s.lu_diag[k] || !std::isnan(uinv[k])) return 4;
        uinv[k] = 1.0 / c;
        lu[e] = NAN;
      } else {
        lu[e] = c;
      }
    }
  }
  *err = 0.0;
  std::vector<double> row(n, 0.0);
  for (int i = 0; i < n; ++i) {
    if (std::isnan(uinv[i])) return 5;
    for (int e = s.lu_rowptr[i]; e < s.lu_rowptr[i + 1]; ++e) {
      const int k = s.lu_col[e];
      if (k > i) row[k] += lu[e];
      else if (k == i) row[k] += 1.0 / uinv[i];
      else
        for (int p = s.lu_diag[k]; p < s.lu_rowptr[k + 1]; ++p)
          row[s.lu_col[p]] += lu[e] * (s.lu_col[p] == k ? 1.0 / uinv[k] : lu[p]);
    }
    for (int e = s.lu_rowptr[i]; e < s.lu_rowptr[i + 1]; ++e) {
      const double d = std::fabs(row[s.lu_col[e]] - A[e]);
      if (!(d <= *err)) *err = std::isnan(d) ? INFINITY : d;
    }
    for (int e = s.lu_rowptr[i]; e < s.lu_rowptr[i + 1]; ++e) {
      row[s.lu_col[e]] = 0.0;
      if (s.lu_col[e] < i)
        for (int p = s.lu_diag[s.lu_col[e]]; p < s.lu_rowptr[s.lu_col[e] + 1]; ++p) row[s.lu_col[p]] = 0.0;
    }
  }
  return 0;
}
