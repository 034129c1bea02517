// Packed records of a symbolic analysis (records.h).
#include "records.h"

#include <algorithm>

namespace pf {

void pack_records(const Symbolic& s, std::vector<int4>& fwd, std::vector<int4>& bwd,
                  std::vector<int4>& fac, std::vector<int4>& tgt, std::vector<int2>& con) {
  const int n = s.n;
  fwd.assign(n, make_int4(0, 0, 0, 0));
  bwd.assign(n, make_int4(0, 0, 0, 0));
  fac.assign(s.fac_items.size(), make_int4(0, 0, 0, 0));
  tgt.assign(s.tgt_entry.size(), make_int4(0, 0, 0, 0));
  for (int t = 0; t < n; ++t) {
    const int i = s.flev_rows[t], j = s.blev_rows[t];
    fwd[t] = make_int4(i, s.lu_rowptr[i], s.lu_diag[i], 0);
    bwd[t] = make_int4(j, s.lu_diag[j] + 1, s.lu_rowptr[j + 1], 0);
  }
  for (size_t t = 0; t < fac.size(); ++t) {
    const int e = s.fac_items[t], k = s.lu_col[e];
    fac[t] = make_int4(e, k, s.lu_diag[k], 0);
  }
  con.clear();
  std::vector<char> touched(s.nnz_lu(), 0);
  std::vector<int> last(n, -1);  // target of a pivot's last update
  for (size_t t = 0; t < tgt.size(); ++t) {
    const int k = s.lu_col[s.tgt_entry[t]];
    if (s.tgt_entry[t] == s.lu_diag[k]) last[k] = (int)t;
  }
  for (int4& f : fac) f.w = last[f.y] >= 0;
  for (size_t t = 0; t < tgt.size(); ++t) {
    const int c0 = s.tgt_cptr[t], c1 = s.tgt_cptr[t + 1];
    const int te = s.tgt_entry[t];
    const bool fill_first = s.lu2y[te] < 0 && !touched[te];
    touched[te] = 1;
    const int k = s.lu_col[te];
    const int mark = te == s.lu_diag[k] && last[k] == (int)t ? -2 - k : -1;
    int rest = mark;
    if (c1 - c0 > 1) {
      rest = (int)con.size();
      for (int c = c0 + 1; c < c1; ++c) con.push_back(make_int2(s.con_l[c], s.con_u[c]));
      con.push_back(make_int2(-1, mark));
    }
    tgt[t] = make_int4(te | (fill_first ? kFillFirst : 0), s.con_l[c0], s.con_u[c0], rest);
  }
  if (con.empty()) con.push_back(make_int2(-1, -1));
}

void sort_records(const Symbolic& s, std::vector<int4>& fac, std::vector<int4>& tgt,
                  const std::vector<int2>& con) {
  auto by_work = [](std::vector<int4>& v, const std::vector<int>& ptr, auto work) {
    for (size_t l = 0; l + 1 < ptr.size(); ++l)
      for (int a = ptr[l]; a < ptr[l + 1]; a += 256)
        std::stable_sort(v.begin() + a, v.begin() + std::min(a + 256, ptr[l + 1]),
                         [&](const int4& x, const int4& y) { return work(x) > work(y); });
  };
  by_work(fac, s.fac_ptr, [](const int4& f) { return f.w ? (f.x == f.z ? 0 : 1) : 2; });
  by_work(tgt, s.tgt_ptr, [&](const int4& t) {
    int len = 1, mark = t.w;
    for (int q = t.w; q >= 0 && con[q].x >= 0; ++q, ++len) mark = con[q + 1].y;
    return len + (mark < -1 ? 1000 : 0);
  });
}

}  // namespace pf
