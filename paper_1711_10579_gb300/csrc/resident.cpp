// Host schedule of resident solves (resident.h): the cut of the elimination
// tree into parts, the blocks of each part, and the rounds of items.
#include <algorithm>
#include <queue>
#include <unordered_map>

#include "resident.h"

namespace pf {

namespace {

struct Item {
  int t, b, c, k;
  bool vec, fin;
};

// Rounds of one level: the items of a target form a chain on one slot.
// Chains go to the slot with the fewest items, long ones first.
class RoundPacker {
 public:
  RoundPacker(int slots, ResPlanHost& out) : T_(slots), out_(out) {}

  void level(std::vector<std::vector<Item>>& chains) {
    if (chains.empty()) return;
    std::stable_sort(chains.begin(), chains.end(),
                     [](const std::vector<Item>& a, const std::vector<Item>& b) {
                       return a.size() > b.size();
                     });
    const int T = std::min(T_, (int)chains.size());  // no more slots are used
    std::vector<std::vector<const Item*>> col(T);
    std::priority_queue<std::pair<int, int>, std::vector<std::pair<int, int>>,
                        std::greater<std::pair<int, int>>>
        pq;
    for (int t = 0; t < T; ++t) pq.push({0, t});
    size_t height = 0;
    for (const auto& ch : chains) {
      const auto top = pq.top();
      pq.pop();
      for (const Item& it : ch) col[top.second].push_back(&it);
      height = std::max(height, col[top.second].size());
      pq.push({top.first + (int)ch.size(), top.second});
    }
    for (size_t r = 0; r < height; ++r) {
      int cnt = 0;
      for (int t = 0; t < T; ++t)
        if (col[t].size() > r) cnt = t + 1;
      out_.rnd.push_back((int)(out_.rec.size() / 2));
      out_.rnd.push_back(cnt | (r + 1 == height ? kResSync : 0));
      for (int t = 0; t < cnt; ++t) {
        if (col[t].size() <= r) {
          out_.rec.push_back((uint32_t)kResNone);
          out_.rec.push_back(0);
          continue;
        }
        const Item& it = *col[t][r];
        out_.rec.push_back((uint32_t)it.t | (uint32_t)it.b << 16);
        out_.rec.push_back((uint32_t)it.c | (uint32_t)it.k << 16 | (it.vec ? kResVec : 0u) |
                           (it.fin ? kResFinal : 0u));
      }
    }
  }

 private:
  int T_;
  ResPlanHost& out_;
};

// The level's chains from its items sorted by (vec, t).
std::vector<std::vector<Item>> chains_of(std::vector<Item>& items) {
  std::stable_sort(items.begin(), items.end(), [](const Item& a, const Item& b) {
    return a.vec != b.vec ? a.vec < b.vec : a.t < b.t;
  });
  std::vector<std::vector<Item>> ch;
  for (size_t q = 0; q < items.size(); ++q) {
    if (q == 0 || items[q].t != items[q - 1].t || items[q].vec != items[q - 1].vec)
      ch.emplace_back();
    ch.back().push_back(items[q]);
  }
  return ch;
}

// part[i] of every row: 0 .. P-1, or P for the top.  The heaviest subtree's
// root moves to the top until the subtrees balance over the P bins.  A pivot of
// d later neighbours weighs 12 + 4 d + quad d^2.
void cut_tree(const Symbolic& s, int P, double quad, std::vector<int>& part) {
  const int n = s.n;
  part.assign(n, P > 1 ? P : 0);
  if (P == 1) return;
  std::vector<int> parent(n, -1);
  std::vector<double> w(n), sub(n, 0.0);
  std::vector<std::vector<int>> child(n);
  for (int k = 0; k < n; ++k) {
    const int d = s.lu_rowptr[k + 1] - s.lu_diag[k] - 1;
    if (d > 0) parent[k] = s.lu_col[s.lu_diag[k] + 1];
    w[k] = 12.0 + 4.0 * d + quad * d * d;  // mismatch and Jacobian; sweeps; updates
  }
  for (int k = 0; k < n; ++k) {
    sub[k] += w[k];
    if (parent[k] >= 0) {
      sub[parent[k]] += sub[k];
      child[parent[k]].push_back(k);
    }
  }
  std::priority_queue<std::pair<double, int>> heap;
  double total = 0.0;
  for (int k = 0; k < n; ++k)
    if (parent[k] < 0) {
      heap.push({sub[k], k});
      total += sub[k];
    }
  // bins of the current subtrees, largest first; the first bin also carries
  // the top's rows
  std::vector<std::vector<int>> bins(P), best_bins;
  double best = 1e300, topw = 0.0;
  std::vector<int> top, best_top;
  for (int step = 0; step <= n && !heap.empty(); ++step) {
    // the top runs after the parts, its rows one after another
    const double after = 2.0 * topw + 40.0 * P * top.size() / 16.0;
    // no bins are better than even ones, nor than the heaviest subtree's
    const double least = std::max(heap.top().first, (total - topw) / P);
    if (((int)heap.size() >= P || step == n) && (least + after) * (1.0 + 1e-9) >= best) {
      if (topw + 40.0 * top.size() > best) break;
    } else if ((int)heap.size() >= P || step == n) {
      std::vector<std::pair<double, int>> all;
      auto h = heap;
      while (!h.empty()) {
        all.push_back(h.top());
        h.pop();
      }
      std::vector<std::vector<int>> bb(P);
      std::priority_queue<std::pair<double, int>, std::vector<std::pair<double, int>>,
                          std::greater<std::pair<double, int>>>
          load;
      for (int q = 0; q < P; ++q) load.push({q == 0 ? 12.0 * top.size() : 0.0, q});
      double worst = 0.0;
      for (const auto& a : all) {
        auto l = load.top();
        load.pop();
        bb[l.second].push_back(a.second);
        l.first += a.first;
        worst = std::max(worst, l.first);
        load.push(l);
      }
      const double cost = worst + after;
      if (cost < best) {
        best = cost;
        best_bins = bb;
        best_top = top;
      } else if (topw + 40.0 * top.size() > best) {
        break;  // a larger top cannot pay off any more
      }
    }
    const int k = heap.top().second;
    heap.pop();
    top.push_back(k);
    topw += w[k];
    for (int c : child[k]) heap.push({sub[c], c});
  }
  if (best_bins.empty()) {  // fewer subtrees than CTAs: everything in one part
    part.assign(n, 0);
    return;
  }
  for (int q = 0; q < P; ++q)
    for (int r : best_bins[q]) part[r] = q;
  for (int k = n - 1; k >= 0; --k)  // subtrees inherit their root's part
    if (parent[k] >= 0 && part[parent[k]] < P) part[k] = part[parent[k]];
}

}  // namespace

bool res_plan(const Symbolic& s, int P, int slots, double quad, ResPlanHost& out) {
  const int n = s.n, nnz = s.nnz_lu();
  out = ResPlanHost();
  out.P = P;
  out.slots = slots;
  std::vector<int> part;
  cut_tree(s, P, quad, part);
  const int Q = P > 1 ? P + 1 : 1;  // parts and the top
  std::vector<std::vector<int>> piv(Q), bnd(Q);
  for (int i = 0; i < n; ++i) piv[part[i]].push_back(i);
  std::vector<int> lidx(n, -1);  // local index of a pivot in its part
  for (int q = 0; q < Q; ++q)
    for (size_t t = 0; t < piv[q].size(); ++t) lidx[piv[q][t]] = (int)t;

  std::vector<int> rowof(nnz);
  for (int i = 0; i < n; ++i)
    for (int p = s.lu_rowptr[i]; p < s.lu_rowptr[i + 1]; ++p) rowof[p] = i;
  auto find = [&](int i, int j) {
    const int* b = s.lu_col.data() + s.lu_rowptr[i];
    const int* e = s.lu_col.data() + s.lu_rowptr[i + 1];
    const int* q = std::lower_bound(b, e, j);
    return q != e && *q == j ? (int)(q - s.lu_col.data()) : -1;
  };
  // home part of an entry: that of its pivot, the smaller of row and column
  auto home = [&](int e) { return part[std::min(rowof[e], s.lu_col[e])]; };

  // blocks of each part: diagonals, other Jacobian entries, fill
  std::vector<int> pos(nnz, -1);
  std::vector<int> nblk(Q, 0), z0(Q, 0);
  for (int q = 0; q < Q; ++q) {
    for (size_t t = 0; t < piv[q].size(); ++t) pos[s.lu_diag[piv[q][t]]] = (int)t;
    nblk[q] = (int)piv[q].size();
  }
  for (int pass = 0; pass < 2; ++pass) {
    for (int e = 0; e < nnz; ++e)
      if (rowof[e] != s.lu_col[e] && (s.lu2y[e] >= 0) == (pass == 0)) pos[e] = nblk[home(e)]++;
    if (pass == 0) z0 = nblk;
  }
  // boundary rows, and their accumulators
  std::vector<std::unordered_map<int, int>> bl(Q), acc(Q);  // top row -> local, entry -> block
  for (int q = 0; q + 1 < Q; ++q) {
    for (int k : piv[q])
      for (int p = s.lu_diag[k] + 1; p < s.lu_rowptr[k + 1]; ++p)
        if (part[s.lu_col[p]] != q) bnd[q].push_back(s.lu_col[p]);
    std::sort(bnd[q].begin(), bnd[q].end());
    bnd[q].erase(std::unique(bnd[q].begin(), bnd[q].end()), bnd[q].end());
    for (size_t t = 0; t < bnd[q].size(); ++t) bl[q][bnd[q][t]] = (int)(piv[q].size() + t);
  }
  auto slot = [&](int q, int i) { return part[i] == q ? lidx[i] : bl[q].at(i); };

  RoundPacker pack(slots, out);
  out.part.resize(Q);
  std::vector<int> lev(n, 0);
  for (int q = 0; q < Q; ++q) {
    ResPart& R = out.part[q];
    R.np = (int)piv[q].size();
    R.nb = (int)bnd[q].size();
    // levels within the part
    int nl = 0;
    for (int k : piv[q]) {
      int l = 0;
      for (int p = s.lu_rowptr[k]; p < s.lu_diag[k]; ++p)
        if (part[s.lu_col[p]] == q) l = std::max(l, lev[s.lu_col[p]] + 1);
      lev[k] = l;
      nl = std::max(nl, l + 1);
    }
    std::vector<std::vector<int>> at(nl);
    for (int k : piv[q]) at[lev[k]].push_back(k);
    // factorisation with the forward sweep, and the forward sweep alone
    std::vector<std::vector<Item>> fwd(nl);
    R.rf = (int)out.rnd.size() / 2;
    for (int l = 0; l < nl; ++l) {
      std::vector<Item> items;
      for (int k : at[l])
        for (int pi = s.lu_diag[k] + 1; pi < s.lu_rowptr[k + 1]; ++pi) {
          const int i = s.lu_col[pi], eik = find(i, k);
          for (int pj = s.lu_diag[k] + 1; pj < s.lu_rowptr[k + 1]; ++pj) {
            const int j = s.lu_col[pj], e = find(i, j);
            if (e < 0) continue;  // ILU(0): outside the pattern
            int t;
            if (home(e) == q) {
              t = pos[e];
            } else {
              auto it = acc[q].find(e);
              if (it == acc[q].end()) it = acc[q].emplace(e, nblk[q]++).first;
              t = it->second;
            }
            items.push_back({t, pos[eik], pos[pj], lidx[k], false, false});
          }
          items.push_back({slot(q, i), pos[eik], 0, lidx[k], true, false});
          fwd[l].push_back(items.back());
        }
      auto ch = chains_of(items);
      // a pivot whose last update this is: its level is the next one
      for (auto& c : ch) {
        const Item& f = c.front();
        if (!f.vec && f.t < R.np && lev[piv[q][f.t]] == l + 1) c.back().fin = true;
      }
      pack.level(ch);
    }
    R.nrf = (int)out.rnd.size() / 2 - R.rf;
    R.rw = (int)out.rnd.size() / 2;
    for (int l = 0; l < nl; ++l) {
      auto ch = chains_of(fwd[l]);
      pack.level(ch);
    }
    R.nrw = (int)out.rnd.size() / 2 - R.rw;
    // backward sweep: row k is finished at step bl(k); entry (k, j) is taken
    // at the step after j's
    std::vector<int> blev(R.np, 0);
    int nbk = R.np > 0 ? 1 : 0;
    for (int t = R.np - 1; t >= 0; --t) {
      const int k = piv[q][t];
      int l = 0;
      for (int p = s.lu_diag[k] + 1; p < s.lu_rowptr[k + 1]; ++p)
        if (part[s.lu_col[p]] == q) l = std::max(l, blev[lidx[s.lu_col[p]]] + 1);
      blev[t] = l;
      nbk = std::max(nbk, l + 1);
    }
    std::vector<std::vector<Item>> step(nbk);
    for (int t = 0; t < R.np; ++t) {
      const int k = piv[q][t];
      if (s.lu_diag[k] + 1 == s.lu_rowptr[k + 1]) {  // a root: no entries
        step[0].push_back({t, kResNone, 0, 0, false, true});
        continue;
      }
      for (int p = s.lu_diag[k] + 1; p < s.lu_rowptr[k + 1]; ++p) {
        const int j = s.lu_col[p];
        const int st = part[j] == q ? blev[lidx[j]] + 1 : 0;
        step[st].push_back({t, pos[p], slot(q, j), 0, false, false});
      }
    }
    R.rb = (int)out.rnd.size() / 2;
    for (int l = 0; l < nbk; ++l) {
      auto ch = chains_of(step[l]);
      for (auto& c : ch)
        if (blev[c.front().t] == l) c.back().fin = true;
      pack.level(ch);
    }
    R.nrb = (int)out.rnd.size() / 2 - R.rb;
    R.nblk = nblk[q];
    R.z0 = z0[q];
    if (R.nblk >= kResNone || R.np + R.nb > kResMaxRows) return false;
    R.bnd = (int)out.bnd.size();
    for (int i : bnd[q]) out.bnd.push_back(lidx[i]);
  }
  // where each part lives: part q in CTA q, the top after part 0
  for (int q = 0; q < Q; ++q) {
    ResPart& R = out.part[q];
    R.blk0 = q == P ? out.part[0].nblk : 0;
    R.vec0 = q == P ? out.part[0].np + out.part[0].nb : 0;
    out.max_blk = std::max(out.max_blk, R.blk0 + R.nblk);
    out.max_vec = std::max(out.max_vec, R.vec0 + R.np + R.nb);
  }
  // the top's sums
  if (Q > 1) {
    const ResPart& R = out.part[P];
    std::vector<std::vector<std::pair<int, int>>> src(R.nblk), vsrc(R.np);
    for (int q = 0; q < P; ++q) {
      for (const auto& a : acc[q]) src[pos[a.first]].push_back({q, a.second});
      for (size_t t = 0; t < bnd[q].size(); ++t)
        vsrc[lidx[bnd[q][t]]].push_back({q, out.part[q].np + (int)t});
    }
    auto put = [&](int t, std::vector<std::pair<int, int>>& v, bool inv) {
      std::sort(v.begin(), v.end());
      out.gat.push_back(t);
      out.gat.push_back((int)out.gsrc.size() / 2);
      for (auto& x : v) {
        out.gsrc.push_back(x.first);
        out.gsrc.push_back(x.second);
      }
      out.gat.push_back((int)out.gsrc.size() / 2);
      out.gat.push_back(inv ? 1 : 0);
    };
    for (int t = 0; t < R.nblk; ++t) {
      const bool inv = t < R.np && lev[piv[P][t]] == 0;
      if (inv || !src[t].empty()) {
        put(t, src[t], inv);
        ++out.ngat_blk;
      }
    }
    for (int t = 0; t < R.np; ++t)
      if (!vsrc[t].empty()) {
        put(t, vsrc[t], false);
        ++out.ngat_vec;
      }
  }
  // mismatch rows and Jacobian entries of each CTA
  out.cta.resize(P);
  for (int c = 0; c < P; ++c) {
    ResCta& C = out.cta[c];
    std::vector<int> rows = piv[c];
    if (c == 0 && Q > 1) rows.insert(rows.end(), piv[P].begin(), piv[P].end());
    auto len = [&](int i) { return s.y_rowptr[i + 1] - s.y_rowptr[i]; };
    std::stable_sort(rows.begin(), rows.end(), [&](int a, int b) { return len(a) > len(b); });
    C.grp = (int)out.grp.size();
    for (size_t g = 0; g < rows.size(); g += 32) {
      const int width = len(rows[g]);
      out.grp.push_back({(int)out.ell_col.size(), width});
      out.ell_col.resize(out.ell_col.size() + (size_t)32 * width, 0);
      out.ell_y.resize(out.ell_col.size(), -1);
      for (int l = 0; l < 32; ++l) {
        if (g + l >= rows.size()) {
          for (int k = 0; k < 4; ++k) out.row.push_back(-1);
          continue;
        }
        const int i = rows[g + l], q = part[i];
        const ResPart& R = out.part[q];
        const int ydiag = s.lu2y[s.lu_diag[i]];
        // a boundary row's or the top's diagonal is final after the sums
        const bool l0 = lev[i] == 0 && q < P;
        out.row.push_back(i | (l0 ? kResRowLevel0 : 0));
        out.row.push_back(R.blk0 + lidx[i]);
        out.row.push_back(R.vec0 + lidx[i]);
        out.row.push_back(ydiag);
        int* col = out.ell_col.data() + out.grp.back().ell + l;
        int* ye = out.ell_y.data() + out.grp.back().ell + l;
        int e = 0;
        col[0] = i;
        ye[0] = ydiag;
        for (int p = s.y_rowptr[i]; p < s.y_rowptr[i + 1]; ++p) {
          if (p == ydiag) continue;
          ++e;
          col[32 * e] = s.y_col[p];
          ye[32 * e] = p;
        }
        for (++e; e < width; ++e) col[32 * e] = i;
      }
    }
    C.ngrp = (int)out.grp.size() - C.grp;
    C.jac = (int)out.jac.size() / 4;
    for (int q : {c, P}) {
      if (q >= Q || (q == P && (c > 0 || Q == 1))) continue;
      for (int e = 0; e < nnz; ++e) {
        if (s.lu2y[e] < 0 || rowof[e] == s.lu_col[e] || home(e) != q) continue;
        out.jac.push_back(out.part[q].blk0 + pos[e]);
        out.jac.push_back(rowof[e]);
        out.jac.push_back(s.lu_col[e]);
        out.jac.push_back(s.lu2y[e]);
      }
    }
    C.njac = (int)out.jac.size() / 4 - C.jac;
    const ResPart& A = out.part[c];
    C.tab = A.rf;
    C.ntab = A.rb + A.nrb - A.rf;
    out.max_tab = std::max(out.max_tab, C.ntab);
  }
  if (Q > 1) {
    const ResPart& A = out.part[P];
    out.max_tab = std::max(out.max_tab, out.cta[0].ntab + A.rb + A.nrb - A.rf);
  }
  return true;
}

bool res_plan_fit(const Symbolic& s, bool fp32, int P, int slots, size_t limit, ResPlanHost& out) {
  for (const double quad : {0.3, 1.0}) {
    ResPlanHost h;
    if (!res_plan(s, P, slots, quad, h) || res_smem(h, fp32) > limit) continue;
    out = std::move(h);
    return true;
  }
  return false;
}

}  // namespace pf
