// Host schedule of resident feeder solves (feeder.h).
#include "feeder.h"

#include <algorithm>
#include <queue>

namespace pf {

namespace {

using Op = std::pair<uint32_t, uint32_t>;

// Rounds of one level: chains of operations over the groups, long ones first.
void pack_level(std::vector<std::vector<Op>>& chains, int groups, FeedPlanHost& out) {
  if (chains.empty()) return;
  std::stable_sort(chains.begin(), chains.end(), [](const std::vector<Op>& a, const std::vector<Op>& b) {
    return a.size() > b.size();
  });
  std::vector<std::vector<Op>> col(groups);
  std::priority_queue<std::pair<int, int>, std::vector<std::pair<int, int>>,
                      std::greater<std::pair<int, int>>>
      pq;
  for (int g = 0; g < groups; ++g) pq.push({0, g});
  size_t height = 0;
  for (auto& c : chains) {
    auto t = pq.top();
    pq.pop();
    col[t.second].insert(col[t.second].end(), c.begin(), c.end());
    height = std::max(height, col[t.second].size());
    pq.push({t.first + (int)c.size(), t.second});
  }
  for (size_t r = 0; r < height; ++r) {
    int cnt = 0;
    for (int g = 0; g < groups; ++g)
      if (col[g].size() > r) cnt = g + 1;
    out.rnd.push_back((int)(out.rec.size() / 2));
    out.rnd.push_back(cnt | (r + 1 == height ? (int)0x80000000 : 0));
    for (int g = 0; g < cnt; ++g) {
      out.rec.push_back(col[g].size() > r ? col[g][r].first : kFeedNone);
      out.rec.push_back(col[g].size() > r ? col[g][r].second : 0);
    }
  }
}

}  // namespace

bool feed_plan(const Symbolic& s, const std::vector<int8_t>& btype, int P, int groups,
               FeedPlanHost& out) {
  const int n = s.n;
  out = FeedPlanHost();
  out.P = P;
  out.groups = groups;
  if (n >= kFeedMaxNodes || s.nnz_y() != n + 2 * (n - 1)) return false;  // connected: a tree
  for (int8_t t : btype)
    if (t & 16) return false;  // a PV node's columns change with the voltage
  auto each = [&](int i, auto fn) {
    for (int p = s.y_rowptr[i]; p < s.y_rowptr[i + 1]; ++p)
      if (s.y_col[p] != i) fn(s.y_col[p], p);
  };
  // the centre: the middle of a longest path
  std::vector<int> order, parent(n);
  auto bfs = [&](int r) {
    order.assign(1, r);
    parent.assign(n, -2);
    parent[r] = -1;
    for (size_t k = 0; k < order.size(); ++k)
      each(order[k], [&](int j, int) {
        if (parent[j] == -2) {
          parent[j] = order[k];
          order.push_back(j);
        }
      });
    return order.back();
  };
  const int far = bfs(bfs(0));
  std::vector<int> path;
  for (int k = far; k >= 0; k = parent[k]) path.push_back(k);
  bfs(path[path.size() / 2]);
  std::vector<std::vector<int>> child(n);
  std::vector<int> size(n, 1);
  out.branch.assign(n, -1);
  for (int t = n - 1; t >= 0; --t) {
    const int k = order[t];
    if (parent[k] < 0) continue;
    size[parent[k]] += size[k];
    child[parent[k]].push_back(k);
    each(k, [&](int j, int p) {
      if (j == parent[k]) out.branch[k] = p;
    });
  }
  // the cut: the heaviest subtree's root joins the top until the subtrees fill
  // the P parts evenly (the first part also carries the top)
  std::vector<int> part(n, P > 1 ? P : 0);
  if (P > 1) {
    std::priority_queue<std::pair<int, int>> heap;
    heap.push({size[order[0]], order[0]});
    int ntop = 0;
    double best = 1e300;
    std::vector<std::vector<int>> bins;
    while (!heap.empty()) {
      // no bins are better than even ones, nor than the heaviest subtree's
      const double least = std::max((double)heap.top().first, (double)(n - ntop) / P) + 0.25 * ntop;
      if ((int)heap.size() >= P && least >= best) {
        if (ntop > best) break;
      } else if ((int)heap.size() >= P) {
        auto h = heap;
        std::vector<std::vector<int>> bb(P);
        std::priority_queue<std::pair<int, int>, std::vector<std::pair<int, int>>,
                            std::greater<std::pair<int, int>>>
            load;
        for (int q = 0; q < P; ++q) load.push({q == 0 ? ntop : 0, q});
        int worst = 0;
        for (; !h.empty(); h.pop()) {
          auto l = load.top();
          load.pop();
          bb[l.second].push_back(h.top().second);
          l.first += h.top().first;
          worst = std::max(worst, l.first);
          load.push(l);
        }
        const double cost = worst + 0.25 * ntop;
        if (cost < best) {
          best = cost;
          bins = bb;
        } else if (ntop > best) {
          break;
        }
      }
      const int k = heap.top().second;
      heap.pop();
      ++ntop;
      for (int c : child[k]) heap.push({size[c], c});
    }
    if (bins.empty()) return false;
    for (int q = 0; q < P; ++q)
      for (int r : bins[q]) part[r] = q;
    for (int k : order)
      if (parent[k] >= 0 && part[parent[k]] < P) part[k] = part[parent[k]];
  }
  const int Q = P > 1 ? P + 1 : 1;
  // slots: a CTA's own nodes, then (first CTA) the top's
  std::vector<std::vector<int>> nodes(Q);
  for (int k : order) nodes[part[k]].push_back(k);  // parents before children
  std::vector<int> slot(n), cta(n);
  for (int q = 0; q < Q; ++q) {
    const int base = q == P ? (int)nodes[0].size() : 0;
    for (size_t t = 0; t < nodes[q].size(); ++t) {
      slot[nodes[q][t]] = base + (int)t;
      cta[nodes[q][t]] = q == P ? 0 : q;
    }
  }
  out.cta.resize(P);
  std::vector<int> slots(P, 0);
  for (int k = 0; k < n; ++k) slots[cta[k]] = std::max(slots[cta[k]], slot[k] + 1);
  out.max_slots = *std::max_element(slots.begin(), slots.end());
  if (out.max_slots >= (1 << 16)) return false;

  // rounds
  out.part.resize(Q);
  std::vector<int> lev(n, 0), dep(n, 0);
  for (int q = 0; q < Q; ++q) {
    FeedPart& R = out.part[q];
    int nl = 0, nd = 0;
    for (size_t t = nodes[q].size(); t-- > 0;) {
      const int k = nodes[q][t];
      int l = 0;
      for (int c : child[k])
        if (part[c] == q) l = std::max(l, lev[c] + 1);
      lev[k] = l;
      nl = std::max(nl, l + 1);
    }
    for (int k : nodes[q]) {
      dep[k] = parent[k] >= 0 && part[parent[k]] == q ? dep[parent[k]] + 1 : 0;
      nd = std::max(nd, dep[k] + 1);
    }
    std::vector<std::vector<std::vector<Op>>> el(nl), sub(nd);
    for (int k : nodes[q]) {
      std::vector<Op> chain;
      uint32_t first = kFeedFirst;
      for (int c : child[k]) {
        chain.push_back({(uint32_t)slot[k] | (uint32_t)slot[c] << 16,
                         (uint32_t)c | (uint32_t)cta[c] << kFeedRankShift | first});
        first = 0;
      }
      chain.push_back({(uint32_t)slot[k], (uint32_t)k | kFeedFactor | first |
                                              (parent[k] < 0 ? kFeedRoot : 0u)});
      el[lev[k]].push_back(chain);
      if (parent[k] < 0) continue;  // x = w
      const int p = parent[k];
      sub[dep[k]].push_back({{(uint32_t)slot[k] | (uint32_t)slot[p] << 16,
                              (uint32_t)k | (uint32_t)cta[p] << kFeedRankShift}});
    }
    R.rf = (int)out.rnd.size() / 2;
    for (auto& l : el) pack_level(l, groups, out);
    R.nrf = (int)out.rnd.size() / 2 - R.rf;
    R.rb = (int)out.rnd.size() / 2;
    for (auto& l : sub) pack_level(l, groups, out);
    R.nrb = (int)out.rnd.size() / 2 - R.rb;
  }
  // records and rounds of a CTA: its part's and (first CTA) the top's
  auto first_rec = [&](int r) { return r < (int)out.rnd.size() / 2 ? out.rnd[2 * r] : (int)out.rec.size() / 2; };
  for (int c = 0; c < P; ++c) {
    int nrec = 0, nrnd = 0;
    for (int q : {c, P}) {
      if (q >= Q || (q == P && (c > 0 || P == 1))) continue;
      const FeedPart& R = out.part[q];
      nrec += first_rec(R.rb + R.nrb) - first_rec(R.rf);
      nrnd += R.nrf + R.nrb;
    }
    out.max_rec = std::max(out.max_rec, nrec);
    out.max_rnd = std::max(out.max_rnd, nrnd);
  }
  // (node, phase) slots of each CTA: the free phases by the node's degree,
  // then the others (absent phases, the source: identity rows)
  for (int c = 0; c < P; ++c) {
    FeedCta& C = out.cta[c];
    std::vector<int> own = nodes[c];
    if (c == 0 && Q > 1) own.insert(own.end(), nodes[P].begin(), nodes[P].end());
    C.own = (int)out.node.size() / 2;
    C.nown = (int)own.size();
    for (int k : own) {
      out.node.push_back(k);
      out.node.push_back(slot[k]);
    }
    std::vector<std::pair<int, int>> items;  // (entries, node | phase << 28 | free << 30)
    for (int k : own)
      for (int a = 0; a < 3; ++a) {
        const bool fr = ((btype[k] >> a) & 1) && !(btype[k] & 8);
        items.push_back({fr ? s.y_rowptr[k + 1] - s.y_rowptr[k] : 0, k | a << 28 | (fr ? 1 << 30 : 0)});
      }
    std::stable_sort(items.begin(), items.end(),
                     [](const std::pair<int, int>& a, const std::pair<int, int>& b) { return a.first > b.first; });
    C.grp = (int)out.grp.size();
    for (size_t g = 0; g < items.size(); g += 32) {
      const int width = items[g].first;
      out.grp.push_back({(int)out.ell_col.size(), width});
      out.ell_col.resize(out.ell_col.size() + (size_t)32 * width, 0);
      out.ell_y.resize(out.ell_col.size(), -1);
      for (int l = 0; l < 32; ++l) {
        const bool on = g + l < items.size();
        const int id = on ? items[g + l].second : -1, k = id & (kFeedMaxNodes - 1);
        out.item.push_back(id);
        out.item.push_back(on ? slot[k] : 0);
        for (int e = 0; on && e < items[g + l].first; ++e) {
          out.ell_col[out.grp.back().ell + 32 * e + l] = s.y_col[s.y_rowptr[k] + e];
          out.ell_y[out.grp.back().ell + 32 * e + l] = s.y_rowptr[k] + e;
        }
      }
    }
    C.ngrp = (int)out.grp.size() - C.grp;
  }
  return true;
}

}  // namespace pf
