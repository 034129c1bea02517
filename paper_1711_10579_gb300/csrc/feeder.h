// Resident solves of radial three-phase feeders: the schedule that keeps the
// 6x6 diagonal blocks of a scenario in the shared memory of one CTA, or of
// the CTAs of one cluster (feeder.cpp builds it, feeder.cu runs it).
//
// On a tree the current-injection Jacobian (Eq. 21-23) has no fill, and its
// off-diagonal blocks are the branches' admittances: -Y_k between node k and
// its parent p, constants.  Written D_k = S_k + Y_k (S_k: what is not the
// branch to the parent), the elimination towards the root is
//   S_k = S_k0 + sum_c Y_c H_c,   y_k = y_k0 + sum_c Y_c w_c   (children c)
//   H_k = (S_k + Y_k)^-1 S_k,     w_k = (S_k + Y_k)^-1 y_k
// and the substitution x_k = w_k + x_p - H_k x_p.  It is block LU on the tree
// with the cancellation taken out: the Schur complement Y_c - Y_c D_c^-1 Y_c
// is formed as Y_c H_c, where the loads in S are three to four digits below
// the admittances they would be subtracted from (mixed precision: the errors
// of 2,000-8,000-node feeders' voltages are Newton's own).  Rooted at the
// tree's centre it has half the levels of a rooting at one end.  A node pulls
// its children's results, so nothing is added to a node from two sides and a
// level of the tree is one barrier.  The tree is cut into one part of subtrees
// per CTA and a top part of common ancestors, as in resident.h.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "device.h"
#include "host.h"

namespace pf {

// An operation of a group of 8 lanes (lane j: column j of the block, lane 6 the
// right-hand side): x = node slot | child (backward: parent) slot << 16,
// y = branch (the child node of the branch) | rank << 24 | flags.
// Factorisation: pull one child, or (kFeedFactor) eliminate the node.
constexpr uint32_t kFeedFirst = 1u << 31;   // start from the node's own block
constexpr uint32_t kFeedFactor = 1u << 30;  // eliminate (else: pull a child)
constexpr uint32_t kFeedRoot = 1u << 29;    // the node has no parent
constexpr int kFeedRankShift = 24;          // CTA of the child / parent: 4 bits
constexpr int kFeedMaxNodes = 1 << 24;
constexpr uint32_t kFeedNone = 0xffffffffu;  // x of an empty place of a round
constexpr int kFeedLanes = 8;                // lanes of a group
constexpr int kFeedRing = 4;                 // branch blocks in flight per group

// One part of the tree: its rounds (offset and count of operations; negative
// count: a block barrier follows).
struct FeedPart {
  int rf, nrf;  // elimination (also the forward sweep of a refinement)
  int rb, nrb;  // substitution
};
struct FeedCta {
  int grp, ngrp;  // groups of 32 (node, phase) slots
  int own, nown;  // its nodes: FeedDev::node[own .. own + nown)
};
// Slots of a group: entry e, column c of lane l at ell + (3 e + c) 32 + l.
struct FeedGroup {
  int ell, width;
};

struct FeedPlanHost {
  int P = 1, groups = 32;
  std::vector<FeedPart> part;  // P parts, then the top (P > 1)
  std::vector<FeedCta> cta;
  std::vector<FeedGroup> grp;
  std::vector<int> item;      // [group][32][2]: node | phase << 28 | free << 30, slot
  std::vector<int> ell_col;   // [entry][32]: column node
  std::vector<int> ell_y;     // [entry][32]: Ybus entry, -1 for padding
  std::vector<int> node;      // [k][2]: node, slot
  std::vector<int> rnd;       // [round][2]
  std::vector<uint32_t> rec;  // [operation][2]
  std::vector<int> branch;    // per node: the Ybus entry (node, parent), -1 at the root
  int max_slots = 0, max_rec = 0, max_rnd = 0;  // per CTA
};

struct FeedDev {
  int P, threads;
  const FeedPart* part;
  const FeedCta* cta;
  const FeedGroup* grp;
  const int2* item;
  const int* ell_col;
  const double2* ell_y;
  const void* ydiag;   // per node: 3x3 block S_k0 without the load (complex, factor precision)
  const int2* node;
  const int2* rnd;
  const uint2* rec;
  const void* branch;  // per node: Y_k to its parent, re[9] im[9] (padded)
  int max_slots, max_rec, max_rnd;
};

// Values of a branch block in shared memory (16-byte multiple) and of a node:
// S (then H), the right-hand side (then w, x) and, in FP32, the inverse that
// refinement passes need; blocks by columns.
template <typename TF>
struct FeedShape {
  static constexpr int branch = sizeof(TF) == 4 ? 20 : 18;
  static constexpr int node = sizeof(TF) == 4 ? 36 + 6 + 36 : 36 + 6;
};

inline size_t feed_smem(const FeedPlanHost& p, bool fp32) {
  const size_t node = fp32 ? FeedShape<float>::node * 4 : FeedShape<double>::node * 8;
  const size_t branch = fp32 ? FeedShape<float>::branch * 4 : FeedShape<double>::branch * 8;
  return (((size_t)p.max_slots * node + 15) & ~(size_t)15) + (size_t)p.groups * kFeedRing * branch +
         (size_t)p.max_rec * 8 + (size_t)p.max_rnd * 8;
}

// The plan of P CTAs of `groups` groups for a case whose Ybus pattern is a
// tree; false if it is not, or exceeds the records' ranges.
bool feed_plan(const Symbolic& s, const std::vector<int8_t>& btype, int P, int groups,
               FeedPlanHost& out);

cudaError_t launch_feeder(bool fp32, const DevSys& S, const DevWork& w, const DevOpts& o,
                          const FeedDev& R, size_t smem, int B, int lin, cudaStream_t st);
cudaError_t launch_feeder_group(bool fp32, const GroupJob* desc, const GroupList& list, size_t smem,
                                int P, int threads, cudaStream_t st);
int feeder_clusters(bool fp32, int P, int threads, size_t smem);

}  // namespace pf
