// Resident single-phase Newton-Raphson solves: the schedule that keeps a
// scenario's whole factor in the shared memory of one CTA, or of the CTAs of
// one cluster (resident.cpp builds it, resident.cu runs it).
//
// The elimination tree is cut into one part of disjoint subtrees per CTA and
// a top part of common ancestors.  A CTA eliminates its own subtrees with
// block barriers only, accumulating what they subtract from the top's
// entries in slots of its own (the top's share of the CTA's Schur
// complement); the first CTA adds those up, eliminates and solves the top
// and the parts substitute back.  So a Newton step costs four cluster
// barriers instead of two per level of the tree.
//
// The work of a part is a list of rounds.  In a round a slot (a thread; FP64: a
// pair of threads, a row of the 2x2 block each) executes at most one item of 8
// bytes:
//   block    A_t -= A_b (A_k^-1 A_c)   (t: target, b = (i, k), c = (k, j))
//   vector   y_t -= A_b (A_k^-1 y_k)   the right-hand side in the same pass
//   backward y_t -= A_b y_c, and y_t = A_t^-1 y_t after the row's last entry
// and the last update of a pivot's diagonal block inverts it in place.  The
// items of one level read only what earlier levels finished, updates of one
// target within a level are successive items of one slot, and a barrier
// ends each level's last round; so a level takes one barrier (not one for
// the column and one for the updates) and the result does not depend on
// timing.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <vector>

#include "device.h"
#include "host.h"

namespace pf {

// Item: x = t | b << 16, y = c | k << 16 | flags.  t = 0xffff: no item.
// Vector items: c unused; backward items: k unused, b = 0xffff: no product.
constexpr uint32_t kResFinal = 1u << 31;  // invert / finish the target
constexpr uint32_t kResVec = 1u << 30;    // a vector item among block items
constexpr int kResMaxRows = 1 << 14;      // rows of a part (14 bits of k)
constexpr int kResNone = 0xffff;
// A round: records [x, x + (y & 0xffff)), one per slot; negative y: a block
// barrier follows.
constexpr int kResSync = (int)0x80000000;

// One part: its rows (local order: pivots, then boundary rows of the top),
// blocks (diagonals of the pivots first, then the other Jacobian entries,
// then fill and Schur accumulators, which start from zero) and rounds.
struct ResPart {
  int np, nb;       // pivots and boundary rows
  int nblk, z0;     // blocks; those from z0 on start from zero
  int blk0, vec0;   // first block and vector slot in its CTA
  int bnd;          // boundary rows' top slots: ResDev::bnd[bnd .. bnd + nb)
  int rf, nrf;      // rounds of the factorisation with the forward sweep
  int rw, nrw;      // ... of the forward sweep alone (refinement)
  int rb, nrb;      // ... of the backward sweep
};

// The Jacobian and mismatch work of one CTA.
struct ResCta {
  int grp, ngrp;  // groups of 32 rows of similar length
  int jac, njac;  // off-diagonal Jacobian entries
  int tab, ntab;  // its rounds (part and, first CTA, top): copied to shared memory
};

// Rows of a group: entry e of lane l at ell + 32 e + l (entry 0 the
// diagonal; shorter rows end in zero entries of their own column).
struct ResGroup {
  int ell, width;
};

struct ResPlanHost {
  int P = 1, slots = 512;
  std::vector<ResPart> part;    // P parts, then the top (P > 1)
  std::vector<ResCta> cta;
  std::vector<ResGroup> grp;
  std::vector<int> row;         // [group][32][4]: row | level-0 flag, block, slot, Ybus diagonal
  std::vector<int> ell_col;     // column of an entry
  std::vector<int> ell_y;       // its Ybus entry, -1 for padding
  std::vector<int> jac;         // [entry][4]: block, row, column, Ybus entry
  std::vector<int> rnd;         // [round][2]
  std::vector<uint32_t> rec;    // [item][2]
  std::vector<int> bnd;
  // the top's sums of the parts' accumulators: target {block (or slot), first
  // source, end, flag: invert}, source {part's CTA, block (or slot) there}
  std::vector<int> gat, gsrc;
  int ngat_blk = 0, ngat_vec = 0;
  int max_blk = 0, max_vec = 0, max_tab = 0;  // per CTA
};

constexpr int kResRowLevel0 = 1 << 30;  // its diagonal block is final at assembly
constexpr int kResRing = 8;             // rounds of items in flight per thread

// The plan on the device, with the Ybus values of one precision.
struct ResDev {
  int P, threads;
  const ResPart* part;
  const ResCta* cta;
  const ResGroup* grp;
  const int4* row;        // row | level-0 flag, block, slot, Ybus diagonal
  const float2* diag32;   // FP32: a row's Ybus diagonal
  const int* ell_col;
  const double2* ell_y;
  const int4* jac;        // block, row, column, bus types and Ybus entry (row's | column's << 2 | entry << 4)
  const void* jac_y;      // Ybus value, float2 or double2
  const int2* rnd;
  const uint2* rec;
  const int* bnd;
  const int4* gat;
  const int2* gsrc;
  int ngat_blk, ngat_vec;
  int max_blk, max_vec;
};

// Threads of a slot.
constexpr int res_lanes(bool fp32) { return fp32 ? 1 : 2; }

// Shared memory of one CTA.
inline size_t res_smem(const ResPlanHost& p, bool fp32) {
  const size_t tf = fp32 ? 4 : 8;
  return (size_t)p.max_blk * 4 * tf + (size_t)p.max_vec * 2 * tf + 16 +
         (size_t)kResRing * p.slots * res_lanes(fp32) * 8 + (size_t)p.max_tab * 8;
}

// The plan of P CTAs of `slots` slots for an analysed case (2x2 blocks; an
// exact factor, or with P = 1 an ILU(0) pattern); false if a part exceeds the
// items' index ranges.
bool res_plan(const Symbolic& s, int P, int slots, double quad, ResPlanHost& out);
// The plan that fits `limit` bytes of shared memory a CTA: cut by quad = 0.3,
// which weighs the rows' assembly more than the blocks of the dense pivots, or
// where a CTA's blocks then do not fit by quad = 1.  Measured (us, 0.3 / 1):
// 10,000 buses mixed 431 / 463 and 500 / 545, 7,000 369 / 371, 2,749 FP64 495 /
// 496, 10,000 FP64 1,303 / 1,347.
bool res_plan_fit(const Symbolic& s, bool fp32, int P, int slots, size_t limit, ResPlanHost& out);

// Launch of B scenarios on clusters of R.P CTAs (resident.cu); w holds the
// state [scenario][row], and lin is set for batches: info.linear_iterations
// counts the triangular passes.
cudaError_t launch_resident(bool fp32, const DevSys& S, const DevWork& w, const DevOpts& o,
                            const ResDev& R, size_t smem, int B, int lin, cudaStream_t st);
// Newton-Krylov (GMRES(m), right ILU(0)) on one CTA per scenario with the ILU(0)
// factor in shared memory (resident_nk.cu), smem from resident_nk_smem.
cudaError_t launch_resident_nk(const DevSys& S, const DevWork& w, const DevOpts& o, const ResDev& R,
                               size_t smem, int B, cudaStream_t st);
size_t resident_nk_smem(size_t plan_smem, int n, int m);
// Several requests in one launch, one cluster each (plans of the same P and threads).
cudaError_t launch_resident_group(bool fp32, const GroupJob* desc, const GroupList& list, size_t smem,
                                  int P, int threads, cudaStream_t st);
// Clusters of P CTAs with this shared memory that the device can run at once.
int resident_clusters(bool fp32, int P, int threads, size_t smem);

}  // namespace pf
