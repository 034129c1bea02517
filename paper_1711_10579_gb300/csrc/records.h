// Packed records of the batched factorisation and sweeps (records.cpp).
#pragma once

#include <cuda_runtime.h>

#include <vector>

#include "device.h"
#include "host.h"

namespace pf {

// The kernels' packed records of a symbolic analysis, one 16-byte load per
// item: forward / backward sweep rows {row, first entry, end, 0} in level
// order; factor items {entry, pivot k, diagonal entry of k, whether an earlier
// target finishes that entry}; targets {entry (| kFillFirst when a fill entry
// gets its first update, which then starts from zero), first L entry, first U
// entry, start of the rest in `con` or a mark}; `con` holds the other (L, U)
// pairs of a target, each list ended by (-1, mark) (most targets receive one
// update per level).  The mark is -1, or -2 - k where the target is the last
// update of pivot k's diagonal entry.
void pack_records(const Symbolic& s, std::vector<int4>& fwd, std::vector<int4>& bwd,
                  std::vector<int4>& fac, std::vector<int4>& tgt, std::vector<int2>& con);

// Sorts the items of fac and tgt so that within 256 of a level those of the same
// work are neighbours, for kernels whose warps run items in step: FP64 with 2 to
// 16 scenarios per CTA (factor_pipe; us, order of the entries / sorted: 2,000
// buses x 305 1,799 / 1,658, 10,000 x 608 10,792 / 10,630 for all launches of a
// solve).  Not for 1 or 32 scenarios (10,000 x 61 4,693 / 4,827, 3,000 x 3,000
// 10,439 / 10,679), nor FP32 (2,000 x 512 1,227 / 1,302): neighbours in memory
// are apart then.
void sort_records(const Symbolic& s, std::vector<int4>& fac, std::vector<int4>& tgt,
                  const std::vector<int2>& con);

}  // namespace pf
