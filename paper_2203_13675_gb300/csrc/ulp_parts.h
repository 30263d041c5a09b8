// ulp_parts.h -- where the resident solvers' blocks hand over their sums (ulp_resident.cu);
// plain C++, so that it can be checked without a GPU.
#pragma once

namespace ulp {

constexpr int kResMaxWarps = 16;  // warps of a block, one tile each: at most that many maps

// In each phase of a solve the four warps of a group add up one sum after the other and leave
// their shares for the group's first thread.  Only the barrier between writing and reading a
// share orders the group; the reads of one sum and the writes of the next ones are not ordered,
// and which maps of the block make a sum differs from phase to phase (stopped maps make none,
// maps in phase A no second one).  So every map's place and sum (d^T q or r^T s, r^T r, b^T b)
// has a slot of its own, which is written again only after the block's barriers of the phase.
constexpr int kPartSlots = 3 * kResMaxWarps;
constexpr int part_slot(int place, int sum) { return sum * kResMaxWarps + place; }

}  // namespace ulp
