// Limits of the kernels' waits, in SM clocks (plain C++ as well, so that the rule can be checked without a GPU).
#pragma once

#ifdef __CUDACC__
#define GPROJ_HD __host__ __device__
#else
#define GPROJ_HD
#endif

namespace gproj {

// A wait for the next stage of a pipeline: about half a second.  The dK/dV side starts beside the end of the dQ side, and its
// first waits last until that has ended: up to one tile of it, 2^24 / 64 steps of at most 2000 clocks.  (Letting all its
// warps pass griddepcontrol.wait first instead cost 0.1 to 0.9 us a call.)
constexpr long long kWaitBudgetCycles = 1000LL * 1000 * 1000;

// A wait from one tile to the next (a tile loader, an epilogue, another CTA's part) lasts as long as the tile: 700 to 2000
// clocks for each of its steps, and a long tile has a million of them (64 query heads on one KV head at 2^20 queries walk
// 2^20 steps of 64 queries).  Eight times that is allowed.  A pipeline that stands still is found by its stage waits, which
// keep the short limit and end every other wait of the CTA.
constexpr long long kStepBudgetCycles = 16384;
GPROJ_HD constexpr long long tile_wait_budget(long long steps) { return kWaitBudgetCycles + steps * kStepBudgetCycles; }

}  // namespace gproj
