// The static deal of work items to the persistent kernels' CTAs, for the kernels and for the host that weighs deals.
#pragma once

#include "wait_budget.h"   // GPROJ_HD

namespace gproj {

// Static persistent schedule: work items are numbered by decreasing work; round r hands item r G + c to CTA c
// on even rounds and item r G + (G - 1 - c) on odd rounds (G = number of CTAs).  With solo > 0 the first `solo` CTAs, whose
// first item is longer than an even share, get nothing after round 0 and the others share the rest in the same way.
// With clusters a whole cluster counts as one CTA here.
struct TileSched {
  int total, W, c, back, round;     // W: CTAs that share the rounds after the first; back: c counted from the other end of them
  GPROJ_HD TileSched(int total_tiles, int solo, int G, int cta) {
    c = cta;
    W = G - solo;
    back = solo + G - 1 - c;
    total = c < solo ? (total_tiles < G ? total_tiles : G) : total_tiles;
    round = 0;
  }
#ifdef __CUDACC__
  __device__ __forceinline__ TileSched(int total_tiles, int solo, int cluster)
      : TileSched(total_tiles, solo, static_cast<int>(gridDim.x) / cluster, static_cast<int>(blockIdx.x) / cluster) {}
#endif
  GPROJ_HD int next() {
    const int idx = round * W + ((round & 1) ? back : c);
    ++round;
    return idx < total ? idx : -1;
  }
};

}  // namespace gproj
