// The end of a team's tile loop in the tensor-core corrector (dg_corrector.cuh).
//
// The workers of a team meet its copy warp at one barrier per tile and its MMA warp at two, and go through
// both once more when they leave the loop.  The two warps learn that from a number: the workers store at which
// barrier, counted from 0, a warp has to stop, and the warp compares it with its own count after every barrier.
// The number is stored before the barrier that it names, so the warp sees it there; a warp that is late after an
// earlier barrier may see it too soon, and goes on, because its count is lower.  (A plain flag in its place would
// let a late warp leave one barrier early, and the workers would wait for it for ever.)
#pragma once

#ifdef __CUDACC__
#define DG_TEAM_FN __host__ __device__ __forceinline__
#else
#define DG_TEAM_FN inline
#endif

namespace dg {

struct TeamStop {
  volatile int copy, mma;                      // barriers at which the copy warp and the MMA warp stop
  DG_TEAM_FN void init() { copy = mma = -1; }
  // The workers leave after `tiles` whole tiles, or in the next one after its first or second MMA barrier
  // (mma_passed 1 or 2), when the wait that follows it has run out.
  DG_TEAM_FN void set(int tiles, int mma_passed) {
    copy = tiles + (mma_passed > 0 ? 1 : 0);
    mma = 2 * tiles + mma_passed;
  }
  // After barrier n of the warp's own count.
  DG_TEAM_FN bool copy_stops(int n) const { return copy == n; }
  DG_TEAM_FN bool mma_stops(int n) const { return mma == n; }
};

}  // namespace dg

#undef DG_TEAM_FN
