// The order in which the four warps of a 128-thread group take an MMA round trip, apart
// from the hardware it runs on (Hw), so that it can be run on host threads as well.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define STF_ROUND_FN __device__ __forceinline__
#else
#define STF_ROUND_FN inline
#endif

namespace stf {

// One MMA round trip of a group: what the threads wrote before is visible to the MMAs that
// issue() starts, and their results to every thread after.  The group's first warp waits at
// the named barrier for the others, which only arrive there, one of its threads issues, and
// every warp waits on the mbarrier itself.  (Through two barriers and one waiting thread,
// the waits at the barriers were the decode's largest stall.)
//
// A warp whose wait runs out is `dead`: it waits for no MMA and issues none any more, but
// goes on to the end of its tiles and takes the barrier of every round, so that the group's
// other warps come to theirs.  At the barriers a dead warp waits for the phase to end: if it
// only arrived, it would come by again before the first warp has been there once, and the
// phases it ended in the first warp's place would leave that warp waiting for good.  (A warp
// that is not dead cannot come by twice: it waits for the MMAs that the first warp issues
// after the phase's end, with a limit far beyond what the first warp does in between.)
// Results of a dead warp are not to be stored.
template <class Hw>
struct RoundOf {
  typename Hw::Bar bar;
  uint32_t parity;             // of the MMAs to wait for, also by drain() when dead
  int g;                       // group
  bool first, dead;            // (the same in all lanes)

  template <class Issue>
  STF_ROUND_FN void operator()(Issue issue) {
    start(issue);
    finish();
  }

  template <class Issue>
  STF_ROUND_FN void start(Issue issue) {
    Hw::before_sync();
    if (first) {
      Hw::sync(g);
      Hw::after_sync();
      if (!dead) Hw::issue_and_commit(issue, bar);
    } else if (dead) {
      Hw::sync(g);
    } else {
      Hw::arrive(g);
    }
  }

  STF_ROUND_FN void finish() {
    if (!dead) {
      dead = !Hw::wait(bar, parity);
      if (!dead) parity ^= 1;
    }
    Hw::after_sync();
  }

  // Before the group gives up its tiles: once more the wait that ran out.
  STF_ROUND_FN void drain() {
    if (dead) Hw::wait(bar, parity);
  }
};

}  // namespace stf
