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
// finish() is false, in all lanes, when the warp's wait ran out.  The warp then leaves its
// tiles, issues, reads and stores nothing more, and takes the barrier phases that it has left
// with give_up(), so that the group's other warps come to the end of theirs.  There it waits
// for each phase to end: if it only arrived, it would come by again before the first warp has
// been there once, and the phases that ended in the first warp's place would leave that warp
// waiting for good.  (A warp that goes on cannot come by twice: it waits for the MMAs that the
// first warp issues after the phase's end, with a limit far beyond what the first warp does in
// between.)  A flag that every round tests instead made the decodes 2 to 3% slower.
template <class Hw>
struct RoundOf {
  typename Hw::Bar bar;
  uint32_t parity;
  int g;                       // group
  bool first, dead;            // (the same in all lanes)

  template <class Issue>
  STF_ROUND_FN bool operator()(Issue issue) {
    start(issue);
    return finish();
  }

  template <class Issue>
  STF_ROUND_FN void start(Issue issue) {
    Hw::before_sync();
    if (first) {
      Hw::sync(g);
      Hw::after_sync();
      Hw::issue_and_commit(issue, bar);
    } else {
      Hw::arrive(g);
    }
  }

  STF_ROUND_FN bool finish() {
    const bool done = Hw::wait(bar, parity);
    parity ^= 1;
    Hw::after_sync();
    return done;
  }

  // After a finish() that was false: takes the `left` barrier phases still to come in the tile
  // and `phases` for each tile after it, and waits once more for the MMAs before the group
  // gives up its tiles.
  template <class I>
  STF_ROUND_FN void give_up(int left, int phases, I tile, I tiles, I step) {
    dead = true;
    for (;;) {
      for (; left > 0; --left) Hw::sync(g);
      tile += step;
      if (tile >= tiles) break;
      left = phases;
    }
    Hw::wait(bar, parity ^ 1);
  }
};

}  // namespace stf
