// RoundOf on four host threads, one for each warp of a group: the named barrier counts
// arrivals as the hardware's does (a phase ends with the fourth, whoever brings it), and an
// mbarrier's wait gives up where a run's plan says so, or where nothing was issued.  A wait
// gives up only after the barrier's phase of its round has ended: its limit, more than a
// second, is far beyond what the first warp does until then.
// Prints nothing and returns 0 when every thread of every run came to its end.
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <mutex>
#include <thread>
#include <vector>

#include "stf_round.h"

constexpr int WARPS = 4;

struct Model {
  std::mutex m;
  std::condition_variable cv;
  int arrived = 0, phases = 0, issued = 0;
  int late[WARPS];                 // round whose wait gives up, for each warp, or -1
  bool lost(int round) const { return round == lost_round; }
  int lost_round = -1;             // round whose MMAs never complete
};

static Model* model;
thread_local int warp, round_no, gave_up_at;

static void fail(const char* what) {
  std::printf("%s: warp %d, round %d; late", what, warp, round_no);
  for (int w = 0; w < WARPS; ++w) std::printf(" %d", model->late[w]);
  std::printf(", lost %d\n", model->lost_round);
  std::fflush(stdout);
  std::_Exit(1);
}

static void until(std::unique_lock<std::mutex>& lk, const char* what, bool (*done)(int), int arg) {
  if (!model->cv.wait_for(lk, std::chrono::seconds(5), [&] { return done(arg); })) fail(what);
}

struct HostGroup {
  using Bar = int;                 // (the rounds issued so far stand for its phase)
  static void before_sync() {}
  static void after_sync() {}
  static int arrive_locked() {
    const int phase = model->phases;
    if (++model->arrived == WARPS) {
      model->arrived = 0;
      ++model->phases;
      model->cv.notify_all();
    }
    return phase;
  }
  static void arrive(int) {
    std::lock_guard<std::mutex> lk(model->m);
    arrive_locked();
  }
  static void sync(int) {
    std::unique_lock<std::mutex> lk(model->m);
    const int phase = arrive_locked();
    until(lk, "a barrier's phase never ends", [](int p) { return model->phases > p; }, phase);
  }
  template <class Issue>
  static void issue_and_commit(Issue issue, int) {
    std::lock_guard<std::mutex> lk(model->m);
    issue();
    ++model->issued;
    model->cv.notify_all();
  }
  // of round round_no (of the one that was given up, when it is waited for again)
  static bool wait(int, uint32_t parity) {
    std::unique_lock<std::mutex> lk(model->m);
    const bool again = gave_up_at >= 0;
    const int r = again ? gave_up_at : round_no;
    if (parity != (uint32_t)(r & 1)) fail("waits for another phase");
    if (!again) until(lk, "the first warp never comes", [](int n) { return model->phases > n; }, r);
    // complete once issued; the first warp issues right after the phase's end or not at all
    const bool done = !model->lost(r) && !(!again && model->late[warp] == r) &&
                      model->cv.wait_for(lk, std::chrono::milliseconds(20), [&] { return model->issued > r; });
    if (!done) gave_up_at = r;
    return done;
  }
};

// Tiles of PHASES rounds each, as the kernels walk them.
constexpr int PHASES = 3;

static void warp_main(int w, int tiles) {
  warp = w;
  gave_up_at = -1;
  round_no = 0;
  stf::RoundOf<HostGroup> round{0, 0, 0, w == 0, false};
  int tile = 0, left = -1;
  for (; tile < tiles && left < 0; left < 0 ? ++tile : 0)
    for (int k = 0; k < PHASES; ++k, ++round_no)
      if (!round([] {})) {
        left = PHASES - 1 - k;
        break;
      }
  if (left >= 0) round.give_up(left, PHASES, tile, tiles, 1);
  if (round.dead != (gave_up_at >= 0)) fail("a wait ran out and the warp goes on");
}

int main(int argc, char** argv) {
  const int tiles = argc > 1 ? std::atoi(argv[1]) : 2, rounds = PHASES * tiles;
  auto run = [&](const int* late, int lost) {
    Model mm;
    for (int w = 0; w < WARPS; ++w) mm.late[w] = late[w];
    mm.lost_round = lost;
    model = &mm;
    std::vector<std::thread> t;
    for (int w = 0; w < WARPS; ++w) t.emplace_back(warp_main, w, tiles);
    for (auto& x : t) x.join();
    if (mm.arrived != 0 || mm.phases != rounds) fail("arrivals left over");
  };
  const int none[WARPS] = {-1, -1, -1, -1};
  run(none, -1);
  for (int r = 0; r < rounds; ++r) run(none, r);
  for (int a = 0; a < WARPS * rounds; ++a)
    for (int b = a; b < WARPS * rounds; ++b) {
      int late[WARPS] = {-1, -1, -1, -1};
      late[a % WARPS] = a / WARPS;
      if (late[b % WARPS] < 0) late[b % WARPS] = b / WARPS;
      run(late, -1);
    }
  const int others[WARPS] = {-1, 0, 0, 0};     // all but the first warp, at once
  run(others, -1);
  return 0;
}
