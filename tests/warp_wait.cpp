// Runs the softmax warps' wait (steel_wait.cuh) on 32 host threads, for tests/test_warp_wait.py.  A vote ends when all
// lanes have come to it; one that a lane has left for good, or that lanes come to by different calls, is an error.
#include <condition_variable>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <mutex>
#include <thread>
#include <vector>

#define __device__
#define __forceinline__ inline

struct Warp {
  std::mutex m;
  std::condition_variable cv;
  int arrived = 0, left = 0, kind = 0;
  long long votes = 0;
  bool all = true, any = false, result_all = true, result_any = false;
  std::function<void(Warp &, std::unique_lock<std::mutex> &, int)> after_vote;  // run by each lane after a vote
};
Warp *g_warp;
thread_local int g_lane;
thread_local long long g_polls, g_clock;
long long g_cycles_per_poll, g_full_at, g_most_polls;

[[noreturn]] void fail(const char *what) {
  std::printf("%s\n", what);
  std::fflush(stdout);
  std::_Exit(1);
}

bool vote(int kind, bool pred) {
  Warp &w = *g_warp;
  std::unique_lock<std::mutex> lock(w.m);
  if (w.left > 0) fail("a lane waits at a vote that another has left for good");
  if (w.arrived > 0 && w.kind != kind) fail("lanes at different votes");
  w.kind = kind;
  w.all = w.all && pred;
  w.any = w.any || pred;
  const long long mine = w.votes;
  if (++w.arrived == 32) {
    w.arrived = 0;
    w.result_all = w.all;
    w.result_any = w.any;
    w.all = true;
    w.any = false;
    ++w.votes;
  }
  w.cv.notify_all();
  w.cv.wait(lock, [&] { return w.votes != mine || w.left > 0; });
  if (w.votes == mine) fail("a lane waits at a vote that another has left for good");
  const bool r = kind == 0 ? w.result_all : w.result_any;
  if (w.after_vote) w.after_vote(w, lock, g_lane);
  return r;
}
bool __all_sync(uint32_t, bool pred) { return vote(0, pred); }
bool __any_sync(uint32_t, bool pred) { return vote(1, pred); }
long long clock64() { return g_clock; }
bool poll() {
  if (++g_polls > g_most_polls) fail("the wait goes on beyond its bound");
  g_clock += g_cycles_per_poll;
  return g_polls >= g_full_at;
}
bool mbar_test_wait(uint64_t *, uint32_t) { return g_full_at == 0; }
bool mbar_try_wait(uint64_t *, uint32_t) { return poll(); }

#include "../paper_2607_09385_b200/csrc/steel_wait.cuh"

struct Ctrl {
  int abort = 0;
  long long timeout_cycles = 0;
};

// Runs `call` in every lane; its result, which has to be the same in all.
bool run(Warp &w, const std::function<bool()> &call, long long *polls) {
  g_warp = &w;
  int passed = 0;
  std::vector<std::thread> lanes;
  for (int lane = 0; lane < 32; ++lane)
    lanes.emplace_back([&, lane] {
      g_lane = lane;
      g_polls = g_clock = 0;
      const bool ok = call();
      std::lock_guard<std::mutex> lock(w.m);
      ++w.left;
      passed += ok;
      if (polls) *polls = g_polls;
      w.cv.notify_all();
    });
  for (std::thread &t : lanes) t.join();
  if (passed != 0 && passed != 32) fail("the lanes disagree");
  return passed == 32;
}

int main(int argc, char **argv) {
  const char *what = argc > 1 ? argv[1] : "";
  Warp w;
  Ctrl ctrl;
  long long polls = 0;
  uint64_t bar = 0;
  const auto wait = [&] { return steel::warp_wait(&bar, 0u, ctrl); };
  ctrl.timeout_cycles = 200'000'000;
  g_most_polls = 1 << 20;
  g_cycles_per_poll = 100;
  if (!std::strcmp(what, "abort")) {
    // even lanes read `abort` before it is set, odd lanes after: after the 64th poll's vote the odd ones stand still
    // until the even ones have come to their next vote
    g_full_at = 1 << 20;
    bool held = false;
    w.after_vote = [&](Warp &self, std::unique_lock<std::mutex> &lock, int lane) {
      if (self.votes != 65 || lane % 2 == 0) return;
      self.cv.wait(lock, [&] { return held || self.arrived == 16; });
      held = true;
      ctrl.abort = 1;
      self.cv.notify_all();
    };
    if (run(w, wait, nullptr)) fail("the wait passed");
  } else if (!std::strcmp(what, "bound")) {
    // a poll may suspend its thread for long: 500 polls to the limit, and the clock is looked at once in 64
    g_full_at = 1 << 20;
    g_cycles_per_poll = 400'000;
    g_most_polls = 500 + 3 * 64;
    if (run(w, wait, &polls)) fail("the wait passed");
    if (polls < 490) fail("the wait ended before its bound");  // the clock is read in units of 65 536 cycles
  } else if (!std::strcmp(what, "full")) {
    for (long long at : {0, 1, 63, 64, 65, 200}) {
      Warp again;
      g_full_at = at;
      if (!run(again, wait, &polls)) fail("the wait expired");
      if (polls != at) fail("polls after the phase was complete");
    }
  } else if (!std::strcmp(what, "leave")) {
    // the flag is set while lanes read it: each has a reading of its own
    for (int seen_by : {0, 16, 32}) {
      Warp again;
      const auto aborted = [&] {
        Ctrl mine;
        mine.abort = g_lane < seen_by;
        return steel::warp_aborted(mine);
      };
      if (run(again, aborted, nullptr) != (seen_by > 0)) fail("the flag was not seen");
    }
  } else {
    return 2;
  }
  return 0;
}
