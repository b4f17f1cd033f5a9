// Waits that a whole warp makes together.  `Ctrl` has `int abort`, set once a role has given up, and
// `long long timeout_cycles`, the bound of one wait (at most kMaxTimeoutCycles).
//
// The lanes of a warp may read a shared word at different moments, so no lane acts on its own reading of `abort`:
// what one has seen is voted on, and all of them leave or all of them stay.  A lane that left alone would be missed
// for ever at the next vote or barrier of the others.  (mbar_test_wait and mbar_try_wait are declared by the file that
// includes this one: tests/warp_wait.cpp runs the code on host threads.)
#pragma once

namespace steel {

// Whether a lane has seen a role give up: the same answer in every lane.
template <class Ctrl>
__device__ __forceinline__ bool warp_aborted(Ctrl &ctrl) {
  return __any_sync(0xffffffffu, *reinterpret_cast<volatile int *>(&ctrl.abort) != 0);
}

// Every lane tests the same barrier; the vote both keeps the warp together and orders its lanes after the
// observation.  In the tile loop of the softmax warps, so it is short: the clock and `abort` are looked at once in 64
// polls (every poll that fails may suspend its thread, so polls are no measure of time), and the status word is left to
// the end of the kernel.  Clock read before the first poll and the status set here: 32 heads x 4096 d128 119.3 us,
// without both 118.5; 16/4 x 2048 26.2 -> 25.6, 12 heads x 512 d64 8.52 -> 8.48.  The time in 64 bits and the branch
// not marked as rare: 32 heads x 4096 d128 118.1 us, as here 116.8; batch 4 24/8 x 1777 83.9 -> 83.0.  A bound kept by
// the producer instead, which then outlives these warps: 8.80 -> 9.01 for 12 heads x 512 d64.
template <class Ctrl>
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, Ctrl &ctrl) {
  if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
  uint32_t n = 0, start = 0;
  while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) {
    if (__builtin_expect((++n & 63u) == 0, 0)) {
      const uint32_t now = uint32_t(clock64() >> 16);
      if (n == 64) start = now;
      const bool stop = *reinterpret_cast<volatile int *>(&ctrl.abort) != 0 ||
                        now - start > uint32_t(ctrl.timeout_cycles >> 16);
      if (__any_sync(0xffffffffu, stop)) return false;
    }
  }
  return true;
}

}  // namespace steel
