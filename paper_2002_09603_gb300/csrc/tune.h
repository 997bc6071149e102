// Which replays the set-up's autotuner times (host only).
#pragma once
#include <algorithm>

namespace mhfp {

// Microseconds of the fastest replay of one candidate, with `best_us` the
// fastest of the candidates before it; replay() runs one and returns its time.
// The first warms the caches and decides only about a candidate at twice
// `best_us`: of an uploaded graph it takes 1.0 to 1.2 times as long as the next
// ones (0 to 7 us more over the candidates of the 47^3 and 45 x 52 x 39
// set-ups, 16 for the first of a process).  A candidate that is 1.15 times as
// slow as `best_us` in the two replays after it has lost; one slow replay, as
// the host or another client of the device causes it, does not drop a close
// candidate.  Any other is replayed a fourth time unless those two agree.
template <class Replay>
float best_replay_us(float best_us, Replay&& replay) {
  const float warm = replay();
  if (warm > 2.f * best_us) return warm;
  const float a = replay(), b = replay(), best = std::min(a, b);
  return best > 1.15f * best_us || std::max(a, b) <= 1.05f * best ? best : std::min(best, replay());
}

}  // namespace mhfp
