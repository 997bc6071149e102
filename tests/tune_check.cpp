// Host-side check of the autotuner's choice of replays (no GPU needed): times that a
// cold start or one slow replay would give, and what is made of them.
// Prints "ok" and returns 0, or prints the first mismatch and returns 1.
#include <cstdio>
#include <vector>

#include "../paper_2002_09603_gb300/csrc/tune.h"

namespace {

int run(const char* what, float best_us, const std::vector<float>& times, float want, size_t want_replays) {
  size_t next = 0;
  const float got = mhfp::best_replay_us(best_us, [&] { return next < times.size() ? times[next++] : 1e9f; });
  if (got == want && next == want_replays) return 0;
  std::printf("%s: %g after %zu replays, expected %g after %zu\n", what, got, next, want, want_replays);
  return 1;
}

}  // namespace

int main() {
  const float none = 1e30f;
  int bad = 0;
  bad |= run("first candidate, cold start", none, {90.f, 10.f, 10.4f, 1.f}, 10.f, 3);
  bad |= run("cold start beside a warm best", 12.f, {23.f, 10.f, 10.1f, 1.f}, 10.f, 3);
  bad |= run("a close candidate's first warm replay slow", 12.f, {14.f, 60.f, 10.f, 10.2f}, 10.f, 4);
  bad |= run("its second one slow", 12.f, {14.f, 10.f, 60.f, 9.9f}, 9.9f, 4);
  bad |= run("its last one slow", 12.f, {14.f, 10.f, 10.6f, 60.f}, 10.f, 4);
  bad |= run("a candidate just behind, unsure", 10.f, {14.f, 11.4f, 13.f, 9.8f}, 9.8f, 4);
  bad |= run("a candidate that has lost", 12.f, {5.f, 16.f, 15.f, 1.f}, 15.f, 3);
  bad |= run("a candidate far behind", 12.f, {30.f, 28.f, 28.f, 28.f}, 30.f, 1);
  if (!bad) std::printf("ok\n");
  return bad;
}
