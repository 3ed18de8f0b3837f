// Host test of csrc/smem_limit.h against a stand-in for the runtime.  Exit code 0 = all well.
#include <chrono>
#include <condition_variable>
#include <cstdio>
#include <map>
#include <mutex>
#include <thread>

#include "smem_limit.h"

static std::mutex mu;
static std::condition_variable cv;
static std::map<std::pair<uint64_t, const void *>, int> attribute;   // what the runtime would hold
static int sets = 0, at_once = 1;
static constexpr int kMost = 232448, kTooMuch = 1;

struct Fake {
  uint64_t ctx = 7;
  bool known = true;
  bool context(uint64_t *id) const { *id = ctx; return known; }
  int most(const void *, int *n) const { *n = kMost; return 0; }
  // The first of two threads sets the attribute, then waits (a while) until the second has set it too.
  int set(const void *kernel, int n) const {
    std::unique_lock<std::mutex> lock(mu);
    attribute[{ctx, kernel}] = n;
    ++sets;
    cv.notify_all();
    cv.wait_for(lock, std::chrono::milliseconds(500), [] { return sets >= at_once; });
    return 0;
  }
};

#define REQUIRE(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)

int main() {
  using Limits = m2rnn::SmemLimits<Fake>;
  static Limits limits(kTooMuch);
  static const char kernels[2000] = {};
  auto held = [](uint64_t ctx, const void *k) { return attribute[{ctx, k}]; };

  // two threads, the first launches of one kernel, the larger one first
  at_once = 2;
  const void *k = &kernels[0];
  std::thread a([&] { Fake api; limits.allow(api, k, 100 << 10); });
  { std::unique_lock<std::mutex> lock(mu); cv.wait_for(lock, std::chrono::seconds(5), [] { return sets >= 1; }); }
  std::thread b([&] { Fake api; limits.allow(api, k, 60 << 10); });
  a.join();
  b.join();
  at_once = 0;
  Fake api;
  for (int kb : {60, 80, 100, 200}) {   // what is granted is there
    REQUIRE(limits.allow(api, k, kb << 10) == 0);
    REQUIRE(held(7, k) >= kb << 10);
  }
  const int before = sets;
  REQUIRE(limits.allow(api, k, 150 << 10) == 0 && sets == before);   // known by now: not asked again
  REQUIRE(limits.allow(api, k, kMost) == 0);
  REQUIRE(limits.allow(api, k, kMost + 1) == kTooMuch);              // more than there is
  REQUIRE(limits.allow(api, &kernels[1], kMost + 1) == kTooMuch);    // ... before it is known, too

  // another context (a second one of the device, or the device's after a reset) starts with the runtime's default
  Fake other;
  other.ctx = 8;
  REQUIRE(limits.allow(other, k, 100 << 10) == 0 && held(8, k) >= 100 << 10);

  // a call that cannot tell its context sets the limit every time
  Fake blind;
  blind.known = false;
  attribute[{7, k}] = 0;
  REQUIRE(limits.allow(blind, k, 100 << 10) == 0 && held(7, k) >= 100 << 10);
  attribute[{7, k}] = 0;
  REQUIRE(limits.allow(blind, k, 50 << 10) == 0 && held(7, k) >= 50 << 10);

  // more pairs than the table has room for
  for (int i = 0; i < 2000; ++i) {
    Fake x;
    x.ctx = 9;
    REQUIRE(limits.allow(x, &kernels[i], 90 << 10) == 0 && held(9, &kernels[i]) >= 90 << 10);
  }
  return 0;
}
