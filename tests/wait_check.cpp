// Host-side check of csrc/nasg_wait.h: how long a bounded wait lasts.
#include <cstdio>
#include <initializer_list>

#include "nasg_wait.h"

static const uint64_t kSecond = 1000000000ull;

// Looks at the clock every `step` ns, `away` ns more after the first; how many until the wait is over.
static int looks(uint64_t step, uint64_t away) {
  nasg::WaitClock c(123456789ull);
  uint64_t now = 123456789ull;
  for (int k = 1; k <= 2000000; ++k) {
    now += step + (k == 1 ? away : 0);
    if (c.over(now, kSecond)) return k;
  }
  return -1;
}

int main() {
  // polling without a break ends after a second
  for (uint64_t step : {1000ull, 180000ull, 1000000ull}) {
    const int k = looks(step, 0);
    if (k != int(kSecond / step) + 1) return std::printf("step %llu: %d looks\n", (unsigned long long)step, k), 1;
  }
  // ten seconds during which nobody ran cost one step, not the wait
  const int k = looks(180000, 10 * kSecond);
  if (k < 5500 || k > 5556) return std::printf("away: %d looks\n", k), 1;
  // steps that are all long (each poll slow) still end
  const int slow = looks(50000000, 0);
  if (slow != 1001) return std::printf("slow: %d looks\n", slow), 1;
  std::printf("ok\n");
  return 0;
}
