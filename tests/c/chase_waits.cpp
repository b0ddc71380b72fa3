// The chase's poll limits (poll_limit, csrc/chase_schedule.cuh) against what a
// wait may last: the whole column, at generous costs of a step and a spike
// rotation with the later columns of a rank-r update, and the shortest poll.
#include <cstdio>
#include <initializer_list>

#include "chase_schedule.cuh"

using namespace bdu::chase;

int main() {
  const int sizes[] = {1, 8, 33, 256, 1003, 4096, 16384}, extra[] = {0, 1, 4, 7, 32, 100, 1000, 4095};
  int bad = 0;
  for (int n : sizes)
    for (int more : {0, 1, 2000, 100000})
      for (int rx : extra) {
        const double waves = rx / kLanes + 1, passes = rx / 32 + 1;
        const double cycles = (11.0 * n + 200) * (3300 + 1500 * waves) + (double)more * (2500 + 1500 * passes);
        const long long limit = poll_limit(n + more, n, rx);
        if (60.0 * limit < 1.5 * cycles || 500.0 * (limit / 8) < 1.5 * cycles) {
          std::printf("m %d n %d rx %d: %lld polls for %.3g cycles\n", n + more, n, rx, limit, cycles);
          bad++;
        }
      }
  return bad ? 1 : 0;
}
