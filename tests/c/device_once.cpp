// OncePerDevice: once a device, again after a failure, together from many threads.
#include <cstdio>
#include <thread>
#include <vector>

#include "device_once.h"

#define EXPECT(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
  sky::OncePerDevice once, other;
  int calls[70] = {};
  auto at = [&](sky::OncePerDevice& o, int d, int result) { return o(d, [&] { ++calls[d]; return result; }); };
  for (int d = 0; d < 8; ++d)
    for (int r = 0; r < 3; ++r) EXPECT(at(once, d, 0) == 0);
  for (int d = 0; d < 8; ++d) EXPECT(calls[d] == 1);  // the first device does not count for the others
  EXPECT(at(other, 0, 0) == 0 && calls[0] == 2);      // nor one kernel for another
  EXPECT(at(once, 63, 7) == 7 && at(once, 63, 0) == 0 && at(once, 63, 9) == 0 && calls[63] == 2);
  EXPECT(at(once, 64, 0) == 0 && at(once, 64, 0) == 0 && calls[64] == 2);
  std::atomic<int> runs{0};
  sky::OncePerDevice shared;
  std::vector<std::thread> ts;
  for (int t = 0; t < 8; ++t)
    ts.emplace_back([&, t] { for (int i = 0; i < 1000; ++i) shared(t & 1, [&] { ++runs; return 0; }); });
  for (auto& t : ts) t.join();
  EXPECT(runs >= 2 && runs <= 8);
  return 0;
}
