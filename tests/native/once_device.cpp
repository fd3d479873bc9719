// OncePerDevice on the host: prints the calls of f for (a) two devices in turn, (b) a device whose
// first try fails, (c) eight threads on four devices (and the threads that returned before f was
// done), (d) a device outside the table.
#include <atomic>
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>

#include "once_device.h"

int main() {
  {
    ltmp2::OncePerDevice once;
    int calls[2] = {0, 0};
    for (int rep = 0; rep < 3; ++rep)
      for (int d = 0; d < 2; ++d) once.run(d, [&] { ++calls[d]; return 0; });
    std::printf("devices %d %d\n", calls[0], calls[1]);
  }
  {
    ltmp2::OncePerDevice once;
    int calls = 0, codes[3];
    for (int rep = 0; rep < 3; ++rep) codes[rep] = once.run(0, [&] { return ++calls == 1 ? 2 : 0; });
    std::printf("retry %d %d %d %d\n", calls, codes[0], codes[1], codes[2]);
  }
  {
    ltmp2::OncePerDevice once;
    std::atomic<int> calls[4] = {}, early{0};
    std::atomic<bool> ready[4] = {};
    std::vector<std::thread> th;
    for (int t = 0; t < 8; ++t)
      th.emplace_back([&, t] {
        for (int d = 0; d < 4; ++d) {
          once.run(d, [&] {
            ++calls[d];
            std::this_thread::sleep_for(std::chrono::milliseconds(5));
            ready[d] = true;
            return 0;
          });
          if (!ready[d]) ++early;
        }
      });
    for (auto &x : th) x.join();
    std::printf("threads %d %d %d %d early %d\n", calls[0].load(), calls[1].load(), calls[2].load(), calls[3].load(),
                early.load());
  }
  {
    ltmp2::OncePerDevice once;
    int calls = 0;
    for (int rep = 0; rep < 3; ++rep) once.run(1000, [&] { ++calls; return 0; });
    std::printf("beyond %d\n", calls);
  }
  return 0;
}
