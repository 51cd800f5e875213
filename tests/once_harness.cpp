// csrc/once.h with two threads: the second arrives while the first is still setting.  Prints
// whether it waited for, or did itself, what it relies on; whether a failure is tried again; and
// how often a device's setting ran when nothing raced.
#include <atomic>
#include <cstdio>
#include <thread>

#include "once.h"

int main() {
  static pdfx::OncePerDevice once;
  std::atomic<int> entered{0}, set{0};
  std::atomic<bool> go{false};
  auto slow = [&] {
    entered.fetch_add(1);
    while (!go.load()) std::this_thread::yield();
    set.fetch_add(1);
    return 0;
  };
  auto quick = [&] { entered.fetch_add(1); set.fetch_add(1); return 0; };
  std::thread first([&] { once.run(3, slow); });
  while (entered.load() == 0) std::this_thread::yield();
  once.run(3, quick);                       // the first thread is inside its setting
  std::printf("ready %d\n", set.load() > 0);
  go = true;
  first.join();
  int again = 0;
  once.run(3, [&] { ++again; return 0; });
  std::printf("again %d\n", again);
  int tries = 0;
  const int r1 = once.run(4, [&] { ++tries; return 7; }), r2 = once.run(4, [&] { ++tries; return 0; });
  once.run(4, [&] { ++tries; return 0; });
  std::printf("failure %d\n", r1 == 7 && r2 == 0 && tries == 2);
  int unknown = 0;
  for (int k = 0; k < 4; ++k) once.run(k % 2 ? -1 : pdfx::kMaxDevices, [&] { ++unknown; return 0; });
  std::printf("unknown %d\n", unknown);
}
