// Host-side check of ScratchSlot (paper_2312_13094_gb300/csrc/fd_slots.h), built with
// g++ by tests/test_slots_host.py.  Prints one word per case.
#include <cstdio>
#include <thread>
#include <vector>

#include "fd_slots.h"

static std::atomic<bool> taken[3];

int main() {
  // a call that has waited gives its slot back at once; one that has not waits
  // first, and nobody can have the slot before that wait ends
  for (bool waited : {true, false}) {
    int waits = 0;
    bool held = true;
    {
      auto wait = [&] {
        ++waits;
        held = held && taken[0];
      };
      fd::ScratchSlot<3, decltype(wait)> s(taken, wait);
      if (waited) s.idle();
    }
    printf("%s %d %d %d\n", waited ? "idle" : "busy", waits, int(held), int(taken[0].load()));
  }
  // distinct slots, then none, and a freed one is taken again
  auto wait = [] {};
  using Slot = fd::ScratchSlot<3, decltype(wait)>;
  {
    Slot a(taken, wait), b(taken, wait), c(taken, wait), d(taken, wait);
    printf("slots %d %d %d %d\n", a.index(), b.index(), c.index(), d.index());
  }
  Slot e(taken, wait);
  printf("again %d\n", e.index());
  // no two threads hold one slot
  std::atomic<int> in_use[3] = {{0}, {0}, {0}};
  std::atomic<int> clashes{0};
  std::vector<std::thread> ts;
  for (int t = 0; t < 4; ++t)
    ts.emplace_back([&] {
      for (int k = 0; k < 20000; ++k) {
        int i = 3;
        auto leave = [&] {
          if (i < 3) --in_use[i];
        };
        fd::ScratchSlot<3, decltype(leave)> s(taken, leave);
        i = s.index();
        if (i < 3 && ++in_use[i] != 1) ++clashes;
      }
    });
  for (std::thread& t : ts) t.join();
  printf("clashes %d\n", clashes.load());
  return 0;
}
