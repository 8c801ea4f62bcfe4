// Host-side check of wave_load (paper_2312_13094_gb300/csrc/fd_sched.cu), built
// with g++ by tests/test_wave_load_host.py: the load it predicts is that of the
// busiest CTA of the schedule itself, counting 2R + 4 per item.  Prints one
// line per case: G, R, predicted, found.
#include <cstdio>
#include <vector>

#include "fd_sched.h"

using namespace fd;

static void check(const std::vector<SchedGrid>& grids, int G, int R) {
  std::vector<int32_t> start;
  std::vector<WorkItem> items;
  const int used = wave_schedule(grids, G, R, start, items);
  long long busiest = 0;
  for (int c = 0; c < used; ++c) {
    long long load = 0;
    for (int i = start[c]; i < start[c + 1]; ++i) load += items[i].ze - items[i].zb + 2 * R + 4;
    busiest = load > busiest ? load : busiest;
  }
  printf("%d %d %lld %lld\n", G, R, wave_load(grids, G, R), busiest);
}

int main() {
  for (int R : {1, 4, 8})
    for (int G : {1, 7, 304, 760})
      for (int tiles : {1, 6, 7, 8, 303, 304, 305, 1521})
        for (int nz : {1, 9, 64, 370}) check({{0, tiles, nz}}, G, R);
  check({{3, 12, 40}, {0, 5, 90}, {7, 30, 12}}, 64, 3);
  check({{0, 304, 100}, {1, 305, 99}, {2, 607, 37}}, 304, 2);
  return 0;
}
