// Prints what the scheduler's internal functions answer, for test_sched_internals.py:
// one line per query, "<query> <numbers>".
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "xe_sched.h"

int main(int argc, char **argv) {
  for (int k = 1; k + 1 < argc; k += 2) {
    const int n_in = std::atoi(argv[k + 1]);
    if (!std::strcmp(argv[k], "tune")) {
      // the autotuner's channels on 152 SMs, and every candidate's CTAs in use
      std::vector<std::vector<xe::XUnit>> units;
      for (int cover : {xe::kCoverWindow, xe::kCoverStrips, xe::kCoverPairs})
        units.push_back(xe::build_schedule(n_in, cover));
      const int C = xe::tune_channels(units, 152);
      std::printf("%d %d", n_in, C);
      for (const auto &u : units) {
        std::vector<xe::XItem> items;
        std::vector<int> first;
        std::printf(" %d", xe::build_items_filled({{&u, C, 256, 1}}, 152, items, first));
      }
      std::printf("\n");
    } else if (!std::strcmp(argv[k], "tm")) {
      // the TMEM-operand kernel's unit: operand rows, accumulator columns and
      // the modelled cycles of a chunk
      const xe::XUnit u = xe::tm_unit(n_in);
      std::printf("%d %d %d %d\n", n_in, u.z_rows, u.work, xe::chunk_cost(u));
    } else if (!std::strcmp(argv[k], "channels")) {
      // units of 8 channels, and the first channel of the last one
      const int n = xe::channel_units(n_in, 8);
      std::printf("%d %d %d\n", n_in, n, (n - 1) * 8);
    }
  }
}
