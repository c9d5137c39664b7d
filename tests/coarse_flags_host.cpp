// The flag and arrival protocol of the register-resident coarse solver, run on the host: blocks in a
// row, each of which waits for its neighbours' generation, then for every block's arrival, over random
// schedules.  Exit code 1 if the order of the flag values is wrong, 2 if a schedule ends with a block
// that waits for ever.
#include <cstdio>
#include <random>
#include <vector>

#include "coarse_flags.h"

using namespace se;

int main() {
  // a generation, once passed, stays passed: by every later one and by the last arrival's value
  for (int last : {0, 1, 2, 30, 31, 500, 2147483646}) {
    for (int d = 0; d < 600 && last - d >= 0; ++d) {
      if (!coarse_flag_reached(coarse_flag_final(last), coarse_flag(last - d))) return 1;
      if (!coarse_flag_reached(coarse_flag(last), coarse_flag(last - d))) return 1;
    }
    if (coarse_flag_reached(0u, coarse_flag(last))) return 1;
    if (last > 0 && coarse_flag_reached(coarse_flag(last - 1), coarse_flag(last))) return 1;
  }
  std::mt19937 rng(1);
  for (int trial = 0; trial < 20000; ++trial) {
    const int nb = 2 + (int)(rng() % 6), last = (int)(rng() % 5), slow = (int)(rng() % nb);
    std::vector<unsigned> flag(nb, 0u);
    std::vector<int> it(nb, 0), step(nb, 0);
    unsigned count = 0;
    // step 0: post the iteration; 1: wait for the neighbours; 2: wait for all; 3: last arrival; 4: wait; 5: left
    int left = 0;
    for (long idle = 0; left < nb;) {
      int b = (int)(rng() % nb);
      if (b == slow && rng() % 16) continue;  // one block is seldom scheduled
      bool moved = true;
      switch (step[b]) {
        case 0:
          flag[b] = coarse_flag(it[b]);
          ++count;
          step[b] = 1;
          break;
        case 1: {
          bool ok = true;
          for (int q = b - 1; q <= b + 1; ++q)
            if (q >= 0 && q < nb && !coarse_flag_reached(flag[q], coarse_flag(it[b]))) ok = false;
          if (ok) step[b] = 2;
          else moved = false;
          break;
        }
        case 2:
          if ((int)(count - (unsigned)((it[b] + 1) * nb)) < 0) {
            moved = false;
          } else if (it[b] == last) {
            step[b] = 3;
          } else {
            ++it[b];
            step[b] = 0;
          }
          break;
        case 3:
          flag[b] = coarse_flag_final(it[b]);
          ++count;
          step[b] = 4;
          break;
        case 4:
          if ((int)(count - (unsigned)((it[b] + 2) * nb)) < 0) moved = false;
          else { step[b] = 5; ++left; }
          break;
        default: moved = false;
      }
      idle = moved ? 0 : idle + 1;
      if (idle > 20000) {
        std::printf("trial %d: %d of %d blocks left, block %d waits at iteration %d\n", trial, left, nb, b, it[b]);
        return 2;
      }
    }
  }
  return 0;
}
