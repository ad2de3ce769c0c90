// How many blocks of 256 threads an ensemble takes per SM where the caller
// leaves it open (batch.cu holds the plan itself). Plain host code.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <functional>
#include <queue>
#include <vector>

namespace lbnr {

// When the last of `workers` blocks is done, in units of the even share, for a
// plan's teams (blocks per run, 0: not stepped): a team's blocks take its run in
// rounds of `block` cells each, and blocks that are free take the runs of one
// block, longest first. 1: perfectly even.
inline double imbalance(const std::vector<double>& cost, const std::vector<int64_t>& cells,
                        const std::vector<int>& team, int workers, int block) {
  double total = 0;
  std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
  std::vector<double> single;
  for (size_t r = 0; r < cost.size(); ++r) {
    if (team[r] < 1) continue;
    total += cost[r];
    const int64_t round = (int64_t)block * team[r];
    const double time = cost[r] / (double)cells[r] * (double)((cells[r] + round - 1) / round * block);
    if (team[r] == 1)
      single.push_back(time);
    else
      for (int k = 0; k < team[r]; ++k) free_at.push(time);
  }
  double last = 0;
  while ((int)free_at.size() < workers) free_at.push(0.0);
  std::sort(single.begin(), single.end(), std::greater<double>());
  for (double t : single) {
    const double end = free_at.top() + t;
    free_at.pop();
    free_at.push(end);
  }
  for (; !free_at.empty(); free_at.pop()) last = std::max(last, free_at.top());
  return total > 0 ? last * workers / total : 1.0;
}

// Two blocks an SM (128 registers) or one (255)? one, two: the imbalance of
// either plan; single: the share of the cost in runs of one block under one
// an SM; cells_2d: the cells of the D2Q9 runs. Time of two relative to one, SYNC:
// - Below 1.2e5 cells a step waits for one block's chain of passes, which more
//   registers shorten (31e3 cells FP32 1.43, FP64 2.06).
// - 16-bit storage waits on latency, which more warps hide: 0.60 to 0.92 over
//   1.7e5 to 1.0e7 cells, even or not.
// - FP64 is bound by its operations: 0.94 to 1.01 for teams whose plans are
//   equally even, less where two is the more even one (1.0e7 uneven cells 0.76).
//   But runs of one block become teams with barriers and spilled registers
//   (152 equal runs 1.14 to 1.24).
// - 4-byte storage: D1Q3 runs gain (0.75 to 0.80, many small ones 1.0). D2Q9 runs
//   gain while they are few (0.93 to 0.95 at 3e5 cells, 1.0 at 7e5) and then lose
//   the L2 to each other (equal runs: 1.05 at 1.2e6, 1.13 at 2.8e6, 1.18 at 5.0e6),
//   unless two is the more even plan. Imbalance of one over two, and the time:
//   at 1.3e6 cells 1.03, 1.00; 1.7e6 1.06, 0.90; 5.1e6 1.06, 1.11; 7.7e6 1.14,
//   0.95; 6.7e6 1.27, 0.88; 1.8e7 0.84, 1.18.
inline bool two_per_sm(size_t storage_bytes, int64_t cells, int64_t cells_2d, double single,
                       double one, double two) {
  if (cells < 120000) return false;
  if (storage_bytes == 2) return true;
  if (storage_bytes == 8) return single <= 0.75;
  return cells_2d <= 700000 || one >= (cells_2d <= 2000000 ? 1.04 : 1.1) * two;
}

}  // namespace lbnr
