// Estimate of a batch's time at a launch shape, for the default shape.
#pragma once
#include <algorithm>
#include <functional>
#include <queue>
#include <vector>

namespace lbeh {

// A step of one box takes the time of its cells, shared by the blocks of its
// cluster, and a part that does not shrink with them (barriers and the first
// loads behind them, the single-block tail), here in cells that one block
// steps in that time.  Measured as t(1, 2, 4, 8 blocks) = latency + cells /
// blocks: 16^3 217, 172, 145, 131 us; 32^3 891, 545, 367, 252; 64^3 6249, 3349,
// 1842, 1042, that is 0.023 us a cell and 120 to 300 us (5 000 to 13 000
// cells); FP64 16^3 1413, 774, 462, 304 and 32^3 10419, 5323, 2784, 1444, 0.31
// us a cell and 150 to 200 us (about 500).
constexpr double kBatchLatency = 8000.0, kBatchLatencyF64 = 500.0;

// Time of boxes, largest first, in clusters of `blocks` blocks of which `slots`
// run at once: each box goes to the cluster that is free first.
inline double batch_estimate(const std::vector<long long> &cells, int blocks, int slots, double latency) {
  std::priority_queue<double, std::vector<double>, std::greater<double>> free_at;
  for (int k = 0; k < slots; ++k) free_at.push(0.0);
  double end = 0.0;
  for (long long n : cells) {
    const double t = free_at.top() + latency + double(n) / blocks;
    free_at.pop();
    free_at.push(t);
    end = std::max(end, t);
  }
  return end;
}

}  // namespace lbeh
