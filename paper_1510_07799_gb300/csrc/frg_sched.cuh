// frg_sched.cuh -- tile schedules of the persistent contraction kernels.
#pragma once
#include <algorithm>
#include <functional>
#include <queue>
#include <utility>
#include <vector>

#include "frg_common.cuh"

namespace frg {

// A schedule on the device: the records of CTA c are work[start[c]] up to
// work[start[c + 1]].
template <typename W>
struct Schedule {
  W *work = nullptr;
  int *start = nullptr;
  int grid = 0;
};

// Longest-processing-time schedule of (cost, record) tiles over at most `sms` CTAs:
// sorted by cost, each given to the CTA with the least work so far (the lowest
// numbered of equals).  The heap keeps a context's set-up short: a search over
// all CTAs for each of the 6000 tiles at N = 256 takes 2 ms of 5.
template <typename W>
bool upload_schedule(Schedule<W> &out, std::vector<std::pair<int, W>> &tiles, int sms) {
  std::stable_sort(tiles.begin(), tiles.end(), [](auto &a, auto &b) { return a.first > b.first; });
  out.grid = std::min((int)tiles.size(), sms);
  if (!out.grid) return true;
  std::vector<std::vector<W>> per(out.grid);
  using Load = std::pair<long, int>;
  std::priority_queue<Load, std::vector<Load>, std::greater<Load>> q;
  for (int c = 0; c < out.grid; ++c) q.push({0, c});
  for (auto &t : tiles) {
    const Load l = q.top();
    q.pop();
    per[l.second].push_back(t.second);
    q.push({l.first + t.first, l.second});
  }
  std::vector<W> flat;
  flat.reserve(tiles.size());
  std::vector<int> start(1, 0);
  for (auto &v : per) {
    flat.insert(flat.end(), v.begin(), v.end());
    start.push_back((int)flat.size());
  }
  return cudaMalloc(&out.work, sizeof(W) * flat.size()) == cudaSuccess &&
         cudaMalloc(&out.start, sizeof(int) * start.size()) == cudaSuccess &&
         cudaMemcpy(out.work, flat.data(), sizeof(W) * flat.size(), cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(out.start, start.data(), sizeof(int) * start.size(), cudaMemcpyHostToDevice) == cudaSuccess;
}
template <typename W>
void drop_schedule(Schedule<W> &s) {
  cudaFree(s.work);
  cudaFree(s.start);
}

}  // namespace frg
