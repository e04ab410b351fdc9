// Host worker threads for set-up loops.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <exception>
#include <mutex>
#include <system_error>
#include <thread>
#include <vector>

namespace oras {

// Number of workers parallel_for(n, grain, ...) uses (at most min(hardware_concurrency(), 16));
// per-worker buffers are sized with it.
inline int workers_for(int64_t n, int64_t grain) {
  unsigned hw = std::thread::hardware_concurrency();
  int64_t nw = std::min<int64_t>(hw ? hw : 1, 16);
  return (int)std::max<int64_t>(1, std::min<int64_t>(nw, (n + grain - 1) / grain));
}

// Runs fn(i, worker) for i in [0, n), worker in [0, workers_for(n, grain)), chunks of `grain`
// taken from a shared counter.  Every i writes only its own outputs, so results do not depend on
// the thread count or the schedule.  An exception in any worker is rethrown here after all
// workers joined.
template <typename F>
void parallel_for(int64_t n, int64_t grain, F fn) {
  const int nw = workers_for(n, grain);
  if (nw <= 1) {
    for (int64_t i = 0; i < n; ++i) fn(i, 0);
    return;
  }
  std::atomic<int64_t> next(0);
  std::exception_ptr err;
  std::mutex err_mu;
  auto work = [&](int w) {
    try {
      for (;;) {
        const int64_t i0 = next.fetch_add(grain);
        if (i0 >= n) return;
        const int64_t i1 = std::min(n, i0 + grain);
        for (int64_t i = i0; i < i1; ++i) fn(i, w);
      }
    } catch (...) {  // keep the first error for the caller; no further chunks are taken
      std::lock_guard<std::mutex> lk(err_mu);
      if (!err) err = std::current_exception();
      next.store(n);
    }
  };
  std::vector<std::thread> th;
  for (int w = 1; w < nw; ++w) {
    try {
      th.emplace_back(work, w);
    } catch (const std::system_error&) {  // no more threads: the started ones take the rest
      break;
    }
  }
  work(0);
  for (auto& x : th) x.join();
  if (err) std::rethrow_exception(err);
}

}  // namespace oras
