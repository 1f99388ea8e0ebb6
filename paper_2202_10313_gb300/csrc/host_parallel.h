// Loops over elements on the host's cores (set-up tables).
#pragma once
#include <algorithm>
#include <cstdint>
#include <exception>
#include <thread>
#include <vector>

namespace lts {

// fn(begin, end) over [0, n) in equal runs on the host's cores (small n: on this one). What a run
// throws is thrown here once all have ended; a thread that cannot be started (no more threads, no
// memory for one) leaves its run to the caller.
template <typename Fn>
void host_parallel(int64_t n, int64_t grain, const Fn& fn, int64_t cores = std::thread::hardware_concurrency()) {
  const int64_t nt = std::max<int64_t>(1, std::min({cores, n / grain, (int64_t)16}));
  if (nt == 1) return fn(0, n);
  std::vector<std::thread> pool;
  pool.reserve(nt - 1);   // no allocation between the first thread's start and the joins
  std::exception_ptr failed[16];
  auto part = [&](int64_t t) {
    try {
      fn(n * t / nt, n * (t + 1) / nt);
    } catch (...) {
      failed[t] = std::current_exception();
    }
  };
  int64_t started = 1;
  try {
    for (; started < nt; ++started) pool.emplace_back(part, started);
  } catch (...) {
  }
  part(0);
  for (int64_t t = started; t < nt; ++t) part(t);
  for (std::thread& t : pool) t.join();
  for (int64_t t = 0; t < nt; ++t)
    if (failed[t]) std::rethrow_exception(failed[t]);
}

}  // namespace lts
