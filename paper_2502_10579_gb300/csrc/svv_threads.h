// svv_threads.h -- host loops over several threads (graph building and loading).
#pragma once

#include <algorithm>
#include <cstdint>
#include <thread>
#include <vector>

namespace svv {

// threads for a loop over n items: at least 64K items each, at most 16
inline unsigned host_threads(uint64_t n) {
  if (n < (2u << 16)) return 1;  // asking for the number of cores takes 15-20 us
  const uint64_t hw = std::max(1u, std::thread::hardware_concurrency());
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(std::min<uint64_t>(hw, 16), n >> 16));
}

// f(0), ..., f(n - 1), each on its own thread where one can be had
template <class F>
void parallel(unsigned n, F f) {
  std::vector<std::thread> th;
  unsigned started = 0;
  try {
    th.reserve(n);
    for (; started + 1 < n; ++started) th.emplace_back(f, started);
  } catch (...) {  // no more threads or no memory for one: the rest runs here
  }
  for (unsigned t = started; t < n; ++t) f(t);
  for (auto& t : th) t.join();
}

// the t-th of n equal parts of [0, total) begins here
inline uint64_t part(uint64_t total, unsigned n, unsigned t) { return total / n * t + std::min<uint64_t>(t, total % n); }

// the t-th of n ranges of rows with about equal numbers of edges begins here
inline uint64_t row_at(const uint64_t* row_ptr, uint64_t V, unsigned n, unsigned t) {
  if (t == 0) return 0;
  if (t >= n) return V;
  return std::min<uint64_t>(V, (uint64_t)(std::lower_bound(row_ptr, row_ptr + V, part(row_ptr[V], n, t)) - row_ptr));
}

}  // namespace svv
