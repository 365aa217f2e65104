// Host-side helpers shared by the mesh builder and the multigrid hierarchy: Morton keys of
// integer octree coordinates and a small parallel loop.
#pragma once

#include <algorithm>
#include <cstdint>
#include <exception>
#include <thread>
#include <vector>

#include "internal.h"

namespace chns {
namespace host {

constexpr uint64_t kFull = 1ull << CHNS_MAXD;

inline uint64_t spread3(uint64_t v) {
  v &= 0x1FFFFFull;
  v = (v | (v << 32)) & 0x1F00000000FFFFull;
  v = (v | (v << 16)) & 0x1F0000FF0000FFull;
  v = (v | (v << 8)) & 0x100F00F00F00F00Full;
  v = (v | (v << 4)) & 0x10C30C30C30C30C3ull;
  v = (v | (v << 2)) & 0x1249249249249249ull;
  return v;
}
inline uint64_t compact3(uint64_t v) {
  v &= 0x1249249249249249ull;
  v = (v | (v >> 2)) & 0x10C30C30C30C30C3ull;
  v = (v | (v >> 4)) & 0x100F00F00F00F00Full;
  v = (v | (v >> 8)) & 0x1F0000FF0000FFull;
  v = (v | (v >> 16)) & 0x1F00000000FFFFull;
  v = (v | (v >> 32)) & 0x1FFFFFull;
  return v;
}
inline uint64_t morton(uint64_t x, uint64_t y, uint64_t z) {
  return spread3(x) | (spread3(y) << 1) | (spread3(z) << 2);
}

// Threads for a loop over n items, and f(part, begin, end) over [0, n) cut into that many parts.
inline int threads_for(int64_t n) {
  const int nt = (int)std::max(1u, std::min(16u, std::thread::hardware_concurrency()));
  return (int)std::max<int64_t>(1, std::min<int64_t>(nt, n / 4096));
}
// The last part runs on the calling thread, and so does a part whose thread cannot be started; the
// first part's exception, if any, is thrown again after all have ended.
template <class F>
void parallel_parts(int64_t n, int nt, F f) {
  const int64_t chunk = (n + nt - 1) / nt;
  std::vector<std::exception_ptr> err((size_t)nt);
  auto run = [&](int t) noexcept {
    try {
      f(t, t * chunk, std::min(n, (t + 1) * chunk));
    } catch (...) {
      err[(size_t)t] = std::current_exception();
    }
  };
  {
    struct Threads {
      std::vector<std::thread> th;
      ~Threads() {
        for (auto& t : th) t.join();
      }
    } threads;
    threads.th.reserve((size_t)nt);
    for (int t = 0; t * chunk < n; ++t) {
      if ((t + 1) * chunk >= n) {
        run(t);
        break;
      }
      try {
        threads.th.emplace_back(run, t);
      } catch (const std::exception&) {
        run(t);
      }
    }
  }
  for (auto& e : err)
    if (e) std::rethrow_exception(e);
}
// Run f(begin, end) over [0, n) on up to 16 threads.
template <class F>
void parallel_for(int64_t n, F f) {
  parallel_parts(n, threads_for(n), [&](int, int64_t b, int64_t e) { f(b, e); });
}

}  // namespace host
}  // namespace chns
