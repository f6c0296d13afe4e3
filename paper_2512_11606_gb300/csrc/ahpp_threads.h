// Host threads and exceptions of the library's host code (plain C++).
#pragma once

#include <exception>
#include <mutex>
#include <thread>
#include <vector>

namespace ahpp {

// fn(t) for every t in [0, n), a thread each.  All have ended when this returns;
// what one of them throws is thrown here, and where a thread cannot be started
// the calling one does its work.
template <typename F>
void run_threads(unsigned n, const F& fn) {
  std::mutex mu;
  std::exception_ptr first;
  auto work = [&](unsigned t) {
    try {
      fn(t);
    } catch (...) {
      std::lock_guard<std::mutex> l(mu);
      if (!first) first = std::current_exception();
    }
  };
  std::vector<std::thread> th;
  unsigned t = 0;
  try {
    th.reserve(n);
    for (; t + 1 < n; ++t) th.emplace_back(work, t);
  } catch (...) {
  }
  for (; t < n; ++t) work(t);
  for (auto& x : th) x.join();
  if (first) std::rethrow_exception(first);
}

}  // namespace ahpp
