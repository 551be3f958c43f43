// host_threads.h -- independent planner work over a few host threads.
#pragma once

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <exception>
#include <mutex>
#include <new>
#include <system_error>
#include <thread>
#include <vector>

namespace dd {

// fn(i) for every i < n until one returns false; `work` is a measure of the
// whole (about a nanosecond each), from which the number of threads follows (a
// thread costs about 20 us to start).  Runs on this thread alone where the
// system gives no other.  Returns false if some fn did; rethrows what one threw.
template <typename Fn>
bool parallel_for(int64_t n, double work, Fn fn) {
  std::atomic<int64_t> next{0};
  std::atomic<bool> ok{true};
  std::exception_ptr error;
  std::mutex error_mu;
  auto run = [&]() {
    try {
      for (int64_t i = next++; i < n && ok; i = next++)
        if (!fn(i)) ok = false;
    } catch (...) {
      std::lock_guard<std::mutex> lock(error_mu);
      if (!error) error = std::current_exception();
      ok = false;
    }
  };
  const int64_t want = std::min<int64_t>(
      {n, static_cast<int64_t>(std::thread::hardware_concurrency()), 16,
       static_cast<int64_t>(work / 100e3) + 1});
  std::vector<std::thread> threads;
  try {
    for (int64_t i = 1; i < want; ++i) threads.emplace_back(run);
  } catch (const std::system_error&) {
  } catch (const std::bad_alloc&) {
  }
  run();
  for (auto& t : threads) t.join();
  if (error) std::rethrow_exception(error);
  return ok;
}

}  // namespace dd
