#include "host_parallel.hpp"

#include <algorithm>
#include <atomic>
#include <exception>
#include <mutex>
#include <thread>
#include <vector>

namespace gbdmrg {

void host_parallel(long n, long work, const std::function<void(long)>& f) {
  const unsigned hw = std::max(1u, std::thread::hardware_concurrency());
  const long nth = std::min({n, (long)std::min(16u, hw), work / 4000 + 1});
  if (nth <= 1) {
    for (long i = 0; i < n; ++i) f(i);
    return;
  }
  std::atomic<long> next{0};
  std::exception_ptr err;
  std::mutex mu;
  auto run = [&] {
    try {
      for (long i = next.fetch_add(1); i < n; i = next.fetch_add(1)) f(i);
    } catch (...) {
      next = n;
      std::lock_guard<std::mutex> lk(mu);
      if (!err) err = std::current_exception();
    }
  };
  std::vector<std::thread> th;
  try {
    th.reserve((size_t)nth);
    for (long w = 1; w < nth; ++w) th.emplace_back(run);
  } catch (const std::exception&) {
    // system_error or bad_alloc: no more threads to be had.  Nothing may leave this function
    // while one of them runs.
  }
  run();
  for (auto& t : th) t.join();
  if (err) std::rethrow_exception(err);
}

}  // namespace gbdmrg
