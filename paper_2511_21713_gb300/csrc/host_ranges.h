// Ranges of a loop over host threads.  Host only, no CUDA types.
#pragma once

#include <algorithm>
#include <cstdint>
#include <exception>
#include <thread>

namespace pbfb {

constexpr int HOST_THREADS = 16;

// A partition of [0, n) into at most HOST_THREADS ranges of `grain` items or more, made once and run any number of
// times: what a pass keeps per range (sizes, buffers) fits every later pass of the same object, whatever the machine's
// processor count says by then.
class HostRanges {
 public:
  HostRanges(int64_t n, int64_t grain) : n_(n) {
    const int64_t hw = std::max(1u, std::min((unsigned)HOST_THREADS, std::thread::hardware_concurrency()));
    parts_ = (int)std::max<int64_t>(1, std::min(hw, n / std::max<int64_t>(1, grain)));
  }
  int parts() const { return parts_; }
  int64_t begin(int k) const { return n_ * k / parts_; }

  // f(k, i0, i1) for the ranges k = 0, 1, ..., each on a host thread of its own; an exception of a range is rethrown
  // here once all have ended
  template <class F>
  void run(F f) const {
    std::exception_ptr err[HOST_THREADS];
    auto part = [&](int k) {
      try {
        f(k, begin(k), begin(k + 1));
      } catch (...) {
        err[k] = std::current_exception();
      }
    };
    std::thread th[HOST_THREADS];
    int k = 1;
    try {
      for (; k < parts_; ++k) th[k] = std::thread(part, k);
    } catch (...) {  // no more threads: the rest runs here
    }
    const int started = k;
    part(0);
    for (; k < parts_; ++k) part(k);
    for (int q = 1; q < started; ++q) th[q].join();
    for (int q = 0; q < parts_; ++q)
      if (err[q]) std::rethrow_exception(err[q]);
  }

 private:
  int64_t n_;
  int parts_;
};

}  // namespace pbfb
