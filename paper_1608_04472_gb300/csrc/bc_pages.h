// bc_pages.h -- host output pages made present while the device works (host code only).
#pragma once

#include <algorithm>
#include <cstddef>
#include <thread>
#include <utility>
#include <vector>

namespace bcg {

// Touches the pages of host outputs from a few threads while the device works.
// A fresh large array has no pages yet, and the copy back would fault them in
// one by one on one thread: 70 rows of 50,001 vertices (70 MB of delta,
// distances and counts) took 26-35 ms a call, 2.6 ms with the threads.
// Outputs below 4 MB are left alone. A touched byte is written with the value it
// had, so a call that fails leaves the arrays as they were.
class PageTouch {
 public:
  void add(void *p, size_t bytes) {
    if (p) parts_.push_back({static_cast<volatile char *>(p), bytes});
  }
  void start() {
    size_t total = 0;
    for (const auto &x : parts_) total += x.second;
    if (total < ((size_t)4 << 20)) return;
    const size_t most = std::max<size_t>(1, std::min<size_t>(8, std::thread::hardware_concurrency() / 2));
    const size_t nt = std::min(most, total >> 21);
    try {
      for (size_t t = 0; t < nt; ++t)
        threads_.emplace_back([this, t, nt] {
          for (const auto &x : parts_) {
            const size_t per = (x.second / nt + 4095) / 4096 * 4096;
            const size_t end = std::min(x.second, (t + 1) * per);
            for (size_t i = t * per; i < end; i += 4096) x.first[i] = x.first[i];
          }
        });
    } catch (...) {  // no thread to be had: the copy faults the rest in itself
    }
  }
  void wait() {
    for (std::thread &t : threads_) t.join();
    threads_.clear();
  }
  ~PageTouch() { wait(); }

 private:
  std::vector<std::pair<volatile char *, size_t>> parts_;
  std::vector<std::thread> threads_;
};

}  // namespace bcg
