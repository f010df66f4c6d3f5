// host_threads.h -- bound on the short-lived threads of host loops (plain C++).
#pragma once

#include <algorithm>
#include <atomic>
#include <thread>

namespace afmpb {

// Threads that a loop may start beside its caller's, until the object goes: up to `want`, and
// two per core of the host for all handles of the process together (one handle's eigensolvers
// start up to four per table, and a server's slots set up at the same time).  What is not
// granted runs on the caller's thread.
class HostThreads {
 public:
  explicit HostThreads(int want) {
    const int limit = 2 * (int)std::max(1u, std::thread::hardware_concurrency());
    int used = in_use().load();
    do {
      count_ = std::max(0, std::min(want, limit - used));
    } while (!in_use().compare_exchange_weak(used, used + count_));
  }
  ~HostThreads() { in_use() -= count_; }
  HostThreads(const HostThreads &) = delete;
  HostThreads &operator=(const HostThreads &) = delete;
  int count() const { return count_; }

 private:
  static std::atomic<int> &in_use() {
    static std::atomic<int> n{0};
    return n;
  }
  int count_ = 0;
};

}  // namespace afmpb
