// host_pool.h -- host threads that the library's large host copies fan out to.
#pragma once
#include <unistd.h>

#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <cstddef>
#include <cstdint>
#include <functional>
#include <mutex>
#include <thread>
#include <vector>

namespace oasm {

// A small pool of host threads, started on first use and kept for the life of
// the process: the host-side copies of a step fan out to it without paying a
// thread start per call.  The workers take one job at a time; a caller that
// finds them busy does its own parts itself, one by one until they are free, so
// that callers on several threads (a context each) never wait for one another
// (8 of them, 3 MiB each: 228 -> 173 us a call).
class HostPool {
 public:
  static HostPool& get() {
    static HostPool pool;
    return pool;
  }
  // the caller works too; a forked child has no workers (threads do not
  // survive fork) and runs every part itself
  size_t size() const { return getpid() == pid_ ? workers_.size() + 1 : 1; }
  // Runs job(i) for i in [0, n) and returns when all have finished.
  void run(size_t n, const std::function<void(size_t)>& job) {
    std::unique_lock<std::mutex> one(job_mu_, std::try_to_lock);
    size_t first = 0;  // parts done here, while the workers were busy
    while (!one.owns_lock() && first < n) {
      job(first++);
      (void)one.try_lock();
    }
    if (first == n) return;
    {
      std::lock_guard<std::mutex> g(mu_);
      job_ = &job;
      n_ = n;
      next_.store(first);
      busy_ = workers_.size();
      ++gen_;
    }
    cv_.notify_all();
    work();
    std::unique_lock<std::mutex> g(mu_);
    done_cv_.wait(g, [&] { return busy_ == 0; });
    job_ = nullptr;
  }
  ~HostPool() {
    if (getpid() != pid_) return;  // a forked child: the workers are not ours
    {
      std::lock_guard<std::mutex> g(mu_);
      stop_ = true;
      ++gen_;
    }
    cv_.notify_all();
    for (auto& t : workers_) t.join();
  }

 private:
  HostPool() : pid_(getpid()) {
    unsigned hw = std::thread::hardware_concurrency();
    const unsigned n = hw ? std::min(hw, 16u) : 1u;
    for (unsigned i = 1; i < n; ++i) workers_.emplace_back([this] { loop(); });
  }
  void work() {
    for (size_t i; (i = next_.fetch_add(1)) < n_;) (*job_)(i);
  }
  void loop() {
    uint64_t seen = 0;
    while (true) {
      {
        std::unique_lock<std::mutex> g(mu_);
        cv_.wait(g, [&] { return gen_ != seen; });
        seen = gen_;
        if (stop_) return;
      }
      work();
      std::lock_guard<std::mutex> g(mu_);
      if (--busy_ == 0) done_cv_.notify_one();
    }
  }
  std::vector<std::thread> workers_;
  std::mutex mu_, job_mu_;
  std::condition_variable cv_, done_cv_;
  const std::function<void(size_t)>* job_ = nullptr;
  size_t n_ = 0, busy_ = 0;
  std::atomic<size_t> next_{0};
  uint64_t gen_ = 0;
  bool stop_ = false;
  pid_t pid_;
};

// Runs f(lo, hi) over [0, n) split into contiguous parts on the host pool
// (one part, on the caller, when n is small).
template <class F>
void parallel_parts(size_t n, size_t min_per_part, F f) {
  HostPool& pool = HostPool::get();
  size_t parts = std::min<size_t>(std::min<size_t>(pool.size(), 16), n / std::max<size_t>(1, min_per_part));
  if (parts <= 1) {
    f(size_t(0), n);
    return;
  }
  const std::function<void(size_t)> job = [&](size_t t) { f(n * t / parts, n * (t + 1) / parts); };
  pool.run(parts, job);
}

}  // namespace oasm
