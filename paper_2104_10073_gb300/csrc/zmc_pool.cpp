// zmc_pool.cpp -- a small pool of host threads for the per-descriptor host work
// (validation and FP64 precompute of the evaluation constants), which is
// independent per descriptor: large tables are cut into ranges that the
// calling thread and the workers take from a shared counter.  The workers are
// created at first use and live until the process exits.
#include <pthread.h>

#include <algorithm>
#include <atomic>
#include <condition_variable>
#include <functional>
#include <memory>
#include <mutex>
#include <thread>
#include <vector>

#include "zmc_runtime.h"

namespace zmc {
namespace {

// One parallel loop.  A worker holds a reference, so one that wakes after the loop
// has ended finds no range left and touches nothing of the caller's.
struct Loop {
  const std::function<void(size_t, size_t)> *fn;
  size_t n, grain;
  std::atomic<size_t> next{0}, done{0};
  // Takes ranges until none is left; true when this call finished the last one.
  bool work() {
    bool last = false;
    for (size_t b; (b = next.fetch_add(grain, std::memory_order_relaxed)) < n;) {
      const size_t e = std::min(n, b + grain);
      (*fn)(b, e);
      last = done.fetch_add(e - b, std::memory_order_acq_rel) + (e - b) == n;
    }
    return last;
  }
  bool left() const { return next.load(std::memory_order_relaxed) < n; }
};

// The caller waits for the ranges, not for the workers: with 15 workers to wake and
// hear from, a loop of 20 us took 60.  For a few ranges it wakes one worker, and each
// that finds work wakes the next; a loop of many ranges wakes them all.
class HostPool {
 public:
  HostPool() {
    const unsigned hw = std::thread::hardware_concurrency();
    const unsigned n = std::min(15u, hw > 1 ? hw - 1 : 0u);
    for (unsigned i = 0; i < n; ++i) workers_.emplace_back([this] { serve(); });
  }
  size_t size() const { return workers_.size() + 1; }

  // fn(begin, end) over [0, n) in ranges of `grain`; returns when all are done.
  void run(size_t n, size_t grain, const std::function<void(size_t, size_t)> &fn) {
    std::lock_guard<std::mutex> one(call_mu_);  // one parallel loop at a time
    auto loop = std::make_shared<Loop>();
    loop->fn = &fn;
    loop->n = n;
    loop->grain = grain;
    {
      std::lock_guard<std::mutex> g(mu_);
      loop_ = loop;
      ++gen_;
    }
    if (n / grain >= 2 * workers_.size())
      cv_.notify_all();
    else
      cv_.notify_one();
    if (loop->work()) return;
    std::unique_lock<std::mutex> lk(mu_);
    done_cv_.wait(lk, [&] { return loop->done.load(std::memory_order_acquire) == n; });
  }

 private:
  void serve() {
    uint64_t seen = 0;
    for (;;) {
      std::shared_ptr<Loop> loop;
      {
        std::unique_lock<std::mutex> lk(mu_);
        cv_.wait(lk, [&] { return gen_ != seen; });
        seen = gen_;
        loop = loop_;
      }
      if (!loop->left()) continue;
      cv_.notify_one();
      if (loop->work()) {
        std::lock_guard<std::mutex> g(mu_);  // the caller is before its check or waiting
        done_cv_.notify_all();
      }
    }
  }

  std::vector<std::thread> workers_;
  std::mutex mu_, call_mu_;
  std::condition_variable cv_, done_cv_;
  std::shared_ptr<Loop> loop_;
  uint64_t gen_ = 0;
};

// A child created by fork() has none of the parent's worker threads: from then
// on it runs every loop inline.
std::atomic<bool> g_forked{false};
void on_fork_child() { g_forked.store(true); }

// Created on first use and never destroyed: the workers wait until the process
// exits (no join at exit, where a forked child would have no threads to join).
HostPool &pool() {
  static HostPool *p = [] {
    pthread_atfork(nullptr, nullptr, on_fork_child);
    return new HostPool;
  }();
  return *p;
}

}  // namespace

void host_parallel_for(size_t n, size_t grain, const std::function<void(size_t, size_t)> &fn) {
  if (n <= grain || g_forked.load() || pool().size() == 1) {
    fn(0, n);
    return;
  }
  pool().run(n, grain, fn);
}

}  // namespace zmc
